"""Narrow z tiles of 243 rows, whose buffers do not fill whole 128-byte lines
(csrc/colfft.cuh): forward with more tiles than blocks and the strict inverse, so
that every buffer of the ring receives TMA boxes, against tiles by copies bit for
bit and the FP64 solver (3e-5 after two steps, force rows 1e-4).
"""
import numpy as np
import pytest

from parity import check_state
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from conftest import build_flusi
    return build_flusi()


def _run(fl, n, prec, **opt):
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0), **opt}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    sim = fl.Solver(cfg, ins, precision=prec)
    sim.set_state(workloads.random_smooth_field(n, 7, mean=(0.3, 0.0, 0.0)))
    sim.step(2)
    out = sim.get_state()[0], sim.forces()[0]
    sim.close()
    return out


# columns My Mxp: 528 (198 narrow forward tiles), 1188, 3080 (97 full inverse tiles)
@pytest.mark.parametrize("strict", [0, 1])
@pytest.mark.parametrize("n", [(36, 48, 243), (48, 54, 243), (162, 81, 243)])
def test_narrow_tiles_of_243_rows(fl, n, strict):
    u, rows = _run(fl, n, "fp32", dealias_strict=strict)
    v, rows2 = _run(fl, n, "fp32", dealias_strict=strict, use_tma=0)
    assert np.array_equal(u, v) and np.array_equal(rows, rows2)
    want, want_rows = _run(fl, n, "fp64", dealias_strict=strict)
    check_state(u, want, 3e-5)
    assert np.linalg.norm(rows[:, 2:22] - want_rows[:, 2:22]) <= 1e-4 * np.linalg.norm(want_rows[:, 2:22])
