"""The two-pass y and z kernels where a step has six forward fields (the vorticity
sponge) and, under RK4, a second state buffer with a tensor map of its own: against
the oracle (3e-5 and 1e-4, the bars of the other FP32 step tests; on grids over a
million points the FP64 solver, whose kernels are the staged ones, stands in for it),
and tiles by TMA against tiles by copies bit for bit.
"""
import numpy as np
import pytest

import oracle
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


# y and z lengths of one group and one buffer, of a ring of three, and of tiles in halves
@pytest.mark.parametrize("scheme", ["ab2", "rk4"])
@pytest.mark.parametrize("n", [(24, 64, 162), (96, 96, 72), (16, 384, 512), (18, 243, 486), (48, 216, 576), (16, 768, 64)])
def test_wake_terms(fl, n, scheme):
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0),
           "time_scheme": scheme, "sponge_c": 0.1, "sponge_width": (L[0] / 6, L[1] / 8, 0.0),
           "layer_width": (L[0] / 16, 0.0, L[2] / 8)}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    u0 = workloads.random_smooth_field(n, 7, mean=(0.3, 0.0, 0.0))

    def run(prec, tma):
        sim = fl.Solver({**cfg, "use_tma": tma}, ins, precision=prec)
        sim.set_state(u0)
        sim.step(2)
        out = sim.get_state()[0], sim.forces()[0]
        sim.close()
        return out

    u, rows = run("fp32", 1)
    v, rows2 = run("fp32", 0)
    assert np.array_equal(u, v) and np.array_equal(rows, rows2)
    if n[0] * n[1] * n[2] < 1000000:
        ref = oracle.Simulation(cfg, ins)
        ref.set_state(u0)
        want = ref.step(2)
        w = ref.get_state()
    else:
        w, want = run("fp64", 0)
    check_state(u, w, 3e-5)
    assert np.linalg.norm(rows[:, 2:22] - want[:, 2:22]) <= 1e-4 * np.linalg.norm(want[:, 2:22])
