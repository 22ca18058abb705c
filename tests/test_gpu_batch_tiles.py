"""Members of an ensemble batch equal solo runs bit for bit on grids where a solo
run takes narrower y and z tiles than the batch (csrc/ypass.cu, zpass.cu): at
every length of the two-pass kernels up to 512, and in FP64.  The narrow tiles
themselves against the FP64 solver (3e-5 after two steps, the bar of the other
FP32 step tests), and the inverse z pass by fields (grids under 2^14 values of
kept columns, FP64 2^15) against the oracle on both sides of those lines.
"""
import numpy as np
import pytest

import oracle
from parity import check_state
import workloads

pytestmark = pytest.mark.gpu

LENGTHS = [64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256, 288, 324, 384, 432, 486, 512]


@pytest.fixture(scope="module")
def fl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from conftest import build_flusi
    return build_flusi()


def _case(n, **kw):
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0), **kw}
    return cfg, workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")


def _solo(fl, cfg, ins, u0, prec):
    s = fl.Solver(cfg, ins, precision=prec)
    s.set_state(u0)
    s.step(2)
    out = s.get_state(u0.dtype)[0], s.forces()[0]
    s.close()
    return out


def _check_batch(fl, n, count, prec):
    dt = np.float64 if prec == "fp64" else np.float32
    cfg, ins = _case(n)
    base = workloads.random_smooth_field(n, 7, mean=(0.3, 0.0, 0.0))
    fields = [((1.0 - 0.05 * i) * base).astype(dt) for i in range(count)]
    members = [fl.Solver(cfg, ins, precision=prec) for _ in fields]
    for s, u0 in zip(members, fields):
        s.set_state(u0)
    ens = fl.Ensemble(members)
    ens.step(2)
    assert ens.batches() == (1, count)
    ens.sync()
    got = [(s.get_state(dt)[0], s.forces()[0]) for s in members]
    ens.close()
    for s in members:
        s.close()
    for i in (0, count - 1):
        u, rows = _solo(fl, cfg, ins, fields[i], prec)
        assert np.array_equal(got[i][0], u) and np.array_equal(got[i][1], rows)
        if prec == "fp32" and i == 0:
            want, _ = _solo(fl, cfg, ins, fields[0].astype(np.float64), "fp64")
            check_state(u, want, 3e-5)


@pytest.mark.parametrize("n", LENGTHS)
def test_y_lengths_in_a_batch(fl, n):
    _check_batch(fl, (18, n, 48), 10, "fp32")   # 6 and 60 runs of 48 planes, by 1 and by up to 8


@pytest.mark.parametrize("n", LENGTHS)
def test_z_lengths_in_a_batch(fl, n):
    _check_batch(fl, (96, 96, n), 5, "fp32")    # 37 to 147 and 185 to 735 full tiles


@pytest.mark.parametrize("n", LENGTHS)
def test_z_forward_lengths_in_a_batch(fl, n):
    _check_batch(fl, (24, 24, n), 10, "fp32")   # 24 to 78 and 240 to 780 full tiles of six fields


@pytest.mark.parametrize("n", [(32, 32, 32), (48, 36, 24), (64, 64, 64)])
def test_fp64_in_a_batch(fl, n):
    _check_batch(fl, n, 6, "fp64")


# 0.01, 0.18, 0.79, 0.88, 0.97 | 1.09, 1.25, 1.93 | 2.17, 2.5, 4.0 of 2^14; ragged tiles,
# lengths that narrow them
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [(8, 8, 8), (18, 9, 54), (8, 8, 648), (36, 36, 36), (48, 48, 24), (48, 48, 27), (8, 8, 1024),
                               (48, 48, 48), (48, 54, 48), (12, 8, 1024), (64, 64, 64)])
def test_inverse_z_by_fields(fl, n, prec):
    cfg, ins = _case(n)
    u0 = workloads.random_smooth_field(n, 7, mean=(0.3, 0.0, 0.0))
    u, rows = _solo(fl, cfg, ins, u0, prec)
    ref = oracle.Simulation(cfg, ins)
    ref.set_state(u0)
    want = ref.step(2)
    tol, tol_rows = (1e-11, 1e-10) if prec == "fp64" else (3e-5, 1e-4)
    check_state(u, ref.get_state(), tol)
    assert np.linalg.norm(rows[:, 2:22] - want[:, 2:22]) <= tol_rows * np.linalg.norm(want[:, 2:22])
