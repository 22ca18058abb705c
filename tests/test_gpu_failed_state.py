"""A non-finite state on many small grids: the scalar kernel records the failure
while blocks of the forward passes beside it are starting, and every block must
leave whole or not at all.  After the failure is reported the handle takes a new
state and steps on as a fresh one does, bit for bit.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from conftest import build_flusi
    return build_flusi()


GRIDS = [(16, 16, 16), (32, 32, 32), (48, 36, 24), (54, 27, 81), (128, 64, 96), (256, 32, 48)]


@pytest.mark.parametrize("n,prec", [(n, p) for n in GRIDS for p in ("fp64", "fp32")] + [((256, 32, 48), "bf16x2")])
def test_failure_while_the_forward_passes_start(fl, n, prec):
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0)}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    good = workloads.random_smooth_field(n, 5, mean=(0.3, 0.0, 0.0))
    bad = good.copy()
    bad[1, 3, 4, 5] = np.nan
    fresh = fl.Solver(cfg, ins, precision=prec)
    fresh.set_state(good)
    fresh.step(2)
    want = fresh.get_state()[0]
    fresh.close()
    sim = fl.Solver(cfg, ins, precision=prec)
    for _ in range(8):
        sim.set_state(bad)
        sim.step(3)
        with pytest.raises(fl.FlusiError) as e:
            sim.sync()
        assert e.value.code == fl.FLUSI_ENONFINITE
        with pytest.raises(fl.FlusiError) as e:
            sim.step(1)
        assert e.value.code == fl.FLUSI_ESTATE
        sim.set_state(good)
        sim.step(2)
        assert np.array_equal(sim.get_state()[0], want)
    sim.close()
