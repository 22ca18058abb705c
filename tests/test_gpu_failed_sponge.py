"""A non-finite state on grids whose vorticity sponge is a pass of its own: that
pass starts while the scalar kernel beside it records the failure, and every block
must leave whole or not at all.  After the failure is reported the handle takes a
new state and steps on as a fresh one does, bit for bit.
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


# FP64 lengths without a line kernel, the shared-memory kernels in FP32, lengths
# under 16, the general line kernels and the tensor-core pass's separate sponge
CASES = [((48, 36, 24), "fp64", 0), ((32, 64, 96), "fp64", 0), ((384, 48, 36), "fp64", 0), ((48, 36, 24), "fp32", 1),
         ((192, 96, 64), "fp32", 1), ((512, 32, 48), "fp32", 1), ((12, 24, 32), "fp32", 0), ((192, 96, 64), "fp32", 0),
         ((256, 32, 48), "bf16x2", 0)]


@pytest.mark.parametrize("scheme", ["ab2", "rk4"])
@pytest.mark.parametrize("n,prec,x_kernel", CASES)
def test_failure_while_the_sponge_pass_starts(fl, n, prec, x_kernel, scheme):
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0),
           "time_scheme": scheme, "sponge_c": 0.1, "sponge_width": (L[0] / 6, L[1] / 8, 0.0)}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    good = workloads.random_smooth_field(n, 5, mean=(0.3, 0.0, 0.0))
    bad = good.copy()
    bad[1, 3, 4, 5] = np.nan

    def solver():
        s = fl.Solver(cfg, ins, precision=prec)
        s.set_tuning(x_kernel=x_kernel)
        return s

    fresh = solver()
    fresh.set_state(good)
    fresh.step(2)
    want = fresh.get_state()[0]
    fresh.close()
    sim = solver()
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
