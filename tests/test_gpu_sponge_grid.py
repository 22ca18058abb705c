"""The sponge switched on and off on a bound handle: at 256, 128 and 64 points in
FP32 it changes the kernel of the x pass and with it the rows of partial sums, which
the scalar kernel must count as the pass does.
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


@pytest.mark.parametrize("nx", [64, 96, 128, 256, 384])
def test_sponge_switched_on_a_bound_handle(fl, nx):
    n = (nx, 64, 96)     # more rows than blocks run
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    plain = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0)}
    wake = {**plain, "sponge_c": 0.1, "sponge_width": (L[0] / 6, L[1] / 8, 0.0)}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    u0 = workloads.random_smooth_field(n, 5, mean=(0.3, 0.0, 0.0)).astype(np.float32)

    def run(sim):
        sim.set_state(u0)
        sim.step(3)
        return sim.get_state(np.float32)[0], sim.forces()[0]

    switched = fl.Solver(plain, ins, precision="fp32")
    run(switched)
    for cfg in (wake, plain):
        fl.flusi_set_options(switched.h, fl.make_options(cfg))
        u, rows = run(switched)
        fresh = fl.Solver(cfg, ins, precision="fp32")
        v, want = run(fresh)
        fresh.close()
        assert np.array_equal(u, v) and np.array_equal(rows, want)
    switched.close()
