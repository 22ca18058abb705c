"""What the FP32 x passes report as non-finite near the end of the range: a
nonlinear term that overflows under a finite velocity is FLUSI_ENONFINITE, a
velocity whose square overflows is not.  The general line kernels (x_kernel 0 at
these lengths) agree with the shared-memory kernels, which test each value.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

LENGTHS = [16, 48, 162, 384, 972]


@pytest.fixture(scope="module")
def fl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from conftest import build_flusi
    return build_flusi()


def _code(fl, nx, u0, L, x_kernel, ins=None, **opt):
    """The status of one step from u0 (0: none) and the state after it."""
    n = u0.shape[:0:-1]
    assert n[0] == nx
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "mean_mode": "fixed", **opt}
    s = fl.Solver(cfg, ins, precision="fp32")
    s.set_tuning(x_kernel=x_kernel)
    s.set_state(u0)
    s.step(1)
    try:
        s.sync()
        return fl.FLUSI_OK, s.get_state(np.float32)[0]
    except fl.FlusiError as e:
        return e.code, None
    finally:
        s.close()


def _constant(nx, value):
    u0 = np.zeros((3, 8, 9, nx), np.float32)
    u0[0] = value
    return u0, {"u_inf": (value, 0.0, 0.0), "dt_fixed": 1e-3}


def _varying(nx):
    u0 = (1e17 * workloads.random_smooth_field((nx, 9, 8), 3, kmax=2)).astype(np.float32)
    assert np.isfinite(u0).all() and 1e16 < np.abs(u0).max() < 1e18
    return u0


@pytest.mark.parametrize("x_kernel", [0, 1])
@pytest.mark.parametrize("nx", LENGTHS)
def test_overflowing_product(fl, nx, x_kernel):
    # |u| about 1e17, cells of 1e-5 / nx: |u x omega| over 1e39, |u|^2 about 1e34
    assert _code(fl, nx, _varying(nx), (1e-5, 1e-5, 1e-5), x_kernel)[0] == fl.FLUSI_ENONFINITE


@pytest.mark.parametrize("x_kernel", [0, 1])
@pytest.mark.parametrize("nx", LENGTHS)
def test_overflowing_penalization(fl, nx, x_kernel):
    dx = 4.0 / nx
    L = (4.0, 9 * dx, 8 * dx)
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    u0 = _varying(nx)
    assert _code(fl, nx, u0, L, x_kernel)[0] == fl.FLUSI_OK
    assert _code(fl, nx, u0, L, x_kernel, ins, eta=1e-30)[0] == fl.FLUSI_ENONFINITE
    # the inflow layer, with the same constant
    assert _code(fl, nx, u0, L, x_kernel, eta=1e-30, layer_width=(2 * dx, 0.0, 0.0))[0] == fl.FLUSI_ENONFINITE


@pytest.mark.parametrize("x_kernel", [0, 1])
@pytest.mark.parametrize("nx", LENGTHS)
def test_overflowing_square(fl, nx, x_kernel):
    u0, opt = _constant(nx, 2e19)
    code, u = _code(fl, nx, u0, (1.0, 1.0, 1.0), x_kernel, **opt)
    assert code == fl.FLUSI_OK and np.abs(u - u0).max() <= 1e-5 * 2e19


@pytest.mark.parametrize("nx", [64, 128, 256])
def test_overflowing_square_at_the_line_kernels_lengths(fl, nx):
    """These lengths have checked the energy sum with and without the sponge."""
    u0, opt = _constant(nx, 2e19)
    for wake in ({}, {"sponge_c": 0.1, "sponge_width": (0.25, 0.0, 0.0)}):
        assert _code(fl, nx, u0, (1.0, 1.0, 1.0), 0, **opt, **wake)[0] == fl.FLUSI_ENONFINITE
