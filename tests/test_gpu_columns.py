"""The two-pass y and z kernels (csrc/colfft.cuh) at every length they serve, on
grids large enough for their full tiles: FP32 steps against the FP64 solver's
staged kernels (3e-5 after two steps, the bar of the other FP32 step tests; force
rows 1e-4), with the strict 2/3 rule where it differs, and tiles by copies against
tiles by TMA bit for bit.
"""
import functools

import numpy as np
import pytest

from parity import check_state
import workloads

pytestmark = pytest.mark.gpu

LENGTHS = [64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256, 288, 324, 384, 432, 486, 512, 576, 648, 768, 864, 1024]


@pytest.fixture(scope="module")
def fl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from conftest import build_flusi
    return build_flusi()


def _full(n, most):
    c = 8
    while 2 * c * n <= (8192 if n <= 512 else 16384) and 2 * c <= most:
        c *= 2
    return c


def _smooth_at_least(v):
    return min(2 ** a * 3 ** b for a in range(11) for b in range(7) if max(8, v) <= 2 ** a * 3 ** b <= 1024)


@functools.lru_cache(maxsize=1)
def _field(n):
    return workloads.random_smooth_field(n, 7, mean=(0.3, 0.0, 0.0)).astype(np.float32)


def _run(fl, n, prec, strict, **opt):
    dx = 4.0 / max(n)
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0),
           "dealias_strict": strict, **opt}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    sim = fl.Solver(cfg, ins, precision=prec)
    sim.set_state(_field(n))
    sim.step(2)
    rows, _ = sim.forces()
    u = sim.get_state()[0]
    tiles = (sim.tuning()["y_tile_cols"], sim.tuning()["z_tile_cols"])
    sim.close()
    return u, rows, tiles


def _check(fl, n, cols, which):
    for strict in (0, 1) if n[1 + which] % 3 == 0 else (0,):
        want, want_rows, _ = _run(fl, n, "fp64", strict)
        u, rows, tiles = _run(fl, n, "fp32", strict)
        assert tiles[which] == cols
        check_state(u, want, 3e-5)
        assert np.linalg.norm(rows[:, 2:22] - want_rows[:, 2:22]) <= 1e-4 * np.linalg.norm(want_rows[:, 2:22])
        v, rows2, _ = _run(fl, n, "fp32", strict, use_tma=0)
        assert np.array_equal(u, v) and np.array_equal(rows, rows2)


@pytest.mark.parametrize("n", LENGTHS)
def test_y_lengths(fl, n):
    cols = _full(n, 256)
    planes = cols // min(cols, 16)
    _check(fl, (18, n, _smooth_at_least(51 * planes)), cols, 0)


@pytest.mark.parametrize("n", LENGTHS)
def test_z_lengths(fl, n):
    cols = _full(n, 64)
    ny = _smooth_at_least(152 * cols * 3 // 2 // 32 + 3)   # My >= 2 ny / 3 - 1 rows of 32 or 36 columns fill 152 tiles
    _check(fl, (96, ny, n), cols, 1)
