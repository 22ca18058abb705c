"""The general FP32 line kernels of the x pass (csrc/xline.cuh) at every length
they serve: physical pass, real-to-complex, complex-to-real and sponge lines
against the oracle.  Tolerances are those of the other FP32 parity tests: per
step 1e-5 relative L2 by the error budget, 3e-5 after a few steps, force rows
1e-4; a transform pair 3e-6.
"""
import numpy as np
import pytest

import oracle
from parity import check_state
import workloads

pytestmark = pytest.mark.gpu

LENGTHS = [n for n in (2 ** a * 3 ** b for a in range(1, 11) for b in range(6)) if 16 <= n <= 1024]


@pytest.fixture(scope="module")
def fl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from conftest import build_flusi
    return build_flusi()


def _case(n, **kw):
    dx = 4.0 / n[0]
    L = tuple(dx * v for v in n)
    cfg = {"n": n, "L": L, "nu": 0.01, "eta": 1e-2, "cfl": 0.1, "mean_mode": "fixed", "u_inf": (0.3, 0.0, 0.0), **kw}
    ins = workloads.sphere(tuple(0.5 * v for v in L), 0.3 * min(L), profile="cos")
    return cfg, ins


def _steps(fl, cfg, ins, steps, x_kernel=0):
    u0 = workloads.random_smooth_field(cfg["n"], 7, mean=(0.3, 0.0, 0.0))
    sim = fl.Solver(cfg, ins, precision="fp32")
    sim.set_tuning(x_kernel=x_kernel)
    sim.set_state(u0)
    sim.step(steps)
    rows, _ = sim.forces()
    u = sim.get_state()[0]
    sim.close()
    ref = oracle.Simulation(cfg, ins)
    ref.set_state(u0)
    ref_rows = ref.step(steps)
    check_state(u, ref.get_state(), 3e-5)
    assert np.linalg.norm(rows[:, 2:22] - ref_rows[:, 2:22]) <= 1e-4 * np.linalg.norm(ref_rows[:, 2:22])


# 108 rows: ragged against the tiles of 16, 10, 8 and 5 rows
@pytest.mark.parametrize("nx", sorted(LENGTHS))
def test_steps_at_every_length(fl, nx):
    _steps(fl, *_case((nx, 9, 12)), 2)


@pytest.mark.parametrize("n", [(162, 9, 8), (54, 27, 9), (384, 8, 9), (972, 8, 9), (32, 8, 8)])
@pytest.mark.parametrize("scheme", ["ab2", "rk4"])
def test_wake_terms(fl, n, scheme):
    cfg, ins = _case(n, sponge_c=0.1, time_scheme=scheme)
    L = cfg["L"]
    cfg.update(sponge_width=(L[0] / 6, L[1] / 8, 0.0), layer_width=(L[0] / 16, 0.0, L[2] / 8))
    _steps(fl, cfg, ins, 3)


@pytest.mark.parametrize("nx", sorted(LENGTHS))
def test_transform_pair_and_unaligned_device_fields(fl, nx):
    """set_state and get_state on device fields at an even and an odd element
    offset (8- and 4-byte aligned real lines) and on FP64 and FP32 host arrays."""
    import torch
    n = (nx, 9, 8)
    cfg, _ = _case(n)
    u0 = workloads.random_smooth_field(n, 3, kmax=2)
    ref = oracle.Simulation(cfg, None)
    ref.set_state(u0)
    want = ref.get_state()
    sim = fl.Solver(cfg, None, precision="fp32")
    size = u0.size
    flat = torch.as_tensor(u0.astype(np.float32).ravel()).cuda()
    for shift in (0, 1):
        src = torch.zeros(size + 2, device="cuda")
        src[shift:shift + size] = flat
        out = torch.zeros(size + 2, device="cuda")
        sim.set_state(src[shift:shift + size].view(3, n[2], n[1], n[0]))
        sim.get_state_device(out[shift:shift + size].view(3, n[2], n[1], n[0]))
        torch.cuda.synchronize()
        check_state(out[shift:shift + size].view(3, n[2], n[1], n[0]).double().cpu().numpy(), want, 3e-6)
        assert float(out[:shift].abs().sum() + out[shift + size:].abs().sum()) == 0.0
    for dtype in (np.float64, np.float32):
        sim.set_state(u0.astype(dtype))
        check_state(sim.get_state(dtype)[0].astype(np.float64), want, 3e-6)
    sim.close()


@pytest.mark.parametrize("nx", [48, 162, 384])
def test_batched_members_equal_single_runs(fl, nx):
    """Members of one grid share launches; each stays bit for bit its own run."""
    n = (nx, 9, 12)
    runs = []
    for batched in (False, True):
        sims = []
        for k in range(3):
            cfg, ins = _case(n)
            cfg["nu"] = 0.01 * (k + 1)
            s = fl.Solver(cfg, ins, precision="fp32")
            s.set_state(workloads.random_smooth_field(n, k, mean=(0.3, 0.0, 0.0)))
            sims.append(s)
        if batched:
            ens = fl.Ensemble(sims)
            ens.step(4)
            ens.sync()
            assert ens.batches() == (1, 3)
        else:
            for s in sims:
                s.step(4)
        runs.append([(s.get_state()[0], s.forces()[0]) for s in sims])
        if batched:
            ens.close()
        for s in sims:
            s.close()
    for (u, r), (v, q) in zip(*runs):
        assert np.array_equal(u, v) and np.array_equal(r, q)
