"""The streamed x + y sweep (pfc_space_march.cu) where it can go wrong: one strip
that wraps onto itself, strips that repeat cells of the one before (17 groups of
8 cells), runs of rows that do not divide ny, halos up to 8 cells, every block
size, mirror rows, and an f that is not 16-byte aligned (the general kernel).

Tolerance: two PFC sweeps in FP32, each within 2e-6 max|f| of the FP64 sweep.
"""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2109_06743_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("bc_y", [0, 1])
@pytest.mark.parametrize("grid,cfl,shift", [
    ((8, 8, 8), 0.45, 0), ((8, 8, 12), 4.7, 0), ((8, 40, 16), 5.8, 0), ((40, 56, 8), 1.9, 0),
    ((136, 24, 8), 0.3, 0), ((136, 8, 12), 5.2, 0), ((24, 24, 20), 2.6, 0), ((16, 16, 24), 0.8, 0),
    ((48, 136, 8), 5.9, 0), ((24, 16, 8), 1.3, 1)])
def test_march(gpu, orc, grid, cfl, shift, bc_y):
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    nx, ny, nv = grid
    cfg = W.harris(nx=nx, ny=ny, nv=nv, lx=25.6 * nx / 128, ly=12.8 * ny / 64, precision=32)
    cfg.bc_y = bc_y
    f0 = [(W.random_blocks((cfg.ncell, nv ** 3), 300 + k) ** 3).astype(np.float32).astype(np.float64) for k in range(2)]
    r = AbiRunner(cfg, f0)
    if shift:  # f four bytes off a 16-byte boundary
        for k in range(2):
            room = gpu.empty(r.f[k].numel() + 4, dtype=gpu.float32, device="cuda")
            moved = room[shift:shift + r.f[k].numel()].view_as(r.f[k])
            abi.pfc_advect_xy(r.ctx, k, 0.0, moved)
            r.f[k] = moved
    g = orc.make_grid(cfg.nvdim, cfg.nx, cfg.ny, cfg.x0, cfg.dx, cfg.y0, cfg.dy, cfg.bc_y)
    for k, sp in enumerate(cfg.species):
        dt = cfl * min(cfg.dx, cfg.dy) / abs(sp.vmin[0])
        if bc_y == 1:
            dt = min(dt, 0.9 * (ny - 3) * cfg.dy / abs(sp.vmin[1]))
        dt *= -1 if k else 1
        out = gpu.full((cfg.ncell, nv ** 3), float("nan"), dtype=gpu.float32, device="cuda")
        abi.pfc_advect_xy(r.ctx, k, dt, out)
        gpu.cuda.synchronize()
        ref = f0[k].copy()
        for axis in (0, 1):
            orc.advect_space(ref, g, orc.make_species(sp.q, sp.m, sp.nv, sp.vmin, sp.vmax), axis, dt)
        err = np.abs(out.double().cpu().numpy() - ref).max()
        assert err <= 4e-6 * ref.max(), (k, err, ref.max())
    assert abi.vl_read_stats(r.ctx)[8] == 0  # no row ran out of time
    r.close()
