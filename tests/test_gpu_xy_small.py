"""Small FP32 grids whose x + y sweep goes to the tile kernel or the streamed one by
the length of the shifts (csrc/pfc_space_march.cu, march_late): either has the bits
of the same cells in a grid that repeats them, which is large enough for the streamed
kernel at every shift (paper Sec. 2.1, Sec. 3.3)."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv,grid", [(8, (8, 8)), (12, (8, 8)), (16, (8, 8)), (8, (8, 24)), (12, (16, 40)), (16, (16, 24))])
@pytest.mark.parametrize("cells", [0.6, 2.4, 4.2, 5.4, 6.2])
def test_small_grid_has_the_bits_of_a_large_one(nv, grid, cells):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    nx, ny = grid
    reps = 7  # periodic in x and y: the repeated grid's cells are the small one's
    f0 = (W.random_blocks((nx * ny, nv ** 3), 7) ** 3).astype(np.float32)
    out = []
    for n in (1, reps):
        cfg = W.harris(nx=nx * n, ny=ny * n, nv=nv, lx=0.2 * nx * n, ly=0.2 * ny * n, precision=32)
        cfg.bc_y = 0
        f = np.tile(f0.reshape(ny, nx, -1), (n, n, 1)).reshape(cfg.ncell, -1)
        r = AbiRunner(cfg, [f, f])
        got = torch.full((cfg.ncell, nv ** 3), float("nan"), dtype=torch.float32, device=r.dev)
        sp = cfg.species[0]
        abi.pfc_advect_xy(r.ctx, 0, cells * cfg.dx / (sp.vmax[0] - 0.5 * sp.dv[0]), got)
        r.sync()
        out.append(got.view(ny * n, nx * n, -1)[:ny, :nx].cpu().numpy().copy())
        r.close()
    assert np.array_equal(out[0], out[1])
