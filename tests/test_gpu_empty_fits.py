"""Cells without density (a species that is absent from part of the grid) in the 2D3V
fits (moment fitting, Sec. 2.2, Algorithm 1): the closed-form kernel settles them, they
do not go to the direct kernels' list; zero parameters, counted as invalid.

The list's length is read from the workspace: its third selection word, after the
sections before it (csrc/abi.cu, layout_of)."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def listed(r):
    """Entries the last fit left to the direct kernels."""
    nc, at = r.cfg.ncell, 0
    for n in (nc * 160, nc * 128, nc * 128, nc * 8, nc * 80, nc * 80, nc * 24, 13 * 8):
        at = (at + n + 255) // 256 * 256
    at += (-r.work.data_ptr()) % 256 + 16
    return int(r.work[at:at + 4].view(r.torch.int32).item())


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("share", [0.5, 1.0])
def test_empty_cells(precision, share):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    cfg = W.harris(nx=100, ny=37, nv=12, lx=5.0, ly=1.85, precision=precision)
    nc, k = cfg.ncell, 1
    sp = cfg.species[k]
    rng = np.random.default_rng(83)
    th = (sp.vmax[0] / 5.0) ** 2
    t = np.zeros((nc, 10))
    # means at the box's centre, where a cell's face is: nothing of these fits rounds
    # closely, and the closed form takes all of them
    t[:, 0] = rng.uniform(0.3, 1.0, nc)
    t[:, [4, 7, 9]] = (t[:, 0] * th)[:, None]
    t[rng.random(nc) < share] = 0.0
    empty = t[:, 0] == 0.0
    r = AbiRunner(cfg, [np.zeros((nc, 12 ** 3), dtype=np.float32)] * 2, fluid=np.stack([t, t]))
    vm = torch.cat([torch.as_tensor(t), torch.zeros(nc, 10, dtype=torch.float64)], 1).to(r.dev)
    theta = [torch.full((nc, 10), float("nan"), dtype=torch.float64, device=r.dev) for _ in range(2)]
    abi.vl_reset_stats(r.ctx)
    abi.moment_fit_solve(r.ctx, k, vm, False, *theta)
    r.sync()
    assert abi.vl_read_stats(r.ctx)[3] == 2 * int(empty.sum())
    left = listed(r)
    full = nc - int(empty.sum())
    assert left <= 0.05 * full, left
    for x in theta:
        x = x.cpu().numpy()
        assert np.all(x[empty] == 0.0)
        assert np.all(np.abs(x[~empty, 0] / t[~empty, 0] - 1.0) < 1e-3)
    r.close()
