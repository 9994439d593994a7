"""The FP32 velocity pass on more cells than the chip holds blocks, on an f that is
16-byte aligned (pfc_advect_v: 16-byte copies and stores) and on one that is not
(pfc_advect_v_static: scalar ones). A cell's arithmetic depends on neither, so
both give the same bits; that the values themselves are right is checked
against the oracle elsewhere.
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


@pytest.mark.parametrize("nv,nx,ny", [(8, 160, 150), (12, 96, 72), (16, 80, 60), (16, 3, 3), (20, 64, 48), (24, 48, 40)])
@pytest.mark.parametrize("e_scale,nshear", [(0.3, 5), (6.0, 5), (0.3, 3)])
def test_aligned_equals_unaligned(gpu, nv, nx, ny, e_scale, nshear):
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    cfg = W.harris(nx=nx, ny=ny, nv=nv, lx=25.6 * nx / 128, ly=12.8 * ny / 64, precision=32)
    cfg.nshear = nshear
    V, n = nv ** 3, cfg.ncell
    # random fields: every axis is the pivot somewhere, and with the larger
    # ones electrons cross whole velocity cells
    eb = W.random_fields(n, 29, e_scale=e_scale, b_scale=1.0)
    small = [W.random_blocks((min(n, 64), V), 410 + k) ** 3 for k in range(2)]
    f0 = [np.resize(f, (n, V)) for f in small]
    r = AbiRunner(cfg, f0, eb=eb)
    for k in range(2):
        room = gpu.empty(n * V + 4, dtype=gpu.float32, device="cuda")
        moved = room[1:1 + n * V].view(n, V)
        moved.copy_(r.f[k])
        mom, mom2 = r.mom(), r.mom()
        abi.pfc_advect_v(r.ctx, k, 0.01, mom)
        abi.pfc_advect_v_static(r.desc, k, moved, r.eb, n, 0.01, mom2)
        gpu.cuda.synchronize()
        assert gpu.equal(moved, r.f[k])
        assert gpu.equal(mom, mom2)
    r.close()
