"""The exchange on more cells than the chip holds blocks: cells n/2 .. n - 1 repeat
cells 0 .. n/2 - 1, so the two halves of the result have the same bits whichever
block works on a cell, before or after which other (blocks that stay, FP64 from
20^3 on, and one block per cell). Values are checked against the oracle
elsewhere; cells with clipped values and cells without are both there.
"""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nv,nx,ny", [(64, 20, 26, 14), (64, 24, 26, 14), (64, 12, 40, 40), (32, 24, 40, 20),
                                               (32, 20, 40, 30), (32, 16, 64, 48), (32, 12, 64, 48), (32, 8, 100, 80)])
@pytest.mark.parametrize("moments", [True, False])
def test_halves_alike(precision, nv, nx, ny, moments):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    cfg = W.harris(nx=nx, ny=ny, nv=nv, lx=25.6 * nx / 128, ly=12.8 * ny / 64, precision=precision)
    n, half = cfg.ncell, cfg.ncell // 2
    assert 2 * half == n
    rng = np.random.default_rng(77)
    f0 = []
    for sp, f in zip(cfg.species, W.harris_state(cfg)):
        f = f.reshape(n, -1)[:half] * (1.0 + 0.05 * rng.uniform(-1, 1, (half, 1)))
        f[::3, ::7] = 0.0  # holes: the exchange drives them negative
        f0.append(np.concatenate([f, f]))
    r = AbiRunner(cfg, f0)
    for k in range(2):
        vmom, mout = r.mom(), r.mom()
        abi.moments(r.ctx, k, vmom)
        r.fluid[k].copy_(vmom[:, :10])
        r.fluid[k][:, 4:] *= 1.02
        abi.moment_fit(r.ctx, k, vmom, False, None, None, mout if moments else None)
        torch.cuda.synchronize()
        assert torch.equal(r.f[k][:half], r.f[k][half:])
        assert torch.equal(mout[:half], mout[half:])
        assert bool((r.f[k] >= 0).all())
    clipped = abi.vl_read_stats(r.ctx)[2]
    assert 0 < clipped < 2 * n
    r.close()
