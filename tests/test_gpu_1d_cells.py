"""1D1V grids with cells enough for a thread per cell (csrc/pfc_velocity.cu, threads1d):
on either side of the line the same cells get the same velocity step (its order of
operations is the same) and moments (sums in another order); the moments of the
step equal those of a call of their own.

Tolerances: FP64 lines bit for bit up to the contraction of one product (1e-15 of the
largest value), FP32 2e-7; moments 1e-13 of their scale (64 FP64 additions)."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nv", [1, 5, 32, 64])
def test_either_side_of_the_line(precision, nv):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    line = 512 + 128 * nv
    rng = np.random.default_rng(nv)
    f0 = rng.uniform(0.0, 1.0, (line, nv)) ** 3
    E = np.resize([0.0, 0.3, -0.3, 2.0, -2.0, 40.0, -40.0], line)
    got = []
    for nx in (line - 1, line):
        cfg = W.landau(nx=nx, nv=nv, precision=precision)
        r = AbiRunner(cfg, [f0[:nx]])
        r.eb[:, 0] = torch.as_tensor(E[:nx], device=r.dev)
        mom, again = r.mom(), r.mom()
        abi.pfc_advect_v(r.ctx, 0, 0.4, mom)
        abi.moments(r.ctx, 0, again)
        r.sync()
        assert torch.equal(mom, again)
        got.append((r.f_np(0)[:line - 1], mom.cpu().numpy()[:line - 1]))
        r.close()
    (fw, mw), (ft, mt) = got
    assert np.abs(fw - ft).max() <= (1e-15 if precision == 64 else 2e-7) * ft.max()
    vmax = 6.0
    scale = np.abs(mt[:, :1]).max() * np.array([1.0, vmax, vmax ** 2, vmax ** 3])
    assert np.all(np.abs(mw - mt) <= (1e-13 if precision == 64 else 1e-6) * scale)
