"""Few 2D3V fits go to the direct kernels at once (csrc/kernels.cuh, closed_first;
moment fitting, Sec. 2.2, Algorithm 1): on either side of the line the same targets
give the same fits, to the bounds of test_gpu_closed_fit.py (1e-8 of their scale at
a tolerance of 1e-11 n, 1e-10 at 1e-13 n), and the same counts of fallbacks and
invalid targets. FP32 12^3 below the line: the bits of the forced direct kernel."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W
from test_gpu_closed_fit import scale_of, targets

pytestmark = pytest.mark.gpu


def solve(precision, nv, t, nx, ny, wide=None):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    cfg = W.harris(nx=nx, ny=ny, nv=nv, lx=0.05 * nx, ly=0.05 * ny, precision=precision)
    cfg.bc_y = 0
    cfg.fit_tol = 1e-13 if precision == 64 else 1e-11
    nc, k = cfg.ncell, 1
    u = np.zeros((nc, 10))
    u[:min(nc, len(t))] = t[:nc]
    r = AbiRunner(cfg, [np.zeros((nc, nv ** 3), dtype=np.float32)] * 2, fluid=np.stack([u, u]))
    vm = torch.cat([torch.as_tensor(u), torch.zeros(nc, 10, dtype=torch.float64)], 1).to(r.dev)
    th = [torch.zeros((nc, 10), dtype=torch.float64, device=r.dev) for _ in range(2)]
    abi.moment_fit_wide(r.ctx, k, wide)
    abi.vl_reset_stats(r.ctx)
    abi.moment_fit_solve(r.ctx, k, vm, False, *th)
    r.sync()
    st = abi.vl_read_stats(r.ctx)
    out = [x.cpu().numpy() for x in th], st
    r.close()
    return out


@pytest.mark.parametrize("precision,nv,few", [(64, 12, 512), (64, 16, 512), (64, 20, 256), (64, 24, 256), (32, 12, 2048)])
def test_either_side_of_the_line(precision, nv, few):
    sp = W.harris(nx=8, ny=8, nv=nv, precision=precision).species[1]
    kinds = 10  # of targets(): the first seven are resolved by every block here
    t = targets(sp, 24 * kinds, 91)
    t = t[[i for i in range(len(t)) if i % kinds < 7]]
    (direct, sd), (closed, sc) = (solve(precision, nv, t, n, 1) for n in (few, few + 1))
    assert sd[1] == sc[1] and sd[3] + 2 == sc[3]  # one more empty cell
    bound = 1e-10 if precision == 64 else 1e-8
    for a, b in zip(direct, closed):
        a, b = a[:len(t)], b[:len(t)]
        assert np.all(np.abs(a - b) <= bound * scale_of(a)), np.max(np.abs(a - b) / scale_of(a))


def test_few_double_float_fits_have_the_direct_bits():
    sp = W.harris(nx=8, ny=8, nv=12, precision=32).species[1]
    t = targets(sp, 400, 93)
    t = t[[i for i in range(len(t)) if i % 10 == 5]]  # "sheet": the common kernel's
    (got, _), (want, _) = (solve(32, 12, t, 64, 8, wide) for wide in (None, False))
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
