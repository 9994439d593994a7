"""Work counters of the 2D3V fits (vl_read_stats): a fit that the closed form begins
and leaves to the direct kernels counts the evaluations of both, and the direct
kernel's iterations. A
tolerance that nothing meets and a cap of one step make every fit one step in
either kernel, then a fallback (moment fit, Sec. 2.2)."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W
from test_gpu_closed_fit import targets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [32, 64])
def test_abandoned_attempts_are_counted(precision):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    cfg = W.harris(nx=64, ny=17, nv=16, lx=3.2, ly=0.85, precision=precision)
    cfg.fit_tol, cfg.fit_max_iter = 1e-30, 1
    nc, k = cfg.ncell, 1
    kinds = 10  # of targets(): the sheet's regime is the ninth (sorted regimes, then three more)
    t = targets(cfg.species[k], 8 * kinds, 71)
    t = t[[i for i in range(len(t)) if i % kinds == 5]]  # "sheet"
    t = t[np.arange(nc) % len(t)]
    r = AbiRunner(cfg, [np.zeros((nc, 16 ** 3), dtype=np.float32)] * 2, fluid=np.stack([t, t]))
    vm = torch.cat([torch.as_tensor(t), torch.zeros(nc, 10, dtype=torch.float64)], 1).to(r.dev)
    abi.vl_reset_stats(r.ctx)
    abi.moment_fit_solve(r.ctx, k, vm, False)
    r.sync()
    st = abi.vl_read_stats(r.ctx)
    evals = st[4] if precision == 32 else st[10]
    assert st[1] == 2 * nc and st[3] == 0
    assert st[0] == 2 * nc, st
    # at the start and after the step, in either kernel; the direct ones may form the
    # Gram sums or damp the step in further ones
    assert evals >= 2 * 2 * 2 * nc, st
    r.close()
