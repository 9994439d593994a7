"""The ten-moment fluid step on grids that end inside a tile, are narrower than
its halo, or are large enough for the larger tile (paper Eqs. 2-4, Sec. 2.3),
against the oracle, with walls and periodic, in both precisions and with both
third moments (from f, gradient closure). Bounds as in test_gpu_kernels.py:
1e-11 relative in FP64 mode, 1e-5 of each component's scale in FP32 mode."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W
from test_gpu_closure import perturbed_state
from test_gpu_kernels import oracle_species

pytestmark = pytest.mark.gpu

GRIDS = [(1, 3), (2, 4), (5, 3), (8, 4), (9, 5), (17, 12), (31, 9), (152, 130)]


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("bc_y", [0, 1])
@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("closure", [False, True])
def test_fluid_step_on_ragged_grids(orc, precision, bc_y, grid, closure):
    import oracle
    import torch
    from paper_2109_06743_gb300 import abi
    from paper_2109_06743_gb300.driver import ClosureFluid
    nx, ny = grid
    cfg = W.orszag_tang(n=24, precision=precision)
    dx = cfg.dx
    cfg.nx, cfg.ny, cfg.lx, cfg.ly, cfg.bc_y = nx, ny, nx * dx, ny * dx, bc_y
    U0 = perturbed_state(cfg, 21)
    EB = W.random_fields(cfg.ncell, 22)
    rng = np.random.default_rng(23)
    sim = ClosureFluid(cfg, U0, np.zeros((6, ny + 1, nx)))
    sim.eb.copy_(torch.as_tensor(EB))
    g = orc.make_grid(3, nx, ny, cfg.x0, cfg.dx, cfg.y0, cfg.dy, bc_y)
    q = [[0.01 * rng.uniform(-1, 1, (cfg.ncell, 20)) for _ in range(2)] for _ in cfg.species]
    if closure:
        abi.fluid_step_closure(sim.ctx, cfg.dt)
    else:
        dev = [[torch.as_tensor(m, device=sim.dev) for m in pair] for pair in q]
        abi.fluid_step(sim.ctx, cfg.dt, [p[0] for p in dev], [p[1] for p in dev])
    torch.cuda.synchronize()
    got = sim.fluid.cpu().numpy()
    for k, sp in enumerate(cfg.species):
        ref = np.ascontiguousarray(U0[k]).copy()
        s = oracle_species(orc, sp)
        if closure:
            orc.fluid_step_closure(ref, g, s, EB, cfg.dt, oracle.closure_chi_k0(sp.q, sp.m))
        else:
            q0, q1 = (np.ascontiguousarray(m[:, 10:]) for m in q[k])
            orc.fluid_step(ref, g, s, q0, 0.5 * (q0 + q1), q1, EB, cfg.dt)
        scale = np.abs(ref).max(axis=0, keepdims=True) + 1e-300
        rel = (np.abs(got[k] - ref) / scale).max()
        assert rel <= (1e-11 if precision == 64 else 1e-5), (k, rel)
    sim.close()
