"""The ten-moment fluid step on grids of a few rows or columns, whose tiles are 32 x 1
or 1 x 32 cells (csrc/fluid.cu, tile_shape): the cells of a wide flat grid that
repeats a narrow one have the bits of the narrow one's, which 8 x 4 tiles step (paper
Eqs. 2-4, Sec. 2.3). Values are checked against the oracle in test_gpu_fluid_tiles.py."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W
from test_gpu_closure import perturbed_state

pytestmark = pytest.mark.gpu


def step(cfg, U, EB, q, closure):
    import torch
    from paper_2109_06743_gb300 import abi
    from paper_2109_06743_gb300.driver import ClosureFluid
    sim = ClosureFluid(cfg, U, np.zeros((6, cfg.ny + 1, cfg.nx)))
    sim.eb.copy_(torch.as_tensor(EB))
    if closure:
        abi.fluid_step_closure(sim.ctx, cfg.dt)
    else:
        dev = [[torch.as_tensor(m, device=sim.dev) for m in pair] for pair in q]
        abi.fluid_step(sim.ctx, cfg.dt, [p[0] for p in dev], [p[1] for p in dev])
    torch.cuda.synchronize()
    out = sim.fluid.cpu().numpy()
    sim.close()
    return out


def grid(nx, ny, precision):
    cfg = W.orszag_tang(n=24, precision=precision)
    dx = cfg.dx
    cfg.nx, cfg.ny, cfg.lx, cfg.ly, cfg.bc_y = nx, ny, nx * dx, ny * dx, 0
    return cfg


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("closure", [False, True])
@pytest.mark.parametrize("unit,reps", [((40, 1), 251), ((37, 2), 280), ((1, 43), 240), ((3, 39), 251)])
def test_repeated_grid(precision, closure, unit, reps):
    nx, ny = unit
    along_x = nx >= ny
    small = grid(nx, ny, precision)
    big = grid(nx * reps if along_x else nx, ny if along_x else ny * reps, precision)

    def spread(a):  # [ncell][k] of the unit, repeated along its longer side
        a = a.reshape(ny, nx, -1)
        return np.ascontiguousarray(np.tile(a, (1, reps, 1) if along_x else (reps, 1, 1)).reshape(big.ncell, -1))

    U = perturbed_state(small, 31)
    EB = W.random_fields(small.ncell, 32)
    rng = np.random.default_rng(33)
    q = [[0.01 * rng.uniform(-1, 1, (small.ncell, 20)) for _ in range(2)] for _ in small.species]
    want = step(small, U, EB, q, closure)
    got = step(big, np.stack([spread(u) for u in U]), spread(EB), [[spread(m) for m in p] for p in q], closure)
    for k in range(len(small.species)):
        assert np.array_equal(got[k], spread(want[k]))
