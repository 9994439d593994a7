"""The 1D1V kernels that share a line or a group of cells among a warp's lanes, at
the sizes where the sharing is uneven: grids that are not whole groups of 6
cells (and smaller than one), velocity lines of fewer than 32, of 33 and of 64
cells, displacements of nothing, whole cells and beyond the box.

Tolerances: FP64, the same operations in another order, 1e-13 of the largest
value (1e-14 for the line update, which keeps its order); FP32 values round at
2^-24 a handful of times per step: 2e-6.
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


def parts(orc, cfg):
    sp = cfg.species[0]
    return (orc.make_grid(1, cfg.nx, 1, cfg.x0, cfg.dx), orc.make_species(sp.q, sp.m, sp.nv, sp.vmin, sp.vmax))


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx,nv", [(1, 5), (3, 31), (6, 32), (7, 33), (50, 64)])
def test_velocity_line_and_moments(gpu, orc, precision, nx, nv):
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    cfg = W.landau(nx=nx, nv=nv, precision=precision)
    rng = np.random.default_rng(nx + nv)
    f0 = rng.uniform(0.0, 1.0, (nx, nv)) ** 3
    if precision == 32:
        f0 = f0.astype(np.float32).astype(np.float64)
    r = AbiRunner(cfg, [f0])
    g, s = parts(orc, cfg)
    eb = np.zeros((nx, 6))
    eb[:, 0] = np.resize([0.0, 0.3, -0.3, 2.0, -2.0, 40.0, -40.0], nx)
    r.eb.copy_(r.torch.as_tensor(eb))
    mom = r.mom()
    abi.pfc_advect_v(r.ctx, 0, 0.4, mom)
    ref = f0.copy()
    orc.advect_velocity(ref, g, s, eb, 0.4, 5)
    got = r.f_np(0)
    assert np.abs(got - ref).max() <= (1e-14 if precision == 64 else 2e-6) * ref.max() * max(1, nv // 8)
    want = orc.moments(np.ascontiguousarray(got), g, s)
    scale = np.abs(want).max(axis=0) + want[:, :1].max()
    assert np.all(np.abs(mom.cpu().numpy() - want) <= 1e-13 * scale)
    again = r.mom()
    abi.moments(r.ctx, 0, again)
    r.sync()
    assert gpu.equal(again, mom)
    r.close()


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("nx", [2, 3, 6, 7, 11, 64])
def test_fluid_step(gpu, orc, precision, nx):
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    cfg = W.landau(nx=nx, nv=32, precision=precision)
    rng = np.random.default_rng(nx)
    f0 = W.landau_state(cfg)[0] * rng.uniform(0.9, 1.1, (nx, 1))
    f1 = f0 * rng.uniform(0.99, 1.01, (nx, 1))
    g, s = parts(orc, cfg)
    q0, q1 = orc.moments(f0, g, s), orc.moments(f1, g, s)
    eb = np.zeros((nx, 6))
    eb[:, 0] = rng.uniform(-0.1, 0.1, nx)
    U0 = np.ascontiguousarray(q0[:, :3])
    r = AbiRunner(cfg, [f0], fluid=U0[None], eb=eb)
    dt = 0.1 * cfg.dx / 6.0
    dev = [r.torch.as_tensor(q).to(r.dev) for q in (q0, q1)]
    abi.fluid_step(r.ctx, dt, [dev[0]], [dev[1]])
    r.sync()
    ref = U0.copy()
    h0, h1 = (np.ascontiguousarray(q[:, 3:]) for q in (q0, q1))  # the third moments
    orc.fluid_step(ref, g, s, h0, 0.5 * (h0 + h1), h1, eb, dt)
    assert np.abs(r.fluid[0].cpu().numpy() - ref).max() <= (1e-13 if precision == 64 else 2e-6) * np.abs(ref).max()
    r.close()
