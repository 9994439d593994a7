"""The closed-form Newton fits and their hand-over to the direct kernels
(moment fitting, Sec. 2.2, Algorithm 1), through the C ABI, on a list of fits
that mixes what the closed form takes (Maxwellians resolved by the block, cut by
a face, cold), what it leaves to the direct kernels (means at a face, strongly
correlated or narrow covariances, targets no grid Maxwellian has) and empty
cells; a fit count that is no multiple of a warp.

FP32 mode: the default call against the direct kernel alone (moment_fit_wide
forced), both converge to 1e-11 n, so fitted parameters agree to 1e-8 of their
scale (the bound of the other fit tests), statuses (zero rows) and the
rescaled fluid state are the same. FP64 mode: against the oracle's fit of the
same targets, to 1e-10 of their scale at a tolerance of 1e-13 n (8^3 blocks
amplify the last digits, see test_gpu_fit_modes.py)."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W
from test_closed_form import REGIMES, maxwellians
from test_gpu_kernels import oracle_species

pytestmark = pytest.mark.gpu


def targets(sp, n, seed):
    """[n][10] raw moments on the species' box: all regimes in turn."""
    rng = np.random.default_rng(seed)
    vth = sp.vmax[0] / 5.0
    out = np.zeros((n, 10))
    kinds = sorted(REGIMES) + ["face", "narrow", "empty"]
    for c in range(n):
        kind = kinds[c % len(kinds)]
        if kind == "empty":
            continue
        spec = REGIMES.get(kind, REGIMES["sheet"])
        if kind == "narrow":
            spec = (0.1, 0.05, 0.5, 0.02)
        r = maxwellians(rng, 1, *spec)[0]
        u, th = r[10:13] * vth, r[4:10] * vth ** 2
        if kind == "face":
            u[c % 3] = 4.2 * vth
        uu = [u[0] * u[0], u[0] * u[1], u[0] * u[2], u[1] * u[1], u[1] * u[2], u[2] * u[2]]
        out[c] = r[0] * np.concatenate([[1.0], u, th + uu])
    return out


def scale_of(th):
    v = np.sqrt(np.abs(th[:, 4] + th[:, 7] + th[:, 9]))[:, None] + np.abs(th[:, 1:4]).max(axis=1, keepdims=True)
    return np.concatenate([np.abs(th[:, :1]), np.repeat(v, 3, 1), np.repeat(v * v, 6, 1)], axis=1) + 1e-300


@pytest.mark.parametrize("nv", [8, 12, 16, 20, 24])
@pytest.mark.parametrize("precision", [32, 64])
def test_default_fits_equal_the_direct_ones(orc, precision, nv):
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    cfg = W.harris(nx=17, ny=5, nv=nv, lx=0.85, ly=0.25, precision=precision)
    if precision == 64:
        cfg.fit_tol = 1e-13
    nc, k = cfg.ncell, 1
    sp = cfg.species[k]
    V = np.concatenate([targets(sp, nc, 61), np.zeros((nc, 10))], axis=1)
    F = targets(sp, nc, 62) * 1.01
    r = AbiRunner(cfg, [np.zeros((nc, nv ** 3), dtype=np.float32)] * 2, fluid=np.stack([F, F]))
    vm = torch.as_tensor(V, device=r.dev)
    got = {}
    for wide in (None, 1) if precision == 32 else (None,):
        r.fluid[k].copy_(torch.as_tensor(F))
        abi.moment_fit_wide(r.ctx, k, wide)
        th = [torch.full((nc, 10), float("nan"), dtype=torch.float64, device=r.dev) for _ in range(2)]
        abi.vl_reset_stats(r.ctx)
        abi.moment_fit_solve(r.ctx, k, vm, False, *th)
        r.sync()
        got[wide] = [t.cpu().numpy() for t in th], r.fluid[k].cpu().numpy(), abi.vl_read_stats(r.ctx)
    (tv, tf), fl, st = got[None]
    if precision == 32:
        (dv, df), dfl, dst = got[1]
        assert np.array_equal(fl, dfl)
        assert st[1] == dst[1] and st[3] == dst[3], (st, dst)
        for a, b in ((tv, dv), (tf, df)):
            assert np.array_equal(a[:, 0] == 0.0, b[:, 0] == 0.0)
            assert np.all(np.abs(a - b) <= 1e-8 * scale_of(b)), np.max(np.abs(a - b) / scale_of(b))
    else:
        s = oracle_species(orc, sp)
        for t, th in ((V[:, :10], tv), (fl, tf)):
            ref, ok = np.zeros((nc, 10)), np.zeros(nc, bool)
            for c in range(nc):
                if t[c, 0] > 0.0:
                    ref[c], _, stt = orc.maxent_fit(np.ascontiguousarray(t[c]), s, 3, cfg.fit_tol, cfg.fit_max_iter)
                    ok[c] = stt == 0
                else:
                    assert np.all(th[c] == 0.0)
            assert ok.sum() > nc // 2
            assert np.all(np.abs(th - ref)[ok] <= 1e-10 * scale_of(ref)[ok]), np.max((np.abs(th - ref) / scale_of(ref))[ok])
    r.close()
