"""Default Newton fits (moment fitting, Sec. 2.2, Algorithm 1) through the C ABI
for Maxwellians that the grid hardly resolves next to a face of the velocity box
(test_closed_form_faces.py): whichever kernel takes a fit, a converged one
reproduces its targets to fit_tol.

The residual is formed here from the returned n, u, Theta by sums over the cells (FP64,
the targets' own cancellations in extended precision), in units of the targets' thermal speeds and relative to n. Bound: fit_tol,
plus the evaluation's error (5e-13 in double-float, 2e-15 in FP64) and 16 roundings
of FP64 for theta and these sums, both times (1 + |m|)^2, m the mean of the fit
from the targets' in thermal speeds. Fits that fall back to the continuous
Maxwellian are counted by the library and miss by far more."""
import numpy as np
import pytest

from paper_2109_06743_gb300 import workloads as W
from test_closed_form_faces import EVAL, TOL, fits, near_faces  # noqa: F401

pytestmark = pytest.mark.gpu


def residuals(th, t, sp):
    """[n] largest residual of the ten moments of the discrete Maxwellians th
    against t (scaled, relative to n), and (1 + |m|)^2."""
    N = sp.nv[0]
    v = [sp.vcentres(a) for a in range(3)]
    res, grow = np.zeros(len(t)), np.zeros(len(t))
    pairs = [(a, b) for a in range(3) for b in range(a, 3)]
    for c, (k, g) in enumerate(zip(th, t)):
        # extended precision where raw moments cancel: (u / sigma)^2 is up to 400 here
        gl = g.astype(np.longdouble)
        ul = gl[1:4] / gl[0]
        cov = [gl[4 + z] / gl[0] - ul[a] * ul[b] for z, (a, b) in enumerate(pairs)]
        sl = [np.sqrt(cov[pairs.index((a, a))]) for a in range(3)]
        sg = np.array(sl, dtype=float)
        S = np.zeros((3, 3))
        for z, (a, b) in enumerate(pairs):
            S[a, b] = S[b, a] = k[4 + z] / (sg[a] * sg[b])
        m = ((k[1:4] - ul) / sl).astype(float)
        P = np.linalg.inv(S)
        w = [((v[a] - ul[a]) / sl[a]).astype(float).reshape([-1 if q == 2 - a else 1 for q in range(3)]) for a in range(3)]
        d = [w[a] - m[a] for a in range(3)]
        q = sum(P[a, b] * d[a] * d[b] for a in range(3) for b in range(3))
        h = [sp.dv[a] / sg[a] for a in range(3)]
        M = k[0] * h[0] * h[1] * h[2] / np.sqrt((2 * np.pi) ** 3 * np.linalg.det(S)) * np.exp(-0.5 * q)
        D = [M.sum()] + [(M * x).sum() for x in w] + [(M * w[a] * w[b]).sum() for a, b in pairs]
        T = [g[0]] + [0.0] * 3 + [float(gl[0] * cov[z] / (sl[a] * sl[b])) for z, (a, b) in enumerate(pairs)]
        res[c] = np.max(np.abs(np.array(D) - np.array(T))) / g[0]
        grow[c] = (1.0 + np.max(np.abs(m))) ** 2
    return res, grow


@pytest.mark.parametrize("nv", [12, 16, 20, 24])
@pytest.mark.parametrize("precision", [32, 64])
def test_converged_fits_meet_the_tolerance(fits, precision, nv):  # noqa: F811
    import torch
    from gpu_util import AbiRunner
    from paper_2109_06743_gb300 import abi
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    arith = "df2" if precision == 32 else "f64"
    # more cells than the direct kernels take at once
    cfg = W.harris(nx=128, ny=17, nv=nv, lx=6.4, ly=0.85, precision=precision)
    cfg.fit_tol = TOL[arith]
    nc, k = cfg.ncell, 1
    sp = cfg.species[k]
    scale = sp.vmax[0] / 5.0  # near_faces' box is +-5
    _, tg = near_faces(np.random.default_rng(41 * nv), 160 if nv <= 16 else 64, nv, 0.6, 1.2)
    # FP64 mode: the fits that the closed form takes (the direct sums' own cancellations,
    # 400 roundings of FP64 in this regime, are not far below its tolerance)
    mine = np.ones(len(tg), bool) if precision == 32 else fits("f64", nv, tg)[:, 0] == 1.0
    assert mine.sum() > len(tg) // 8
    tg = tg * scale ** np.array([0, 1, 1, 1, 2, 2, 2, 2, 2, 2])
    at = np.arange(nc) % len(tg)
    t = torch.as_tensor(tg[at])
    r = AbiRunner(cfg, [np.zeros((nc, nv ** 3), dtype=np.float32)] * 2, fluid=np.stack([tg[at], tg[at]]))
    vm = torch.cat([t, torch.zeros(nc, 10, dtype=torch.float64)], 1).to(r.dev)
    th = [torch.zeros((nc, 10), dtype=torch.float64, device=r.dev) for _ in range(2)]
    abi.vl_reset_stats(r.ctx)
    abi.moment_fit_solve(r.ctx, k, vm, False, *th)
    r.sync()
    st = abi.vl_read_stats(r.ctx)
    far = 0
    for x in th:
        res, grow = residuals(x[:len(tg)].cpu().numpy(), tg, sp)
        bound = cfg.fit_tol + (EVAL[arith] + 16 * 2.2e-16) * grow
        over = mine & (res > bound) & (res <= 1e-7)
        assert not over.any(), res[over]
        far += int((np.bincount(at, minlength=len(tg)) * (res > 1e-7)).sum())
    assert far == st[1], (far, st)
    assert st[3] == 0
    r.close()
