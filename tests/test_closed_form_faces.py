"""The closed form of the discrete moments (csrc/closed_form.cuh) and whole fits
on it (csrc/closed_newton.cuh; the moment fit of Sec. 2.2, Algorithm 1) on the
host, for Maxwellians that the grid hardly resolves and a face of the velocity
box cuts at once: 0.6 to 1.2 cells per standard deviation, a mean 1.5 to 4.5
standard deviations inside the first cell outside. There the Poisson modes of the
cells outside weigh up to 1e-4 of the density.

Bounds: evaluations as in test_closed_form.py (5e-13 of the density in
double-float, 2e-15 in FP64, against sums in extended precision). Fits that are
kept: the true residual stays within fit_tol, plus the evaluation's error times
(1 + |m|)^2 (moments about the mean m turned into moments about the targets').
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from test_closed_form import host  # noqa: F401

HERE = os.path.dirname(os.path.abspath(__file__))
EVAL = {"df2": 5e-13, "f64": 2e-15}
TOL = {"df2": 1e-11, "f64": 1e-13}


def build_fits(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fits") / "fits.so")
    inc = tmp_path_factory.mktemp("inc")
    (inc / "cuda_runtime.h").write_text("")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(inc),
                    os.path.join(HERE, "host", "closed_newton_host.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def fits(tmp_path_factory):
    lib = build_fits(tmp_path_factory)
    dp = np.ctypeslib.ndpointer(np.float64, flags="C_CONTIGUOUS")

    def run(arith, N, targets, tol=None, max_iter=20):
        out = np.zeros((len(targets), 8))
        f = getattr(lib, "closed_fit_" + arith)
        if arith == "apart":
            out = np.zeros((len(targets), 4))
        f.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int, ctypes.c_int, dp, dp]
        f(N, 5.0, TOL.get(arith, 1e-11) if tol is None else tol, max_iter, len(targets), np.ascontiguousarray(targets), out)
        return out

    return run


def near_faces(rng, n, N, lo, hi, rho=0.0):
    """n Maxwellians of lo to hi cells per standard deviation (every other one
    isotropic), three of four near a face: rows of test_closed_form.py and the raw
    moments of the discrete Maxwellian on the box of +-5."""
    dv = 10.0 / N
    v = -5.0 + (np.arange(N) + 0.5) * dv
    rows, tg = np.zeros((n, 13)), np.zeros((n, 10))
    for c in range(n):
        s = dv * np.exp(rng.uniform(np.log(lo), np.log(hi), 1 if c % 2 else 3)) * np.ones(3)
        r = rho * rng.uniform(-1, 1, 3)
        S = np.array([[s[0] ** 2, r[0] * s[0] * s[1], r[1] * s[0] * s[2]],
                      [r[0] * s[0] * s[1], s[1] ** 2, r[2] * s[1] * s[2]],
                      [r[1] * s[0] * s[2], r[2] * s[1] * s[2], s[2] ** 2]])
        u = rng.uniform(-0.5, 0.5, 3) * s
        if c % 4:
            a = rng.integers(3)
            u[a] = rng.choice([-1, 1]) * (5.0 + 0.5 * dv - rng.uniform(1.5, 4.5) * s[a])
        P = np.linalg.inv(S)
        d = [(v - u[0])[None, None, :], (v - u[1])[None, :, None], (v - u[2])[:, None, None]]
        q = sum(P[a, b] * d[a] * d[b] for a in range(3) for b in range(3))
        dens = rng.uniform(0.05, 1.2)
        M = dens * dv ** 3 / np.sqrt((2 * np.pi) ** 3 * np.linalg.det(S)) * np.exp(-0.5 * q)
        w = [v[None, None, :], v[None, :, None], v[:, None, None]]
        tg[c] = [M.sum()] + [(M * x).sum() for x in w] + [(M * w[a] * w[b]).sum() for a in range(3) for b in range(a, 3)]
        rows[c, 0], rows[c, 10:] = dens, u
        rows[c, 4:10] = [S[a, b] for a in range(3) for b in range(a, 3)]
    return rows, tg


# cells per standard deviation: FP64 mode down to where the lattice's modes beyond
# |k|^2 = 2 matter
RANGES = {"df2": (0.6, 1.2), "f64": (0.78, 1.2)}


@pytest.mark.parametrize("arith", ["df2", "f64"])
@pytest.mark.parametrize("N", [12, 16, 20, 24])
def test_evaluations_near_a_face(host, arith, N):  # noqa: F811
    rows, _ = near_faces(np.random.default_rng(31 * N), 240 if N <= 16 else 80, N, *RANGES[arith])
    out = np.zeros((len(rows), 3))
    getattr(host, "closed_form_" + arith)(N, 5.0, len(rows), rows, out)
    taken = out[:, 0] == 1.0
    assert taken.sum() > len(rows) // 8
    assert np.all(out[taken, 1] <= EVAL[arith]), out[taken, 1].max()


@pytest.mark.parametrize("arith", ["df2", "f64"])
@pytest.mark.parametrize("N", [12, 16, 20, 24])
def test_kept_fits_meet_their_tolerance(fits, arith, N):
    _, tg = near_faces(np.random.default_rng(37 * N), 240 if N <= 16 else 80, N, *RANGES[arith])
    out = fits(arith, N, tg)
    taken = out[:, 0] == 1.0
    assert taken.sum() > len(tg) // 8
    over = out[taken, 2] - TOL[arith] - EVAL[arith] * out[taken, 4]
    assert np.all(over <= 0.0), out[taken][over > 0.0]


@pytest.mark.parametrize("N", [12, 16, 20, 24])
def test_barely_resolved_in_fp64(host, fits, N):  # noqa: F811
    """0.6 to 0.78 cells per standard deviation in FP64 mode: the lattice's modes
    beyond |k|^2 = 2 weigh up to 1e-7 of the density, too much for FP32."""
    rows, tg = near_faces(np.random.default_rng(43 * N), 480 if N <= 16 else 160, N, 0.6, 0.78)
    out = np.zeros((len(rows), 3))
    host.closed_form_f64(N, 5.0, len(rows), rows, out)
    taken = out[:, 0] == 1.0
    assert taken.sum() > len(rows) // 16
    assert np.all(out[taken, 1] <= EVAL["f64"]), out[taken, 1].max()
    fit = fits("f64", N, tg)
    kept = fit[:, 0] == 1.0
    assert np.all(fit[kept, 2] <= TOL["f64"] + EVAL["f64"] * fit[kept, 4]), fit[kept, 2].max()


@pytest.mark.parametrize("N", [12, 16, 20, 24])
@pytest.mark.parametrize("cells", [(0.6, 1.2), (1.2, 2.5)])
def test_fits_lie_within_their_slack(fits, N, cells):
    """FP32 mode keeps a closed-form fit where no line parameter of the exchange can
    round otherwise within fit_slack of it: 1.5 of it for L and the means, 3 for P
    (rounds_alike). The exact fit has to lie that close, with Gram sums that leave
    out up to 1e-3 of the density too."""
    _, tg = near_faces(np.random.default_rng(47 * N), 1200 if N <= 16 else 300, N, *cells)
    out = fits("apart", N, tg)
    both = out[:, 0] == 1.0
    assert both.sum() > len(tg) // 20
    o = out[both]
    assert np.all(o[:, 1] <= 1.5 * o[:, 3]), np.max(o[:, 1] / o[:, 3])
    assert np.all(o[:, 2] <= 3.0 * o[:, 3]), np.max(o[:, 2] / o[:, 3])


@pytest.mark.parametrize("N", [12, 16, 24])
def test_heavy_corners_in_fp64(host, N):  # noqa: F811
    """Faces at 2 to 4 standard deviations along two axes, correlations up to 0.2: the
    doubly outside cells weigh up to 1e-4 of the density, partly summed in FP64 and
    partly in FP32."""
    rng = np.random.default_rng(59 * N)
    dv, n = 10.0 / N, 2000 if N <= 16 else 400
    rows = np.zeros((n, 13))
    for c, r in enumerate(rows):
        s = dv * rng.uniform(1.0, 1.0 + N / 24, 3)
        k = 0.2 * rng.uniform(-1, 1, 3) * (c % 3 > 0)
        r[0] = rng.uniform(0.05, 1.2)
        r[4:10] = [s[0] ** 2, k[0] * s[0] * s[1], k[1] * s[0] * s[2], s[1] ** 2, k[2] * s[1] * s[2], s[2] ** 2]
        u = rng.uniform(-0.5, 0.5, 3) * s
        for a in rng.permutation(3)[:2]:
            u[a] = rng.choice([-1, 1]) * (5.0 + 0.5 * dv - rng.uniform(2.0, 4.0) * s[a])
        r[10:] = u
    out = np.zeros((n, 3))
    host.closed_form_f64(N, 5.0, n, rows, out)
    taken = out[:, 0] == 1.0
    assert taken.sum() > 20
    assert np.all(out[taken, 1] <= EVAL["f64"]), out[taken, 1].max()
