"""The closed-form evaluation of a discrete Maxwellian's moments
(csrc/closed_form.cuh: Poisson summation of the lattice, minus the cells
outside the box; the moment fit of Sec. 2.2, Algorithm 1) on the host, in both
arithmetics, against direct sums over the cells in extended precision. The
header compiles with a plain C++ compiler; FP32 operations round one by one
(no contraction), as the device's do.

Bounds, relative to the density (moments in units of the thermal speed): the
direct double-float sums are accurate to about 1e-13, the fit's tolerance is
1e-11, so 5e-13 for double-float; FP64 sums of 512 to 13824 cells round to about
1e-15, so 2e-15 for FP64 (whose parts below 1e-16 are dropped by design). The Gram
sums only steer Newton's steps: 1e-5 (both leave the doubly outside cells out).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host", "closed_form_host.cpp")


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("closed") / "closed.so")
    # the device header's includes of the CUDA runtime resolve to nothing here
    inc = tmp_path_factory.mktemp("inc")
    (inc / "cuda_runtime.h").write_text("")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(inc), SRC, "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)
    dp = np.ctypeslib.ndpointer(np.float64, flags="C_CONTIGUOUS")
    for f in (lib.closed_form_df2, lib.closed_form_f64):
        f.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_int, dp, dp]
    return lib


def maxwellians(rng, n, spread, rho, drift, temp):
    """Density, centre offset, Theta (anisotropy +-spread, correlations up to
    rho, times temp) and mean velocity (up to drift along z)."""
    rows = np.empty((n, 13))
    for r in rows:
        d = temp * (1.0 + spread * rng.uniform(-1, 1, 3))
        c = rho * rng.uniform(-1, 1, 3)
        r[0] = rng.uniform(0.05, 1.2)
        r[1:4] = 1e-3 * rng.uniform(-1, 1, 3)
        r[4:10] = [d[0], c[0] * np.sqrt(d[0] * d[1]), c[1] * np.sqrt(d[0] * d[2]), d[1], c[2] * np.sqrt(d[1] * d[2]), d[2]]
        r[10:13] = 0.1 * np.sqrt(temp) * rng.uniform(-1, 1, 3)
        r[12] += drift * rng.uniform(-1, 1)
    return rows


# (anisotropy, correlation, drift, temperature) against a box of +-5
REGIMES = {"isotropic": (0.0, 0.0, 0.0, 1.0), "sheet": (0.1, 0.05, 0.0, 1.0), "strong": (0.3, 0.3, 0.0, 1.0),
           "cut": (0.1, 0.05, 2.2, 1.0), "cold": (0.1, 0.05, 0.3, 1.0 / 3.0), "hot": (0.1, 0.05, 0.2, 1.5),
           "correlated": (0.1, 0.7, 0.0, 1.0)}


@pytest.mark.parametrize("N", [8, 12, 16, 20, 24])
@pytest.mark.parametrize("regime", sorted(REGIMES))
def test_closed_form_equals_the_direct_sums(host, N, regime):
    rng = np.random.default_rng(1000 * N + len(regime))
    rows = maxwellians(rng, 24 if N <= 16 else 8, *REGIMES[regime])
    for fn, tol in ((host.closed_form_df2, 5e-13), (host.closed_form_f64, 2e-15)):
        out = np.empty((len(rows), 3))
        fn(N, 5.0, len(rows), rows, out)
        taken = out[:, 0] == 1.0
        assert np.all(out[taken, 1] <= tol), out[taken, 1].max()
        assert np.all(out[taken, 2] <= 1e-5), out[taken, 2].max()
        if N >= 12 and regime in ("isotropic", "sheet", "cold", "cut"):
            assert taken.all()  # the workloads' Maxwellians take the closed form


def test_what_it_cannot_give_is_refused(host):
    """Means at or beyond a face, near-singular covariances and Maxwellians
    thinner than the modes kept resolve."""
    base = np.array([1.0, 0, 0, 0, 1.0, 0, 0, 1.0, 0, 1.0, 0, 0, 0])
    rows = np.tile(base, (6, 1))
    rows[0, 10] = 4.8                  # within a standard deviation of the face
    rows[1, 12] = -9.0                 # outside the box
    rows[2, 5] = 0.999                 # nearly degenerate
    rows[3, 4:10] = [0.04, 0, 0, 0.04, 0, 0.04]  # a third of a cell wide at N = 16
    rows[4, 4] = np.nan
    rows[5, 0] = np.inf
    for fn in (host.closed_form_df2, host.closed_form_f64):
        out = np.empty((6, 3))
        fn(16, 5.0, 6, np.ascontiguousarray(rows), out)
        assert np.all(out[:, 0] == 0.0), out[:, 0]
