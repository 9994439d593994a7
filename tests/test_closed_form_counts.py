"""Work counters of the closed-form fits (csrc/closed_newton.cuh) on the host: the
Newton steps of a start that fails are counted with those of the start that
succeeds, as the direct kernels count them (moment fit, Sec. 2.2)."""
import ctypes

import numpy as np

from test_closed_form_faces import build_fits, near_faces


def test_steps_of_a_failed_start_are_counted(tmp_path_factory):
    lib = build_fits(tmp_path_factory)
    rng = np.random.default_rng(53)
    _, tg = near_faces(rng, 200, 16, 1.2, 2.0)
    # starts off by up to 0.3: a few steps more than from the continuous Maxwellian
    dw = (0.3 * rng.uniform(-1, 1, (len(tg), 10))).astype(np.float32)
    dp = np.ctypeslib.ndpointer(np.float64, flags="C_CONTIGUOUS")
    fp = np.ctypeslib.ndpointer(np.float32, flags="C_CONTIGUOUS")
    lib.closed_fit_started.argtypes = [ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int, ctypes.c_int, dp, fp, dp]

    cap = 3
    out = np.zeros((len(tg), 7))
    lib.closed_fit_started(16, 5.0, 1e-11, cap, len(tg), np.ascontiguousarray(tg), dw, out)
    cold, started, alone = out[:, :3], out[:, 3:6], out[:, 6]
    # the start alone takes more steps than the cap: it fails after cap steps, then
    # the cold pass succeeds
    fails = (cold[:, 0] == 1.0) & (alone > cap)
    assert fails.sum() > 20
    assert np.all(started[fails, 0] == 1.0)
    assert np.all(started[fails, 1] == cap + cold[fails, 1]), started[fails]
