"""The periodizer's interpolative decompositions on candidate contour nodes: the residual of all members, rebuilt
from the skeleton on a second subsample, against the tolerance that they are found to (1e-13)."""
import numpy as np
import pytest

from gpu_util import relerr, require_lib
from paper_1301_1247_gb300 import inputs

pytestmark = pytest.mark.gpu


def _qr_launches(hbs, build):
    hbs.profile_reset()
    hbs.profile_enable(True)
    try:
        h = build()
    finally:
        hbs.profile_enable(False)
    return h, hbs.profile_get()["in:build:periodizer_id:k_pqr"]["launches"]


@pytest.mark.parametrize("omega,precision", [(9.0, 0), (60.0, 2), (90.0, 1)])
@pytest.mark.parametrize("options", [dict(), dict(contour_c=0.7), dict(contour_c=4.0), dict(contour_w=1.0), dict(contour_w=6.0),
                                     dict(contour_c=4.0, contour_w=0.7), dict(contour_h=0.1), dict(contour_h=0.31)])
def test_residual_is_within_the_tolerance(omega, options, precision):
    """Wavenumbers up to 90, contours flatter, deeper, tighter and wider than the default, every, every second and
    every third node a candidate; found at the first attempt."""
    hbs = require_lib()
    geo = inputs.wiggly(0, 0.35, 20, 0.03).sample(2400)
    h, n = _qr_launches(hbs, lambda: hbs.Handle(*geo, 1.0, omega, 1e-12, hbs.default_options(precision=precision, **options)))
    assert n == 1 and 0 < h.info()["pid_residual"] < 1e-13


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_a_failed_check_repeats_the_ids_on_all_nodes(precision):
    """A second QR with every member a candidate, whose solver gives the same amplitudes (1e-10, as elsewhere)."""
    hbs = require_lib()
    geo, th = inputs.wiggly(0, 0.35, 20, 0.03).sample(2400), np.linspace(-2.9, -0.2, 7)
    opts = hbs.default_options(precision=precision)
    want = hbs.Handle(*geo, 1.0, 30.0, 1e-12, opts)
    hbs.fault_inject(hbs.INJECT_ID_RESIDUAL, 1)
    try:
        h, n = _qr_launches(hbs, lambda: hbs.Handle(*geo, 1.0, 30.0, 1e-12, opts))
    finally:
        hbs.fault_inject(hbs.INJECT_CLEAR)
    assert n == 2 and 0 < h.info()["pid_residual"] < 1e-13
    a, b = h.solve(th), want.solve(th)
    for i in range(len(th)):
        assert relerr(np.concatenate(a.bragg(i)[1:3]), np.concatenate(b.bragg(i)[1:3])) < 1e-10
