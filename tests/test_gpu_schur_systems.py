"""The Schur systems of the Bloch phases at the edges of their kernels' ranges: right-hand sides a system,
systems a call, unknowns a system."""
import numpy as np
import pytest

from gpu_util import relerr, require_lib
from paper_1301_1247_gb300 import inputs

pytestmark = pytest.mark.gpu

OMEGA = 60.0  # up to 19 angles share a Bloch phase


def _amplitudes(res):
    return np.concatenate([np.concatenate(res.bragg(i)[1:3]) for i in range(res.n)])


@pytest.mark.parametrize("groups,q", [(1, 1), (3, 2), (1, 3), (2, 5), (1, 6), (2, 11), (200, 1), (300, 4)])
def test_refined_double_float_solutions_match_fp64(groups, q):
    """Blocks of one to five right-hand sides a system, few and many systems: refined against the FP64 system,
    the double-float solve of a double-float solver agrees with an FP64 solver's to 1e-10, the bar of the
    library's other comparisons of the two."""
    hbs = require_lib()
    geo = inputs.wiggly(0, 0.35, 20, 0.03).sample(1600)
    th = inputs.bloch_grouped_angles(5, OMEGA, 1.0, groups, q).ravel()
    got = hbs.Handle(*geo, 1.0, OMEGA, 1e-12, hbs.default_options(precision=1)).solve(th)
    want = hbs.Handle(*geo, 1.0, OMEGA, 1e-12).solve(th)
    assert relerr(_amplitudes(got), _amplitudes(want)) < 1e-10
