"""The reduced solve's batched products over angles, groups and contours, and the periodizer's IDs on
candidate contour nodes, at the edges of their ranges."""
import math

import numpy as np
import pytest

from gpu_util import relerr, require_lib
from paper_1301_1247_gb300 import inputs

pytestmark = pytest.mark.gpu

OMEGA = 30.0
NEAR_WOOD = [-math.acos(1.0 - 2.0 * math.pi * n / OMEGA) + 1e-3 for n in (1, 2, 4)]


def _geometry(n=1500):
    return inputs.wiggly(0, 0.35, 20, 0.03).sample(n)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("angles", ["one", "near_wood", "mixed"])
def test_reduced_solve_matches_the_plain_path(angles, precision):
    """One angle; angles whose contour is the shifted one; groups of one and three angles on both contours in
    turn.  Against the FP64 path that forms every group's full system: 1e-10, as for the library's
    other comparison of the two."""
    hbs = require_lib()
    geo = _geometry()
    th = {"one": [-1.1], "near_wood": NEAR_WOOD,
          "mixed": NEAR_WOOD + list(np.linspace(-3.0, -0.1, 33))
          + list(inputs.bloch_grouped_angles(5, OMEGA, 1.0, 4, 3).ravel())}[angles]
    th = np.array(th)
    got = hbs.Handle(*geo, 1.0, OMEGA, 1e-12, hbs.default_options(precision=precision)).solve(th)
    want = hbs.Handle(*geo, 1.0, OMEGA, 1e-12).solve_plain(th)
    for i in range(len(th)):
        o1, c1, d1, f1 = got.bragg(i)
        o2, c2, d2, f2 = want.bragg(i)
        assert np.array_equal(o1, o2)
        assert relerr(np.concatenate([c1, d1]), np.concatenate([c2, d2])) < 1e-10
        assert abs(f1 - f2) < 1e-9


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("contour_h", [0.05, 0.2, 0.25, 0.31, 0.7])
def test_candidate_members_at_other_contour_steps(contour_h, precision):
    """Every third, second or each node a candidate: the members rebuilt from the skeleton on the second
    subsample agree as in the library's other check of this residual."""
    hbs = require_lib()
    info = hbs.Handle(*_geometry(), 1.0, OMEGA, 1e-12,
                      hbs.default_options(precision=precision, contour_h=contour_h)).info()
    assert 0 < info["pid_residual"] < 1e-11


def test_build_and_solve_on_a_stream_of_their_own():
    """On a stream that does not order itself after the default stream, the same operations give the
    default stream's amplitudes."""
    import torch
    hbs = require_lib()
    geo, th = _geometry(600), np.linspace(-2.8, -0.4, 5)
    want = hbs.Handle(*geo, 1.0, OMEGA, 1e-12).solve(th)
    for _ in range(5):
        stream = torch.cuda.Stream()
        got = hbs.Handle(*geo, 1.0, OMEGA, 1e-12, stream=stream.cuda_stream).solve(th, stream=stream.cuda_stream)
        for i in range(len(th)):
            assert np.allclose(got.bragg(i)[1], want.bragg(i)[1], rtol=0, atol=1e-11)
            assert np.allclose(got.bragg(i)[2], want.bragg(i)[2], rtol=0, atol=1e-11)
