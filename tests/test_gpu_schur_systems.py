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


@pytest.mark.parametrize("precision", [0, 1])
def test_systems_of_more_unknowns_than_fit_in_registers(precision):
    """A fine contour makes the plain path's system one of more than 4096 unknowns (2 l + 2 M); the reduced
    system of the same contour stays small, and both give the same amplitudes (1e-10, as elsewhere)."""
    hbs = require_lib()
    geo = inputs.star(0.3, 0.3, 5).sample(800)
    h = hbs.Handle(*geo, 1.0, 20.0, 1e-12, hbs.default_options(precision=precision, contour_h=0.042))
    info = h.info()
    assert 4096 < 2 * info["nb_rank"] + 2 * info["m"] < 6000, (info["nb_rank"], info["m"])
    th = [-1.1, -0.6]
    assert relerr(_amplitudes(h.solve_plain(th)), _amplitudes(h.solve(th))) < 1e-10


@pytest.mark.parametrize("precision", [0, 1])
def test_a_dense_root_of_more_than_4096_unknowns(precision):
    """One leaf of 4200 nodes, a single inverse: A x = b to the bound of the library's other check of this."""
    import torch

    from gpu_util import dev
    hbs = require_lib()
    n, omega = 4200, 25.0
    geo = [dev(v) for v in inputs.wiggly(4, 0.35, 20, 0.03).sample(n)]
    h = hbs.Handle(*geo, 1.0, omega, 1e-12, hbs.default_options(leaf_size=5000, precision=precision))
    idx = torch.arange(n, device="cuda", dtype=torch.int64)
    at = torch.empty((n, n), device="cuda", dtype=torch.complex128)  # column-major: A transposed
    hbs.kernel_block(*geo, omega, 0, 0.0, idx, idx, at)
    rng = np.random.default_rng(1)
    b = dev(rng.standard_normal((3, n)) + 1j * rng.standard_normal((3, n)))
    x = torch.empty_like(b)
    h.apply_inverse(b, x, 3)
    torch.cuda.synchronize()
    assert float(torch.linalg.norm(x @ at - b) / torch.linalg.norm(b)) < 1e-10


def test_bragg_products_of_a_tensor_solver_are_double_float():
    """The amplitudes' products (gamma, the E rows' samples, xi, the wall samples) of a solver in tensor precision
    run in double-float, whatever the number of angles: the profiler's record of the phase names no tensor-core
    kernel."""
    hbs = require_lib()
    geo = inputs.wiggly(0, 0.35, 20, 0.03).sample(2000)
    h = hbs.Handle(*geo, 1.0, OMEGA, 1e-12, hbs.default_options(precision=2))
    th = np.linspace(-3.0, -0.1, 300)
    hbs.profile_reset()
    hbs.profile_enable(True)
    try:
        h.solve(th)
    finally:
        hbs.profile_enable(False)
    names = [k.split(":")[-1] for k in hbs.profile_get() if k.startswith("in:solve:bragg:")]
    assert "k_zgemm_batched_df" in names and not [n for n in names if n.startswith("k_oz")], names
