"""Blocks that hold a NaN or an infinity, through every kernel of hbs_batched_inverse: the shared-memory
one (blocks of at most 56, or of at most 72 in large batches) and the cluster elimination on one and on
several CTAs."""
import numpy as np
import pytest

from gpu_util import dev, relerr, require_lib

pytestmark = pytest.mark.gpu

SIZES = [(3, 1), (2, 40), (600, 33), (520, 72), (5, 64), (2, 130), (2, 600), (1, 1025)]


def _blocks(count, n):
    rng = np.random.default_rng(7 * n + count)
    a = rng.standard_normal((count, n, n)) + 1j * rng.standard_normal((count, n, n))
    return a + 4 * np.sqrt(n) * np.eye(n)[None]


def _inverse(hbs, a, precision):
    count, n, _ = a.shape
    buf = dev(np.ascontiguousarray(np.transpose(a, (0, 2, 1))).ravel())
    st = hbs.batched_inverse(buf, n, count, precision)
    return st, np.transpose(buf.cpu().numpy().reshape(count, n, n), (0, 2, 1))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count,n", SIZES)
def test_a_nan_of_any_payload_is_no_missing_pivot(count, n, precision):
    """A buffer filled with ones in every bit (sign and payload) has a pivot row in every column like any
    other block: the call returns, and the next one is right."""
    hbs = require_lib()
    a = _blocks(count, n)
    ref = np.linalg.inv(a)
    bad = a.copy()
    bad[count // 2] = np.full(2 * n * n, -1, np.int64).view(np.complex128).reshape(n, n)
    assert _inverse(hbs, bad, precision)[0] in (hbs.HBS_OK, hbs.HBS_WARN_ILLCOND)
    st, got = _inverse(hbs, a, precision)
    assert st == hbs.HBS_OK and relerr(got, ref) < (1e-13 if precision == 0 else 1e-12)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1j * np.inf, complex(np.nan, np.nan)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count,n", SIZES)
def test_a_block_that_is_not_finite_is_reported(count, n, precision, value):
    """One entry anywhere (on the diagonal, below it in a row already used as a pivot, in the last column) is
    enough, and the other blocks' inverses are not touched by it."""
    hbs = require_lib()
    a = _blocks(count, n)
    for i, j in {(0, 0), (n // 3, n // 6), (n // 6, n // 3), (n - 1, 0), (n // 2, n - 1)}:
        bad = a.copy()
        bad[count // 2, i, j] = value
        assert _inverse(hbs, bad, precision)[0] == hbs.HBS_WARN_ILLCOND, (i, j)


@pytest.mark.parametrize("count,n", SIZES)
def test_small_and_large_scales_are_no_fault_in_fp64(count, n):
    """Entries near 1e-150 and 1e150: their squares are still numbers, and the inverse is the scaled one."""
    hbs = require_lib()
    a = _blocks(count, n)
    ref = np.linalg.inv(a)
    for scale in (1e-150, 1e150):
        st, got = _inverse(hbs, a * scale, 0)
        assert st == hbs.HBS_OK and relerr(got * scale, ref) < 1e-13
