"""The factorization kernels at the edges of their tiles: the blocked Gauss-Jordan elimination (panels of
16 or 8 columns, 64-row strips, clusters of 1 to 8 CTAs, one or two rows per thread) through
hbs_batched_inverse, and the cluster QR of the node matrices through builds whose leaves are much
smaller or larger than usual, so that matrices of every cluster size and of the all-SM path occur."""
import numpy as np
import pytest

from gpu_util import dev, relerr, require_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count,n", [(1, 1), (3, 15), (2, 16), (2, 17), (600, 33), (513, 73), (5, 64), (2, 65), (1, 129),
                                     (1, 257), (3, 511), (1, 1025), (1, 2049)])
def test_inverse_at_panel_and_cluster_edges(count, n, precision):
    """Bounds as for the library's other inverse test: the same matrices, well conditioned."""
    hbs = require_lib()
    rng = np.random.default_rng(n)
    a = rng.standard_normal((count, n, n)) + 1j * rng.standard_normal((count, n, n))
    a += 4 * np.sqrt(n) * np.eye(n)[None]
    a = a[:, rng.permutation(n), :]  # no pivot on the diagonal
    buf = dev(np.ascontiguousarray(np.transpose(a, (0, 2, 1))).ravel())
    assert hbs.batched_inverse(buf, n, count, precision) == hbs.HBS_OK
    got = np.transpose(buf.cpu().numpy().reshape(count, n, n), (0, 2, 1))
    assert relerr(got, np.linalg.inv(a)) < (1e-13 if precision == 0 else 1e-12)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("leaf", [12, 40, 150, 500])
def test_compressed_inverse_with_unusual_leaves(leaf, precision):
    """A x = b for x = A^{-1} b of the compressed inverse, with A's entries from hbs_kernel_block: the
    residual is at the decomposition tolerance (1e-12) times the levels' growth, 1e-10 as elsewhere."""
    import torch

    from paper_1301_1247_gb300 import inputs
    hbs = require_lib()
    n, omega = 1601, 25.0
    geo = [dev(v) for v in inputs.wiggly(4, 0.35, 20, 0.03).sample(n)]
    h = hbs.Handle(*geo, 1.0, omega, 1e-12, hbs.default_options(leaf_size=leaf, precision=precision))
    idx = torch.arange(n, device="cuda", dtype=torch.int64)
    at = torch.empty((n, n), device="cuda", dtype=torch.complex128)  # column-major: A transposed
    hbs.kernel_block(*geo, omega, 0, 0.0, idx, idx, at)
    rng = np.random.default_rng(leaf)
    b = dev(rng.standard_normal((3, n)) + 1j * rng.standard_normal((3, n)))
    x = torch.empty_like(b)
    h.apply_inverse(b, x, 3)
    torch.cuda.synchronize()
    assert float(torch.linalg.norm(x @ at - b) / torch.linalg.norm(b)) < 1e-10


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 72])
def test_many_small_inverses(n, precision):
    """Enough blocks for the kernel that holds a block in shared memory, at the edges of its warps and of its
    largest size in use; bounds as above.  A block of exact zeros is reported."""
    hbs = require_lib()
    rng = np.random.default_rng(100 + n)
    count = 520
    a = rng.standard_normal((count, n, n)) + 1j * rng.standard_normal((count, n, n))
    a += 4 * np.sqrt(n) * np.eye(n)[None]
    a = a[:, rng.permutation(n), :]  # no pivot on the diagonal
    buf = dev(np.ascontiguousarray(np.transpose(a, (0, 2, 1))).ravel())
    assert hbs.batched_inverse(buf, n, count, precision) == hbs.HBS_OK
    got = np.transpose(buf.cpu().numpy().reshape(count, n, n), (0, 2, 1))
    assert relerr(got, np.linalg.inv(a)) < (1e-13 if precision == 0 else 1e-12)
    a[count // 2] = 0.0
    buf = dev(np.ascontiguousarray(np.transpose(a, (0, 2, 1))).ravel())
    assert hbs.batched_inverse(buf, n, count, precision) == hbs.HBS_WARN_ILLCOND
