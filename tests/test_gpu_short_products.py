"""hbs_zgemm in tensor precision below the inner dimension at which products go to the digit planes."""
import numpy as np
import pytest

from gpu_util import dev, require_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("grade", [0, 6, 12])
@pytest.mark.parametrize("m,n,k", [(1500, 700, 32), (1500, 700, 49), (2000, 600, 95), (96, 16, 64)])
def test_short_products_are_accurate_term_by_term(m, n, k, grade, trans):
    """Columns of A that fall by `grade` decades and rows of B that rise by as many: every term has the same
    size, and each is multiplied and added within a few roundings of 2^-47, at most k of them: k 2^-46 of
    sum |a| |b| for every entry."""
    import torch
    hbs = require_lib()
    rng = np.random.default_rng(k + grade)
    fall = 10.0 ** (-grade * np.arange(k) / k)
    a = (rng.standard_normal((m, k)) + 1j * rng.standard_normal((m, k))) * fall
    b = (rng.standard_normal((k, n)) + 1j * rng.standard_normal((k, n))) / fall[:, None]
    c = dev(np.zeros(m * n, dtype=np.complex128))
    st = a.T if trans else a
    hbs.zgemm(m, n, k, 1.0, dev(np.asfortranarray(st).ravel(order="F")), k if trans else m, trans,
              dev(np.asfortranarray(b).ravel(order="F")), k, 0.0, c, m, hbs.PRECISION_TENSOR)
    torch.cuda.synchronize()
    got = c.cpu().numpy().reshape((n, m)).T
    assert (np.abs(got - a @ b) / (np.abs(a) @ np.abs(b))).max() < k * 2.0 ** -46
