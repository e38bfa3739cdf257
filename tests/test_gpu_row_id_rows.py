"""hbs_row_id on matrices whose rows fill the persistent QR's shared memory to just below and above 48 KB: the
column kept there (16 bytes a row, 6144 rows at most) and the kernel's own few KB."""
import numpy as np
import pytest

from gpu_util import dev, require_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2800, 2880, 2900, 3000, 3072, 3073, 6144, 6145])
def test_rank_of_tall_matrices(m):
    """A matrix of rank 12 with columns n > 4096 (the persistent kernel's share of this entry point)."""
    import torch
    hbs = require_lib()
    rng = np.random.default_rng(m)
    n, r = 4200, 12
    a = rng.standard_normal((m, r)) + 1j * rng.standard_normal((m, r))
    b = rng.standard_normal((r, n)) + 1j * rng.standard_normal((r, n))
    mt = (dev(a) @ dev(b)).T.contiguous().ravel()  # column-major
    want = mt.clone()
    perm = torch.zeros(n, dtype=torch.int32, device="cuda")
    t = torch.zeros(m * n, dtype=torch.complex128, device="cuda")
    k = hbs.row_id(mt, m, n, 1e-12, perm, t)
    assert k == r
    cols = want.reshape(n, m)[perm.long()]  # skeleton columns first: rest = skel T
    got = t[:k * (n - k)].reshape(n - k, k) @ cols[:k]
    assert float(torch.linalg.norm(got - cols[k:]) / torch.linalg.norm(cols)) < 1e-11
