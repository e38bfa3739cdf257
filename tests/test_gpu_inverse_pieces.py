"""Batches of blocks that the cluster elimination takes in pieces: more than 4096 blocks, more than 1 GB of
copies, pieces that end inside the batch; and blocks of 73 to 96 in batches that large, which the shared-memory
kernel takes."""
import numpy as np
import pytest

from gpu_util import require_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("count,n", [(4097, 80), (4097, 96), (4096, 96), (4097, 97), (4200, 100), (140, 720), (9000, 73)])
def test_inverse_in_pieces(count, n, precision):
    """A X = I for a dominant diagonal: the residual's largest entry is bounded by the arithmetic's rounding
    times n, 1e-12 with room to spare (2e-13 FP64 products, 48-bit sums of 720 terms).  A block of zeros in the last
    piece, and one in the first, are reported."""
    import torch
    hbs = require_lib()
    gen = torch.Generator(device="cuda").manual_seed(count)
    a = torch.randn((count, n, n), generator=gen, device="cuda", dtype=torch.complex128)
    a += 4 * np.sqrt(n) * torch.eye(n, device="cuda", dtype=torch.complex128)
    x = a.clone()
    assert hbs.batched_inverse(x, n, count, precision) == hbs.HBS_OK
    for part in (slice(0, 50), slice(count - 50, count)):
        assert float((a[part] @ x[part] - torch.eye(n, device="cuda")).abs().max()) < 1e-12
    del x
    for where in (0, count - 1):
        bad = a.clone()
        bad[where] = 0
        assert hbs.batched_inverse(bad, n, count, precision) == hbs.HBS_WARN_ILLCOND
        del bad


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [3585, 4096])
def test_the_largest_blocks(n, precision):
    """Two rows a thread on eight CTAs, up to the last one.  An entry of A X sums n products of about 1/4 n^-1/2, each
    within 2^-44 (a 48-bit inverse whose error grows with its pivots): n^1/2 2^-46 at random, 1e-11 with room."""
    import torch
    hbs = require_lib()
    gen = torch.Generator(device="cuda").manual_seed(n)
    a = torch.randn((1, n, n), generator=gen, device="cuda", dtype=torch.complex128)
    a += 4 * np.sqrt(n) * torch.eye(n, device="cuda", dtype=torch.complex128)
    x = a.clone()
    assert hbs.batched_inverse(x, n, 1, precision) == hbs.HBS_OK
    assert float((a[0] @ x[0] - torch.eye(n, device="cuda")).abs().max()) < 1e-11


@pytest.mark.parametrize("after", [0, 2, 6])
def test_a_full_device_halves_the_piece(after):
    """An allocation of the working copies that finds the device full: the blocks go in two pieces.  A single
    block's copy has no second chance."""
    import torch
    hbs = require_lib()
    gen = torch.Generator(device="cuda").manual_seed(3)
    a = torch.randn((9, 130, 130), generator=gen, device="cuda", dtype=torch.complex128)
    a += 4 * np.sqrt(130) * torch.eye(130, device="cuda", dtype=torch.complex128)
    try:
        x = a.clone()
        hbs.fault_inject(hbs.INJECT_DEVICE_FULL, after)
        assert hbs.batched_inverse(x, 130, 9, 1) == hbs.HBS_OK
        hbs.fault_inject(hbs.INJECT_DEVICE_FULL, after)
        with pytest.raises(hbs.HbsError) as e:
            hbs.batched_inverse(a[0].clone(), 130, 1, 1)
        assert e.value.status == hbs.HBS_ERR_OOM
    finally:
        hbs.fault_inject(hbs.INJECT_CLEAR)
    assert float((a @ x - torch.eye(130, device="cuda")).abs().max()) < 1e-12
