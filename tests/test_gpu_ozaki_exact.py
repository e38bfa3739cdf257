"""The tensor-core product against its own definition in integers: with alpha = 1 and beta = 0 every
step up to the last (scaling, balanced 7-bit digits, level sums over 224 values of k, 64-bit sums)
is exact and the result is rounded to FP64 once, so it must agree with the integer arithmetic to
the bit.  Sizes sit at the edges of the tiles (128 x 32), stages (16 k) and periods (224 k).  Few tiles
with k >= 4096 are split along k, here into single periods; each part is rounded once and the parts
are added in FP64 in order."""
import numpy as np
import pytest

from gpu_util import dev, require_lib

pytestmark = pytest.mark.gpu


def _digits(x, e):
    """The seven digits (leading axis) of x 2^-e as integers; |x| < 2^e."""
    mant, ex = np.frexp(x)
    mag = np.array([int(abs(m) * 2 ** 53) for m in mant.ravel()], dtype=object)
    sh = 4 + (np.asarray(e) - ex).ravel()  # 53 bits to 49
    m = np.array([0 if s > 63 else (g + (1 << int(s - 1))) >> int(s) for g, s in zip(mag, sh)], dtype=object)
    m = np.where(x.ravel() < 0, -m, m) + sum(64 << (7 * i) for i in range(6))
    q = [((m >> (7 * (6 - i))) & 127) - 64 if i else m >> 42 for i in range(7)]
    return np.array(q, dtype=np.int64).reshape((7,) + x.shape)


def _exponents(a):
    mx = np.maximum(np.abs(a.real).max(axis=1), np.abs(a.imag).max(axis=1))
    return np.where(mx == 0.0, 0, np.frexp(mx)[1])


def _product(a, b, part=None):
    """The product that the kernel defines; a is m x k, b is k x n, split into parts of `part` k."""
    ea, eb = _exponents(a), _exponents(b.T)
    d = [_digits(p, ea[:, None] + np.zeros(p.shape, int)) for p in (a.real, a.imag)]
    f = [_digits(p, eb[None, :] + np.zeros(p.shape, int)) for p in (b.real, b.imag)]
    k = a.shape[1]
    if part:
        total = np.zeros((a.shape[0], b.shape[1]), dtype=np.complex128)
        for k0 in range(0, k, part):
            ks = slice(k0, k0 + part)
            total = total + _levels([x[:, :, ks] for x in d], [x[:, ks] for x in f], ea, eb)
        return total
    return _levels(d, f, ea, eb)


def _levels(d, f, ea, eb):
    out = []
    for pairs in (((0, 0, 1), (1, 1, -1)), ((0, 1, 1), (1, 0, 1))):
        v = np.zeros((d[0].shape[1], f[0].shape[2]), dtype=object)
        for lev in range(7):
            s = sum(sg * (d[x][i] @ f[y][lev - i]) for i in range(lev + 1) for x, y, sg in pairs)
            v = v + s.astype(object) * (1 << (7 * (6 - lev)))
        # one rounding: an integer to the nearest FP64 value, then an exact scaling
        out.append(np.ldexp(v.astype(np.float64), ea[:, None] + eb[None, :] - 56))
    return out[0] + 1j * out[1]


def _run(hbs, a, b, trans):
    import torch
    (m, k), n = a.shape, b.shape[1]
    st = a.T if trans else a  # stored k x m, or m x k, by columns
    c = dev(np.zeros(m * n, dtype=np.complex128))
    hbs.zgemm(m, n, k, 1.0, dev(np.asfortranarray(st).ravel(order="F")), k if trans else m, trans,
              dev(np.asfortranarray(b).ravel(order="F")), k, 0.0, c, m, hbs.PRECISION_TENSOR)
    torch.cuda.synchronize()
    return c.cpu().numpy().reshape((n, m)).T


@pytest.mark.parametrize("m,n,k,trans", [(48, 8, 96, 0), (49, 33, 223, 1), (128, 32, 224, 0), (129, 31, 225, 1),
                                         (130, 9, 449, 0), (60, 40, 4500, 1)])
def test_tensor_product_equals_its_integers(m, n, k, trans):
    hbs = require_lib()
    rng = np.random.default_rng(m * n + k)
    a = rng.standard_normal((m, k)) + 1j * rng.standard_normal((m, k))
    b = rng.standard_normal((k, n)) + 1j * rng.standard_normal((k, n))
    a *= 2.0 ** rng.integers(-40, 40, (m, 1)) * 2.0 ** rng.integers(-30, 1, (m, k))
    b *= 2.0 ** rng.integers(-40, 40, (1, n))
    a[3], b[:, 5] = 0.0, 0.0
    assert np.array_equal(_run(hbs, a, b, trans), _product(a, b, 224 if k >= 4096 else None))


@pytest.mark.parametrize("sign", [1, -1])
def test_level_sums_at_their_largest(sign):
    """Every digit at 63 (127 for the first) and all products of one sign: the level sums pass 2^23
    and stay below 2^24, the limit of exact FP32 accumulation."""
    hbs = require_lib()
    x = sum(q << (7 * (6 - i)) for i, q in enumerate((127,) + (63,) * 6)) * 2.0 ** -49
    a = np.full((128, 448), x * (1 + 1j))
    b = np.full((448, 32), sign * x * (1 - 1j))
    b[:, 16:] = sign * x * (1 + 1j)
    assert np.array_equal(_run(hbs, a, b, 0), _product(a, b))
