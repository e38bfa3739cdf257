"""The power form of the Hankel tables (csrc/hankel_table.h, kHankelPoly and kHankelPolyDF), evaluated on the
CPU as the device does: Horner's rule, the float pairs' terms from t^7 on in FP32."""
import math

import numpy as np
import pytest

import test_hankel_table as ht


def _poly():
    T = ht._table()
    txt = open(ht.os.path.join(ht.ROOT, "paper_1301_1247_gb300", "csrc", "hankel_table.h")).read()

    def numbers(name):
        body = txt.split(name + "[", 1)[1].split("= {", 1)[1].split("};", 1)[0]
        return np.array([float(v.strip().rstrip("f")) for v in body.replace("\n", " ").split(",") if v.strip()])
    n = T["tab"].shape[0]
    T["pow"] = numbers("kHankelPoly").reshape(n, T["nd"], 4)
    T["powdf"] = numbers("kHankelPolyDF").astype(np.float32).reshape(n, T["nd"], 4, 2)
    return T


def _interval(T, z):
    i = int(T["pu"] * z)
    return i, 2.0 * (T["pu"] * z - i) - 1.0


def _eval(T, z):
    i, t = _interval(T, z)
    b = T["pow"][i, -1].copy()
    for k in range(T["nd"] - 2, -1, -1):
        b = t * b + T["pow"][i, k]
    return ht._combine(T, i, z, *b)


def _eval_df(T, z):
    i, t = _interval(T, z)
    th, tl = ht._split(t)
    out = []
    for f in range(4):
        c = T["powdf"][i, :, f]
        bh, bl = c[-1, 0], ht.F(0)
        for k in range(T["nd"] - 2, -1, -1):
            if k >= 7:
                bh = ht._fma(th, bh, c[k, 0])
            else:
                bh, bl = ht._norm(*ht._mac(th, tl, bh, bl, c[k, 0], c[k, 1]))
        out.append(float(bh) + float(bl))
    return ht._combine(T, i, z, *out)


@pytest.mark.parametrize("evaluate,bound", [(_eval, 1e-15), (_eval_df, 1e-14)])
def test_horner_matches_mpmath(evaluate, bound):
    """At random points, at interval ends and around z = 4.  The bounds: that of the Chebyshev form in FP64,
    and about 40 float-pair operations of 2^-48 each in double-float."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 30
    T = _poly()
    rng = np.random.default_rng(5)
    zs = np.concatenate([10.0 ** rng.uniform(-3, math.log10(119.9), 100), rng.uniform(4, 119.9, 100),
                         [0.5, np.nextafter(0.5, 0), 1.0, np.nextafter(4.0, 0), 4.0, 119.5, np.nextafter(120.0, 0)]])
    for z in zs:
        j0, j1, y0, y1 = evaluate(T, z)
        h0 = complex(mp.besselj(0, z) + 1j * mp.bessely(0, z))
        h1 = complex(mp.besselj(1, z) + 1j * mp.bessely(1, z))
        assert abs(complex(j0, y0) - h0) < bound * abs(h0)
        assert abs(complex(j1, y1) - h1) < bound * abs(h1)
