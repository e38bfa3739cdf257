"""Writes hankel_table.h: piecewise Chebyshev coefficients for the Bessel functions used
by the kernel evaluations (Sec. 2.3, G = (i/4) H_0 and its normal derivative with H_1).

On each interval [i/PU, (i+1)/PU), i = 0..NI-1 (PU intervals per unit of z), four entire
functions are expanded in Chebyshev polynomials of t = 2 (PU z - i) - 1 to degree ND-1:

    J0(z),  J1(z),
    R0(z) = Y0(z) - (2/pi) (log(z/2) + gamma) J0(z),
    R1(z) = Y1(z) - (2/pi) (log(z/2) + gamma) J1(z) + 2 / (pi z),

so that Y0 and Y1 follow from the tabulated values with one logarithm (the log and pole
terms are the singular parts of Neumann's expansions).  From z = DIRECT/PU = 4 on, where
the logarithmic singularity at z = 0 is far enough away, Y0 and Y1 themselves are
tabulated instead of R0, R1 (their coefficients fall below 6e-18 from k = 11 on), so
those evaluations need neither the logarithm nor 1/z.  Each expansion is also written out as
the same polynomial in powers of t, for Horner's rule: with |t| <= 1 and coefficients that
fall like the Chebyshev ones there is no cancellation, and a term costs one multiply-add
where Clenshaw's recurrence takes two operations.  Coefficients come from
interpolation at the Chebyshev points, with the functions evaluated by mpmath at 40
significant digits; the first coefficient is stored halved (f = sum_k c_k T_k(t)).  On
intervals of width 1/2 the coefficients of all four functions fall below 2e-18 from
k = 11 on (below 2e-20 from k = 12), so 11 terms leave a truncation error far under
the FP64 rounding of values of size >= 0.1 (|H_0|, |H_1| >= sqrt(2 / (pi z)) on (0, 40)).

Run once:  python gen_hankel_table.py  (needs mpmath; the output is committed).
"""
import os

import mpmath as mp

PU = 2   # intervals per unit of z
NI = 240  # intervals covering [0, 120)
ND = 11  # coefficients per function and interval
DIRECT = 8  # first interval tabulating Y0, Y1 directly

mp.mp.dps = 40


def funcs(z, direct):
    j0, j1 = mp.besselj(0, z), mp.besselj(1, z)
    y0, y1 = mp.bessely(0, z), mp.bessely(1, z)
    if direct:
        return [j0, j1, y0, y1]
    lg = mp.log(z / 2) + mp.euler
    r0 = y0 - 2 / mp.pi * lg * j0
    r1 = y1 - 2 / mp.pi * lg * j1 + 2 / (mp.pi * z)
    return [j0, j1, r0, r1]


def coefficients(i):
    nodes = [mp.cos(mp.pi * (j + mp.mpf(1) / 2) / ND) for j in range(ND)]
    vals = [funcs((i + (t + 1) / 2) / PU, i >= DIRECT) for t in nodes]
    out = []
    for f in range(4):
        cs = []
        for k in range(ND):
            s = mp.fsum(vals[j][f] * mp.cos(k * mp.pi * (j + mp.mpf(1) / 2) / ND) for j in range(ND))
            c = 2 * s / ND
            if k == 0:
                c /= 2
            cs.append(c)
        out.append(cs)
    return out


def powers(cs):
    """Coefficients in powers of t of sum_k c_k T_k(t)."""
    t0, t1 = [mp.mpf(1)] + [mp.mpf(0)] * (ND - 1), [mp.mpf(0), mp.mpf(1)] + [mp.mpf(0)] * (ND - 2)
    out = [mp.mpf(0)] * ND
    for c in cs:
        out = [o + c * t for o, t in zip(out, t0)]
        t0, t1 = t1, [2 * a - b for a, b in zip([mp.mpf(0)] + t1[:-1], t0)]
    return out


def pair(c):
    import numpy as np
    hi = np.float32(float(c))
    return [hi, np.float32(float(c - mp.mpf(float(hi))))]


def main():
    lines = ["// Generated by gen_hankel_table.py: piecewise Chebyshev coefficients of J0, J1 and",
             "// R0 = Y0 - (2/pi)(log(z/2)+gamma) J0, R1 = Y1 - (2/pi)(log(z/2)+gamma) J1 + 2/(pi z)",
             "// (intervals i < kHankelDirect) or Y0, Y1 (i >= kHankelDirect) on [i/P, (i+1)/P),",
             "// i < kHankelIntervals, P = kHankelPerUnit, in t = 2(P z - i) - 1 (first coefficient",
             "// halved).  Layout: [interval][function][coefficient]; kHankelChebDF holds each",
             "// coefficient as a float pair (hi, lo), hi + lo = c to 2^-48.  kHankelPoly, kHankelPolyDF: the",
             "// same polynomials in powers of t, layout [interval][power][function].  The kernels read these two",
             "// only; the Chebyshev forms are what they are derived from and are checked against.",
             "#pragma once",
             f"constexpr int kHankelIntervals = {NI};",
             f"constexpr int kHankelDegree = {ND};",
             f"constexpr int kHankelPerUnit = {PU};",
             f"constexpr int kHankelDirect = {DIRECT};",
             f"static __device__ const double kHankelCheb[{NI * 4 * ND}] = {{"]
    pairs, polys = [], []
    for i in range(NI):
        cs = coefficients(i)
        for f in range(4):
            lines.append("    " + ", ".join(mp.nstr(c, 17, min_fixed=0, max_fixed=0) for c in cs[f]) + ",")
            pairs.append([v for c in cs[f] for v in pair(c)])
        ps = [powers(cs[f]) for f in range(4)]
        polys += [[ps[f][k] for f in range(4)] for k in range(ND)]
    lines.append("};")
    lines.append(f"static __device__ const float kHankelChebDF[{2 * NI * 4 * ND}] = {{")
    for row in pairs:
        lines.append("    " + ", ".join(repr(float(v)) + "f" if v != 0 else "0.0f" for v in row) + ",")
    lines.append("};")
    lines.append(f"static __device__ __align__(16) const double kHankelPoly[{NI * 4 * ND}] = {{")
    for row in polys:
        lines.append("    " + ", ".join(mp.nstr(c, 17, min_fixed=0, max_fixed=0) for c in row) + ",")
    lines.append("};")
    lines.append(f"static __device__ __align__(16) const float kHankelPolyDF[{2 * NI * 4 * ND}] = {{")
    for row in polys:
        lines.append("    " + ", ".join(repr(float(v)) + "f" if v != 0 else "0.0f" for c in row for v in pair(c)) + ",")
    lines.append("};")
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "hankel_table.h")
    with open(path, "w") as fh:
        fh.write("\n".join(lines) + "\n")


if __name__ == "__main__":
    main()
