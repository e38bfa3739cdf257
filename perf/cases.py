"""The work that users of the solver have it do, as timed cases.

Every case goes through the Python binding's public entry points.  A case is a dict of plain
values; `kind` says which path it takes:

* ``grating``: build a solver for one obstacle and solve its incident angles (the whole call);
* ``batch``:   build many small solvers at once and solve each one's angles;
* ``solve``:   the angles of a solver that is already built and resident;
* ``apply``:   the compressed inverse applied to a block of right-hand sides;
* ``gemm``:    the complex product of the dense steps, as its own entry point;
* ``inverse``: the batched inversion of per-node blocks, as its own entry point.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1301_1247_gb300 import hbs, inputs

PRECISION = {"fp64": hbs.PRECISION_FP64, "df": hbs.PRECISION_DOUBLE_FLOAT, "tensor": hbs.PRECISION_TENSOR}
D = 1.0       # grating period of every workload
W_HI = 40.0   # largest wavenumber of a batch
TOL = 1e-12   # interpolative-decomposition tolerance of every workload


# --------------------------------------------------------------------------- the cases

def listed():
    return [
        # The first call of most users: one small star, one angle, default options.  Launches and
        # host latency count here.
        dict(name="star_400", kind="grating", shape="star", n=400, omega=10.0, index=0.0, groups=1, q=1, wood=False,
             precision="fp64"),
        # An odd, ragged size at an intermediate wavenumber in double-float arithmetic, a handful
        # of angles, one of them exactly at a Wood's anomaly.
        dict(name="star_3001_df", kind="grating", shape="star", n=3001, omega=17.5, index=0.0, groups=7, q=1, wood=True,
             precision="df"),
        # The ordinary grating (wiggly obstacle, 20 unrelated angles) with every step in FP64: the
        # default options, and the mode that reference results are computed in.
        dict(name="wiggly_10k_fp64", kind="grating", shape="wiggly", n=10000, omega=30.0, index=0.0, groups=20, q=1,
             wood=True, precision="fp64"),
        # The same in the fastest mode.
        dict(name="wiggly_10k_tensor", kind="grating", shape="wiggly", n=10000, omega=30.0, index=0.0, groups=20, q=1,
             wood=True, precision="tensor"),
        # The benchmark's size: a complicated obstacle and 1000 angles in 100 groups that share a
        # Bloch phase.
        dict(name="complicated_100k", kind="grating", shape="complicated", n=100000, omega=60.0, index=0.0, groups=100,
             q=10, wood=False, precision="tensor"),
        # Dielectric obstacles: two unknowns per node, 900 angles.
        dict(name="transmission_10k", kind="grating", shape="complicated", n=10000, omega=30.0, index=1.5, groups=100,
             q=9, wood=False, precision="tensor"),
        # A parameter study: many independent gratings of mixed sizes, eight angles each.
        dict(name="batch_16", kind="batch", count=16, n_lo=400, n_hi=20000, angles=8, precision="tensor"),
        # One request to a resident solver.
        dict(name="resident_one_angle", kind="solve", shape="wiggly", n=10000, omega=30.0, index=0.0, groups=1, q=1,
             wood=False, precision="tensor"),
        # A full sweep of angles on a resident solver at the highest wavenumber in use.
        dict(name="resident_1000_angles", kind="solve", shape="complicated", n=10000, omega=60.0, index=0.0, groups=100,
             q=10, wood=False, precision="tensor"),
        # The compressed inverse as an operator: a block of right-hand sides in FP64.
        dict(name="apply_10k_x192", kind="apply", shape="wiggly", n=10000, omega=30.0, index=0.0, nrhs=192,
             precision="fp64"),
        # The largest products of the precompute, on the tensor cores.
        dict(name="gemm_690x192x100000", kind="gemm", m=690, n=192, k=100000, trans=False, precision="tensor"),
        # The per-node inversions of a middle tree level.
        dict(name="inverse_16x300", kind="inverse", n=300, count=16, precision="df"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grating"] * 6 + ["batch", "solve", "solve", "apply", "gemm", "gemm", "inverse"])
    precision = rng.choice(["fp64", "df", "tensor", "tensor"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 6 if precision == "fp64" else 12), n_lo=400, n_hi=_log(rng, 2000, 20000), angles=rng.randint(1, 12),
                    precision=precision)
    if kind == "gemm":
        k = _log(rng, 32, 100000)
        return dict(kind=kind, m=_log(rng, 16, 1500), n=_log(rng, 16, 700), k=k, trans=rng.random() < 0.4,
                    precision=precision)
    if kind == "inverse":
        n = _log(rng, 24, 1000)
        return dict(kind=kind, n=n, count=_log(rng, 1, max(2, min(1024, 40_000_000 // n ** 3 * 16 + 1))), precision=precision)
    # Complicated obstacles and dielectric ones are solved in the fastest mode.
    shape = rng.choice(["star", "wiggly", "complicated"] if precision == "tensor" else ["star", "wiggly"])
    index = rng.choice([0.0, 0.0, 0.0, 1.3, 1.5]) if kind != "apply" and precision == "tensor" else 0.0
    lo, hi = {"star": (400, 20000), "wiggly": (2000, 50000), "complicated": (8000, 100000)}[shape]
    hi = min(hi, 9000 if index else 10000 if precision == "fp64" or kind != "grating" else hi)
    n = _log(rng, lo, hi)
    omega = round(rng.uniform(8.0, 30.0 if n < 2000 or index else 60.0 if precision == "tensor" else 40.0), 3)
    c = dict(kind=kind, shape=shape, n=n, omega=omega, index=index, precision=precision)
    if kind == "apply":
        return dict(c, nrhs=_log(rng, 1, 400))
    q = rng.randint(1, max(1, min(10, int(omega * D / math.pi) - 1)))
    return dict(c, groups=_log(rng, 1, 100), q=q, wood=rng.random() < 0.5)


# --------------------------------------------------------------------------- inputs

def _obstacle(shape, seed):
    if shape == "star":
        rng = np.random.default_rng(seed)
        return inputs.star(float(rng.uniform(0.2, 0.3)), float(rng.uniform(0.1, 0.3)), int(rng.integers(3, 7)))
    return inputs.wiggly(seed, 0.35, 20, 0.03) if shape == "wiggly" else inputs.wiggly(seed, 0.3, 60, 0.05)


def _angles(case, seed):
    """Groups of q angles that share a Bloch phase (single unrelated angles for q = 1); with `wood`, the
    last one lies exactly at a Rayleigh-Wood anomaly."""
    if case["q"] > 1:
        th = inputs.bloch_grouped_angles(seed + 1, case["omega"], D, case["groups"], case["q"]).ravel()
    else:
        th = np.random.default_rng(seed + 1).uniform(-math.pi / 2 + 0.02, -0.1, case["groups"])
    if case["wood"] and len(th) > case["q"]:
        n = int(np.random.default_rng(seed + 2).integers(1, max(2, int(case["omega"] * D / math.pi))))
        th[-1] = -math.acos(1.0 - 2.0 * math.pi * n / (case["omega"] * D))
    return th


def _complex(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128)


def _options(case):
    return hbs.default_options(precision=PRECISION[case["precision"]], index=case.get("index", 0.0))


def _build(case, geom):
    return hbs.Handle(*geom, D, case["omega"], TOL, _options(case))


def prepare(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind in ("grating", "solve", "apply"):
        geom = [torch.from_numpy(a).cuda() for a in _obstacle(case["shape"], seed).sample(case["n"])]
        if kind == "grating":
            return dict(case=case, geom=geom, thetas=_angles(case, seed))
        h = _build(case, geom)
        if kind == "solve":
            return dict(case=case, handle=h, thetas=_angles(case, seed))
        b = _complex((case["nrhs"], h.unknowns), gen)
        return dict(case=case, handle=h, b=b, x=torch.empty_like(b))
    if kind == "batch":
        jobs = inputs.workload_batch(seed, case["count"], case["n_lo"], case["n_hi"], w_hi=W_HI,
                                     n_angles=case["angles"])
        return dict(case=case, geoms=[j["obstacle"].sample(j["N"]) for j in jobs], omegas=[j["omega"] for j in jobs],
                    thetas=[j["thetas"] for j in jobs])
    if kind == "gemm":  # column-major operands: torch shape (columns, rows)
        m, n, k = case["m"], case["n"], case["k"]
        a = _complex((m, k) if case["trans"] else (k, m), gen)
        return dict(case=case, a=a, b=_complex((n, k), gen), c=torch.empty((n, m), device="cuda", dtype=torch.complex128))
    # Diagonally weighted random blocks: well conditioned, as the second-kind operator's blocks are.
    n = case["n"]
    a = _complex((case["count"], n, n), gen) / math.sqrt(n) + 2.0 * torch.eye(n, device="cuda", dtype=torch.complex128)
    return dict(case=case, a=a, work=torch.empty_like(a))


# --------------------------------------------------------------------------- one pass

def _table(results, omega):
    """The Bragg amplitudes of all angles as tables over the orders -K..K that can propagate, zero where
    one does not, and each angle's range of propagating orders.  (The flux error is a rounding-level
    difference of their squares and no output of its own.)"""
    per = [r.bragg(i) for r in results for i in range(r.n)]
    k = int(omega * D / math.pi) + 1
    span = np.empty((len(per), 2), dtype=np.int64)
    refl, trans = (np.zeros((len(per), 2 * k + 1), dtype=np.complex128) for _ in range(2))
    for i, (orders, c, d, _) in enumerate(per):
        span[i] = orders[0], orders[-1]
        refl[i, orders[0] + k:orders[-1] + k + 1] = c
        trans[i, orders[0] + k:orders[-1] + k + 1] = d
    return span, refl, trans


def _amplitudes(res, case):
    """The table of the first Bloch phase's angles, and that of the others."""
    span, refl, trans = _table([res], case["omega"])
    return [dict(orders=span[part], refl=refl[part], trans=trans[part])
            for part in (slice(0, case["q"]), slice(case["q"], None)) if len(span[part])]


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "grating":
        return _amplitudes(_build(case, state["geom"]).solve(state["thetas"]), case)
    if kind == "solve":
        return _amplitudes(state["handle"].solve(state["thetas"]), case)
    if kind == "batch":
        hs = hbs.build_batch(state["geoms"], state["omegas"], D, TOL, _options(case))
        return _table([h.solve(th) for h, th in zip(hs, state["thetas"])], W_HI)
    if kind == "apply":
        state["handle"].apply_inverse(state["b"], state["x"], case["nrhs"])
        return state["x"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        hbs.zgemm(m, n, k, 1.0, state["a"], k if case["trans"] else m, int(case["trans"]), state["b"], k, 0.0, state["c"], m,
                  PRECISION[case["precision"]])
        return state["c"]
    state["work"].copy_(state["a"])  # the entry point works in place
    hbs.batched_inverse(state["work"], case["n"], case["count"], PRECISION[case["precision"]])
    return state["work"]


# --------------------------------------------------------------------------- unavoidable work

def _factor(unknowns):
    """Complex values of a compressed inverse: about three leaf-sized blocks (64) per unknown."""
    return 3 * 64 * unknowns


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=16 * (m * k + k * n + m * n), flops=8 * m * n * k)
    if kind == "inverse":
        n, c = case["n"], case["count"]
        return dict(bytes=32 * n * n * c, flops=8 * n ** 3 * c)
    if kind == "batch":
        n = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        return dict(bytes=32 * n + 16 * _factor(n), flops=24 * 64 ** 2 * n)
    unknowns = case["n"] * (2 if case["index"] else 1)
    if kind == "apply":
        return dict(bytes=16 * (_factor(unknowns) + 2 * unknowns * case["nrhs"]), flops=8 * _factor(unknowns) * case["nrhs"])
    # One reduced system per Bloch phase (about 4 omega + 190 unknowns at these wavenumbers) and its
    # angles; the whole call also forms the factor once: fill, decomposition and inversion of
    # 64-point blocks.
    r = 4 * case["omega"] + 190
    flops = case["groups"] * (8 / 3 * r ** 3 + 8 * r * r * case["q"])
    data = 16 * r * r + 16 * r * case["groups"] * case["q"]
    if kind == "grating":
        flops += 24 * 64 ** 2 * unknowns + 8 * _factor(unknowns) * r
        data += 32 * case["n"] + 16 * _factor(unknowns) + 32 * r * unknowns
    return dict(bytes=data, flops=flops)


# --------------------------------------------------------------------------- values in 64 bits

# Kapur-Rokhlin corrections of sixth order (the published table).
_GAMMA = (4.967362978287758, -16.20501504859126, 25.85153761832639, -22.22599466791883, 9.930104998037539,
          -1.817995878141594)
_MOST_UNKNOWNS = 12000  # a dense factorization of more takes too long


def _hankel(z):
    """H0 and H1 of the first kind.  Below z = 25: J_n by downward recurrence, normalised by
    1 = J_0 + 2 sum J_2k, and Neumann's series for Y_0 and Y_1.  Above: Hankel's expansion."""
    x = z.clamp(min=1e-12, max=25.0)
    zero = torch.zeros_like(x)
    up, cur, norm, y0, y1 = zero, zero + 1e-250, zero, zero, zero
    for n in range(80, 0, -1):  # cur = J_n up to a factor
        if n % 2 == 0:
            norm = norm + 2.0 * cur
            y0 = y0 - (-1) ** (n // 2) * (4.0 / math.pi / (n // 2)) * cur
        else:
            k = n // 2
            if k:
                y1 = y1 - (-1) ** k * (2.0 / math.pi) * (2 * k + 1) / (k * (k + 1)) * cur
            j1 = cur
        up, cur = cur, (2.0 * n / x) * cur - up
        big = torch.where(cur.abs() > 1e200, x.new_tensor(1e-200), x.new_tensor(1.0))
        up, cur, norm, y0, y1 = (v * big for v in (up, cur, norm, y0, y1))
    norm, j1 = norm + cur, up
    j0, j1, y0, y1 = (v / norm for v in (cur, j1, y0, y1))
    log = (2.0 / math.pi) * (torch.log(x / 2.0) + 0.57721566490153286061)
    y0, y1 = y0 + log * j0, y1 + (log - 2.0 / math.pi) * j1 - (2.0 / math.pi) * j0 / x
    far = z.clamp(min=25.0)
    out = []
    for nu, j, y in ((0, j0, y0), (1, j1, y1)):
        p, q, t = zero + 1.0, zero, zero + 1.0
        for k in range(1, 24):
            t = t * ((4 * nu * nu - (2 * k - 1) ** 2) / (8.0 * k)) / far
            if k % 2:
                q = q + (-1) ** (k // 2) * t
            else:
                p = p + (-1) ** (k // 2) * t
        c = torch.sqrt(2.0 / math.pi / far)
        ph = far - (2 * nu + 1) * math.pi / 4.0
        wave = torch.complex(ph.cos(), ph.sin()) * torch.complex(p, q) * c
        out.append(torch.where(z < 25.0, torch.complex(j, y), wave))
    return out


def _layers(t, s, k):
    """Single and double layer at wavenumber k, targets t = (x, y) by sources s = (x, y, nx, ny): the two
    values and the two gradients (S, D, (Sx, Sy), (Dx, Dy))."""
    dx, dy = t[0][:, None] - s[0][None, :], t[1][:, None] - s[1][None, :]
    r = torch.hypot(dx, dy)
    h0, h1 = _hankel(k * r)
    dn = (dx * s[2] + dy * s[3]) / r
    g, p, a = 0.25j * h0, 0.25j * k * h1 / r, 0.25j * k * k * h0 * dn / r
    return g, p * r * dn, (-p * dx, -p * dy), (a * dx + p * (s[2] - 2.0 * dx * dn / r), a * dy + p * (s[3] - 2.0 * dy * dn / r))


def _pair(case, parts):
    """The columns of one obstacle source: the combined layer D - i w S, or the interlaced pair (w S, D)."""
    s, d = parts
    if not case["index"]:
        return d - 1j * case["omega"] * s
    return torch.stack((case["omega"] * s, d), -1).reshape(s.shape[0], -1)


def _obstacle_rows(case, bd, s, d, ds, dd):
    """Rows of a field on the obstacle: its value, or interlaced minus its normal derivative / w and its value."""
    value = _pair(case, (s, d))
    if not case["index"]:
        return value
    slope = _pair(case, tuple(bd[2][:, None] * g[0] + bd[3][:, None] * g[1] for g in (ds, dd)))
    return torch.stack((-slope / case["omega"], value), 1).reshape(-1, value.shape[1])


def _boundary(case, geom):
    x, y, dx, dy = geom
    sp = torch.hypot(dx, dy)
    return x, y, dy / sp, -dx / sp, 2.0 * math.pi / len(x) * sp


def _columns(case, w):
    return w.repeat_interleave(2) if case["index"] else w


def _own_block(case, bd):
    """The Nystrom matrix of one isolated obstacle."""
    n, index = len(bd[0]), case["index"]
    i = torch.arange(n, device="cuda")
    gap = (i[:, None] - i[None, :]).abs()
    gap = torch.minimum(gap, n - gap)
    kr = torch.cat((torch.tensor((0.0,) + tuple(1.0 + g for g in _GAMMA), device="cuda", dtype=torch.float64),
                    torch.ones(1, device="cuda", dtype=torch.float64)))[gap.clamp(max=7)]
    del gap

    def part(k):
        s, d, ds, dd = _layers(bd[:2], bd[:4], k)
        return [torch.where(kr == 0.0, 0.0, v) for v in (s, d)] + [tuple(torch.where(kr == 0.0, 0.0, g) for g in v) for v in (ds, dd)]

    out = part(case["omega"])
    if index:
        other = part(index * case["omega"])
        out = [u - v if torch.is_tensor(u) else tuple(p - q for p, q in zip(u, v)) for u, v in zip(out, other)]
        kr = kr.repeat_interleave(2, 0).repeat_interleave(2, 1)
    a = _obstacle_rows(case, bd, *out) * kr * _columns(case, bd[4])[None, :]
    a.diagonal().add_(1.0 if index else 0.5)
    return a


def _shifted(bd, j):
    return bd[0] + j * D, bd[1], bd[2], bd[3]


def _bragg_exact(case, geom, thetas):
    """Bragg amplitudes of angles sharing one Bloch phase from the dense periodized system: the box
    |x| <= D/2, |y| <= h, sources on a circle around it for the far images, Rayleigh-Bloch expansions
    matched on y = +-h; least squares.  The densities are eliminated first."""
    omega, index = case["omega"], case["index"]
    bd = _boundary(case, geom)
    wq = _columns(case, bd[4])[None, :]
    f64 = dict(device="cuda", dtype=torch.float64)
    ymax = float(bd[1].abs().max())
    h, y0 = ymax + D / 8, ymax + D / 4
    rp = max(0.75 * D, 1.4 * math.hypot(D / 2, h))
    mp, kk, mw = max(100, 2 * math.ceil(omega * rp) + 60), math.ceil(omega * D / math.pi) + 40, 40
    mt, nu = 2 * (2 * kk + 1) + 8, 2 * kk + 1
    phi = 2.0 * math.pi * torch.arange(mp, **f64) / mp
    px = (rp * phi.cos(), rp * phi.sin(), phi.cos(), phi.sin())
    alpha = complex(np.exp(1j * omega * D * math.cos(thetas[0])))

    def combined(parts):
        return parts[1] - 1j * omega * parts[0]

    proxies = _layers(bd[:2], px, omega)
    rows = combined(proxies[:2])
    if index:
        slope = combined(tuple(bd[2][:, None] * g[0] + bd[3][:, None] * g[1] for g in proxies[2:]))
        rows = torch.stack((-slope / omega, rows), 1).reshape(-1, mp)
    a = _own_block(case, bd)
    for j in (-1, 1):
        a += alpha ** j * _obstacle_rows(case, bd, *_layers(bd[:2], _shifted(bd, j), omega)) * wq
    inc = []
    for t in thetas:
        kx, ky = omega * math.cos(t), omega * math.sin(t)
        u = torch.exp(1j * (kx * bd[0] + ky * bd[1]))
        inc.append(torch.stack((-1j * (kx * bd[2] + ky * bd[3]) * u / omega, u), 1).reshape(-1) if index else u)
    sol = torch.linalg.solve(a, torch.cat((rows, torch.stack(inc, 1)), 1))  # eta = -sol [c; 1]
    del a

    def layer_rows(targets, shift, der):
        s, d, ds, dd = _layers(targets, _shifted(bd, shift), omega)
        return _pair(case, (s, d) if der is None else (ds[der], dd[der])) * wq

    def proxy_rows(targets, der):
        s, d, ds, dd = _layers(targets, px, omega)
        return combined((s, d) if der is None else (ds[der], dd[der]))

    yw = torch.tensor(np.polynomial.legendre.leggauss(mw)[0] * h, **f64)
    left, right = (torch.full_like(yw, -D / 2), yw), (torch.full_like(yw, D / 2), yw)
    xt = -D / 2 + (torch.arange(mt, **f64) + 0.5) * D / mt
    n = torch.arange(-kk, kk + 1, **f64)
    kap = omega * math.cos(thetas[0]) + 2.0 * math.pi * n / D
    kn2 = omega ** 2 - kap ** 2
    kn2[kn2.abs() <= 1e-12 * omega ** 2] = 0.0
    kn = torch.sqrt(kn2.to(torch.complex128))
    waves = torch.exp(1j * xt[:, None] * kap[None, :])
    big, rhs = [], []
    for der in (None, 0):
        dens = alpha * layer_rows(left, 1, der) - layer_rows(right, -1, der) / alpha ** 2
        far = proxy_rows(left, der) - proxy_rows(right, der) / alpha
        e = dens @ sol
        big.append(torch.cat((far - e[:, :mp], torch.zeros(mw, 2 * nu, device="cuda")), 1))
        rhs.append(e[:, mp:])
    for sgn in (1.0, -1.0):
        line = (xt, torch.full_like(xt, sgn * h))
        for der in (None, 1):
            e = sum(alpha ** j * layer_rows(line, j, der) for j in (-1, 0, 1)) @ sol
            out = -(waves if der is None else waves * (1j * sgn * kn)[None, :])
            zero = torch.zeros_like(out)
            big.append(torch.cat((proxy_rows(line, der) - e[:, :mp],) + ((out, zero) if sgn > 0 else (zero, out)), 1))
            rhs.append(e[:, mp:])
    big, rhs = torch.cat(big).cpu().numpy(), torch.cat(rhs).cpu().numpy()
    scale = 1.0 / np.linalg.norm(big, axis=0)
    z = np.linalg.lstsq(big * scale, rhs, rcond=1e-15)[0] * scale[:, None]
    kn, kn2 = kn.cpu().numpy(), kn2.cpu().numpy()
    sel = np.flatnonzero(kn2 >= 0.0)
    shift = np.exp(1j * kn[sel] * (y0 - h))
    k = int(omega * D / math.pi) + 1
    span, table = np.empty((len(thetas), 2), dtype=np.int64), np.zeros((2, len(thetas), 2 * k + 1), dtype=np.complex128)
    for i, t in enumerate(thetas):
        # this angle's number of the mode that is order 0 of the first angle
        n0 = int(round(omega * (math.cos(thetas[0]) - math.cos(t)) * D / (2.0 * math.pi)))
        span[i] = sel[0] - kk + n0, sel[-1] - kk + n0
        table[0, i, sel - kk + n0 + k] = z[mp + sel, i] * shift
        table[1, i, sel - kk + n0 + k] = z[mp + nu + sel, i] * shift
    return dict(orders=span, refl=table[0], trans=table[1])


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        s = prepare(case, seed)
        a = s["a"].T if not case["trans"] else s["a"]
        return (a @ s["b"].T).T.contiguous()
    if kind == "inverse":
        return torch.linalg.inv(prepare(case, seed)["a"].transpose(1, 2)).transpose(1, 2).contiguous()
    if kind == "batch" or case["n"] * (2 if case["index"] else 1) > _MOST_UNKNOWNS:
        return None
    geom = [torch.from_numpy(v).cuda() for v in _obstacle(case["shape"], seed).sample(case["n"])]
    if kind == "apply":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        b = _complex((case["nrhs"], case["n"]), gen)
        return torch.linalg.solve(_own_block(case, _boundary(case, geom)), b.T).T.contiguous()
    thetas = _angles(case, seed)
    first = _bragg_exact(case, geom, thetas[:case["q"]])
    return [first, dict(orders=None, refl=None, trans=None)] if len(thetas) > case["q"] else [first]
