"""What is timed: the calls that a user of the library makes, over the range of sizes,
types and options that it is used with.

    listed()             the cases, each a dict of plain values
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU and the handles that a program keeps between calls
    run(state)           one pass through the public entry points, with all its outputs
    work(case)           bytes and operations that the pass cannot do without
    exact(case, seed)    the outputs in 64 bits by direct sums in plain torch (no fast method)

Keys of a case: `kind` (apply, adjoint, gradient, cross, batch, build), `precision`
(fp64, mixed), `n` points, `nvec` density vectors, `p` expansion order, `depth` of the
uniform tree (-1: chosen by the library), `leaf` target points per leaf, `adaptive` tree,
`length` of the strip in x, `points` (strip: y in [-0.9 d, -0.1 d] or the headline's
[-0.95 d, -0.05 d] when `wide`; clustered: half of them within 0.01 of y = 0), the medium
`k1 k2 k3 d`, and the walls `top` / `bottom` with `top_alpha` / `bottom_alpha`.

Mixed-precision trees take complex64 densities here, the type of their arithmetic; FP64
trees take complex128.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1902_08250_gb300 as lm

BASE = dict(kind="apply", precision="fp64", n=1000, nvec=1, p=20, depth=-1, leaf=48, adaptive=False, length=4.0,
            points="strip", wide=False, k1=1.0, k2=1.5, k3=2.0, d=1.0, top="transmission", top_alpha=0.0,
            bottom="transmission", bottom_alpha=0.0)


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The paper's experiment size in FP64, one right-hand side: launches and the depth of the
        # level sweeps decide, not throughput.
        _case("small_fp64", n=1000),
        # A few thousand points and four fields in mixed precision: the small end of batched and
        # interactive use.
        _case("small_mixed", precision="mixed", n=3000, nvec=4, p=14),
        # The headline of the benchmark: a million points, 16 fields, k2 = 8 (guided modes).
        _case("strip_mixed", precision="mixed", n=1_000_000, nvec=16, p=14, depth=5, length=20.0, wide=True, k2=8.0),
        # The same strip per unit length in FP64 at the library's own depth: the reference solution
        # that mixed results are checked against, and the form for ill-conditioned systems.
        _case("strip_fp64", n=250_000, nvec=16, length=5.0, wide=True, k2=8.0),
        # Points crowding an interface (scatterers at a surface), adaptive tree, FP64 at the least
        # order that gives 1e-10.
        _case("clustered_fp64", n=100_000, p=22, leaf=16, adaptive=True, length=10.0, points="clustered"),
        # The same in mixed precision.
        _case("clustered_mixed", precision="mixed", n=100_000, p=14, leaf=16, adaptive=True, length=10.0,
              points="clustered"),
        # One matrix-vector product of an iterative solver: mixed precision, one vector.
        _case("solver_mixed", precision="mixed", n=200_000, p=14, length=10.0),
        # Many independent media and sizes captured in one graph (parameter sweeps), 4 fields each.
        _case("batch_mixed", kind="batch", precision="mixed", n=500_000, n_lo=10_000, count=12, nvec=4, p=14,
              length=10.0),
        # Full-wave inversion step: misfit and its gradients in densities, coordinates and thickness.
        _case("gradient_fp64", kind="gradient", n=200_000, length=40.0),
        # Sources above the interface, receivers below it.
        _case("cross_fp64", kind="cross", n=20_000, nvec=2, p=22, length=6.0),
        # Adjoint apply between walls (impedance above, Neumann below).
        _case("walls_adjoint_fp64", kind="adjoint", n=30_000, nvec=2, p=22, length=6.0, top="impedance",
              top_alpha=0.7, bottom="neumann"),
        # Points that move between applies (time stepping, shape optimisation): a new tree, then
        # one apply of 4 fields on it.
        _case("build_mixed", kind="build", precision="mixed", n=100_000, nvec=4, p=14, length=10.0),
    ]


def _logn(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | rng.randrange(2)


def draw(rng: random.Random):
    """A case of the listed ranges: any kind, sizes log-uniform and odd ones among them."""
    med = dict(k1=round(rng.uniform(0.5, 2.0), 3), k2=round(rng.uniform(0.8, 8.0), 3),
               k3=round(rng.uniform(0.5, 3.0), 3), d=round(rng.uniform(0.6, 1.6), 3))
    low = dict(med, k2=round(rng.uniform(0.8, 3.0), 3))
    kind = rng.choice(["fp64", "fp64", "mixed", "mixed", "clustered", "batch", "gradient", "cross", "walls", "build"])
    nvec = rng.choice([1, 1, 2, 3, 4, 5, 8, 11, 16])
    if kind == "fp64":
        return _case(n=_logn(rng, 700, 150_000), nvec=nvec, p=rng.choice([18, 20, 22, 24]),
                     kind=rng.choice(["apply", "adjoint"]), length=round(rng.uniform(2.0, 12.0), 2),
                     wide=rng.random() < 0.5, **med)
    if kind == "mixed":
        return _case(precision="mixed", n=_logn(rng, 1500, 700_000), nvec=nvec, p=rng.choice([12, 13, 14, 14, 16]),
                     kind=rng.choice(["apply", "adjoint"]), length=round(rng.uniform(2.0, 16.0), 2),
                     wide=rng.random() < 0.5, **med)
    if kind == "clustered":
        mixed = rng.random() < 0.5
        return _case(precision="mixed" if mixed else "fp64", n=_logn(rng, 3000, 90_000), nvec=min(nvec, 4),
                     p=14 if mixed else 22, leaf=rng.choice([16, 24, 32]), adaptive=True,
                     length=round(rng.uniform(4.0, 12.0), 2), points="clustered", **low)
    if kind == "batch":
        return _case(kind="batch", precision="mixed", n=_logn(rng, 30_000, 250_000), n_lo=_logn(rng, 4000, 20_000),
                     count=rng.choice([3, 5, 6, 8]), nvec=rng.choice([2, 4, 4, 16]), p=14, length=10.0, **low)
    if kind == "gradient":
        return _case(kind="gradient", n=_logn(rng, 2000, 150_000), length=round(rng.uniform(4.0, 30.0), 2), **low)
    if kind == "cross":
        mixed = rng.random() < 0.4
        return _case(kind="cross", precision="mixed" if mixed else "fp64", n=_logn(rng, 1000, 20_000),
                     nvec=min(nvec, 4), p=14 if mixed else 22, length=round(rng.uniform(3.0, 8.0), 2), **low)
    if kind == "walls":
        mixed = rng.random() < 0.4
        top, bottom = rng.choice([("impedance", "neumann"), ("dirichlet", "transmission"), ("neumann", "dirichlet"),
                                  ("transmission", "impedance")])
        return _case(kind=rng.choice(["apply", "adjoint"]), precision="mixed" if mixed else "fp64",
                     n=_logn(rng, 2000, 30_000), nvec=min(nvec, 4), p=14 if mixed else 22,
                     length=round(rng.uniform(3.0, 8.0), 2), top=top, top_alpha=0.7, bottom=bottom, bottom_alpha=0.5,
                     **low)
    mixed = rng.random() < 0.7
    return _case(kind="build", precision="mixed" if mixed else "fp64", n=_logn(rng, 3000, 200_000),
                 nvec=min(nvec, 4), p=14 if mixed else 20, length=round(rng.uniform(3.0, 12.0), 2), **low)


# ---------------------------------------------------------------------------
# inputs and passes
# ---------------------------------------------------------------------------
def _ctype(c):
    return torch.complex64 if c["precision"] == "mixed" and c["kind"] != "cross" else torch.complex128


def _uniform(g, n, lo, hi):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * (hi - lo) + lo


def _density(g, nvec, n, dtype):
    return torch.complex(*(torch.randn(nvec, n, dtype=torch.float64, device="cuda", generator=g) for _ in "ri")).to(dtype)


def _points(c, g):
    n, d = c["n"], c["d"]
    x = _uniform(g, n, 0.0, c["length"])
    if c["points"] == "clustered":
        h = n // 2
        y = torch.cat([_uniform(g, h, -0.9 * d, -0.1 * d), -0.01 * (1.0 - _uniform(g, n - h, 0.0, 1.0))])
    else:
        e = 0.05 if c["wide"] else 0.1
        y = _uniform(g, n, (e - 1.0) * d, -e * d)
    return x, y


def _inputs(c, seed):
    """Points and densities of a case: (x, y, q), for cross (xs, ys, xt, yt, q), for batch a list."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    if c["kind"] == "batch":
        r, out = random.Random(c["count"]), []
        for i in range(c["count"]):
            n = int(c["n_lo"] * (c["n"] / c["n_lo"]) ** (i / (c["count"] - 1)))
            m = dict(c, kind="apply", n=n, k1=r.uniform(0.5, 4.0), k2=r.uniform(0.5, 4.0), k3=r.uniform(0.5, 4.0),
                     d=r.uniform(0.5, 2.0))
            x, y = _points(m, g)
            out.append((m, x, y, _density(g, c["nvec"], n, _ctype(c))))
        return out
    if c["kind"] == "cross":
        ns, nt, d = c["n"], c["n"] + c["n"] // 5, c["d"]
        xs, ys = _uniform(g, ns, 0.0, c["length"]), _uniform(g, ns, 0.05 * d, 0.95 * d)
        xt, yt = _uniform(g, nt, 0.0, c["length"]), _uniform(g, nt, -0.95 * d, -0.05 * d)
        return xs, ys, xt, yt, _density(g, c["nvec"], ns, _ctype(c))
    x, y = _points(c, g)
    q = _density(g, c["nvec"], c["n"], _ctype(c))
    if c["kind"] == "gradient":
        return x, y, q, _density(g, c["nvec"], c["n"], _ctype(c))
    return x, y, q


def _medium(c):
    return lm.create_medium(c["k1"], c["k2"], c["k3"], c["d"], p=c["p"], depth=c["depth"], leaf_target=c["leaf"],
                            precision=c["precision"], adaptive=c["adaptive"], top_bc=c["top"],
                            top_alpha=c["top_alpha"], bottom_bc=c["bottom"], bottom_alpha=c["bottom_alpha"])


def prepare(case, seed):
    c, kind = case, case["kind"]
    inp = _inputs(c, seed)
    if kind == "batch":
        trees = [lm.build_tree(_medium(m), x, y) for m, x, y, _ in inp]
        qs = [q for _, _, _, q in inp]
        us = [torch.empty_like(q) for q in qs]
        return dict(kind=kind, batch=lm.Batch(trees, qs, us), us=us)
    if kind == "cross":
        return dict(kind=kind, op=lm.build_cross(_medium(c), *inp[:4]), q=inp[4])
    if kind == "build":
        return dict(kind=kind, medium=_medium(c), x=inp[0], y=inp[1], q=inp[2])
    tree = lm.build_tree(_medium(c), inp[0], inp[1])
    if kind == "gradient":
        tree.d_tree()  # the dG/dd operator, built once per geometry
        return dict(kind=kind, tree=tree, x=inp[0], y=inp[1], q=inp[2], d=c["d"], u_obs=inp[3])
    return dict(kind=kind, tree=tree, q=inp[2])


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return lm.apply(state["tree"], state["q"])
    if kind == "adjoint":
        return lm.apply_adjoint(state["tree"], state["q"])
    if kind == "cross":
        return state["op"].apply(state["q"])
    if kind == "batch":
        state["batch"].launch()
        return state["us"]
    if kind == "build":
        return lm.apply(lm.build_tree(state["medium"], state["x"], state["y"]), state["q"])
    q, x, y = (state[k].detach().clone().requires_grad_(True) for k in ("q", "x", "y"))
    d = torch.tensor(state["d"], dtype=torch.float64, requires_grad=True)
    u = lm.green_apply(state["tree"], q, x, y, d)
    misfit = torch.sum(torch.abs(u - state["u_obs"]) ** 2)
    gq, gx, gy, gd = torch.autograd.grad(misfit, (q, x, y, d))
    return dict(u=u.detach(), gq=gq, gx=gx, gy=gy, gd=gd)


def work(case):
    """Each input read once and each output written once; the operations of the method's steps at
    their usual counts: 8 per complex multiply-add of S2M, M2M, M2L, L2L and L2T (27 translations
    per box), and 9 near leaves per target at 60 per kernel value and 8 per vector."""
    c = case
    if c["kind"] == "batch":
        sizes = [int(c["n_lo"] * (c["n"] / c["n_lo"]) ** (i / (c["count"] - 1))) for i in range(c["count"])]
    else:
        sizes = [c["n"]]
    size = 8 if _ctype(c) == torch.complex64 else 16
    np_, nv, passes = 2 * c["p"] + 1, c["nvec"], 1
    if c["kind"] == "gradient":
        passes = 5  # forward, adjoint, two target-gradient vectors, dG/dd
    flops = nbytes = 0.0
    for n in sizes:
        leaf = min(n, c["leaf"])
        boxes = 4.0 / 3.0 * n / leaf
        flops += passes * (2 * 8 * n * np_ * nv + (27 + 2) * 8 * boxes * np_ * np_ * nv + 9 * leaf * n * (60 + 8 * nv))
        nbytes += 16 * n + 2 * n * nv * size
        if c["kind"] == "gradient":
            nbytes += 2 * n * nv * size + 16 * n
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the outputs in 64 bits: direct sums over all pairs
# ---------------------------------------------------------------------------
EXACT_PAIRS = 100_000 ** 2  # more pairs than this take too long


def _gl(order):
    x, w = np.polynomial.legendre.leggauss(order)
    return torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()


def _panels(z0, z1, order=16):
    """Gauss-Legendre nodes and weights on the straight panels z0[i] -> z1[i]."""
    x, w = _gl(order)
    z0, z1 = (torch.tensor(z, dtype=torch.complex128, device="cuda") for z in (z0, z1))
    dz = (z1 - z0)[:, None]
    return (z0[:, None] + 0.5 * (x + 1.0)[None, :] * dz).reshape(-1), (0.5 * w[None, :] * dz).reshape(-1)


def _contour(ks, span, hmin):
    """Nodes on 0 -> infinity: below the real axis past every branch point and pole (all at most
    max k), then along it until e^{-lambda h} < 1e-17; e^{+-i lambda X} stays resolved and bounded
    for |X| <= span."""
    c, a = 1.5 * max(ks) + 1.0, min(0.5, 1.0 / span)
    de = min(0.25, 0.5 * min(ks))
    m = int(math.ceil((c - 2 * de) / min(a, 6.0 / span)))
    corner = [0.0] + [de - 1j * a + (c - 2 * de) * i / m for i in range(m + 1)] + [c]
    top, step = c + 39.0 / hmin, min(8.0 / span, 1.0)
    m = int(math.ceil((top - c) / step))
    corner += [c + (top - c) * (i + 1) / m for i in range(m)]
    return (*_panels(corner[:-1], corner[1:]), top)


def _s(lam, k):
    return torch.sqrt(lam * lam - k * k)  # Re s >= 0 on and below the positive real axis


def _reflection(c, side, lam, s2):
    kind, kj = (c["top"], c["k1"]) if side == 0 else (c["bottom"], c["k3"])
    if kind == "dirichlet":
        return -torch.ones_like(lam)
    if kind == "neumann":
        return torch.ones_like(lam)
    if kind == "impedance":
        b = 1j * c["k2"] * (c["top_alpha"] if side == 0 else c["bottom_alpha"])
        return (s2 + b) / (s2 - b)
    sj = _s(lam, kj)
    return (kj * kj - c["k2"] ** 2) / (s2 + sj) ** 2


def _densities(c, lam, ddd):
    """sigma_tt, sigma_bb, sigma_tb of the four image terms, or their derivatives in d."""
    s2 = _s(lam, c["k2"])
    rt, rb = _reflection(c, 0, lam, s2), _reflection(c, 1, lam, s2)
    e = rt * rb * torch.exp(-2.0 * c["d"] * s2)
    m = 1.0 / (1.0 - e)
    tt, bb, tb = rt * m, rb * m, rt * rb * m
    if ddd:  # d/dd of sigma e^{-s2 h}, h = 2d + ... for all but tt
        f = -2.0 * s2 * e * m
        tt, bb, tb = f * tt, (f - 2.0 * s2) * bb, (f - 2.0 * s2) * tb
    return s2, tt, bb, tb


def _bessel(xmax):
    """J0, W0, J1, W1 on panels of width 1 over [0, xmax] as polynomials in the offset from the
    panel's middle, [4][panel][16], where Y0 = (2/pi) ln(x/2) J0 + W0 and Y1 = (2/pi) ln(x/2) J1 -
    2/(pi x) + W1: W0 and W1 are entire.  Values from the ascending series (DLMF 10.2.2, 10.8.1)
    below 2 and from Hankel's integral (DLMF 10.9.10 turned onto the ray) by the trapezoid rule."""
    m = int(xmax) + 1
    node = np.cos(np.pi * (np.arange(16) + 0.5) / 16)
    x = (np.arange(m)[:, None] + 0.5 + 0.5 * node[None, :]).reshape(-1)
    z, lg = 0.25 * x * x, np.log(0.5 * x) * 2.0 / np.pi
    f, h, pw = 1.0, 0.0, np.where(x < 2.0, 1.0, 0.0)
    j0, w0, j1, w1 = (np.zeros_like(x) for _ in range(4))
    for i in range(24):
        j0 += f * pw
        w0 += 2.0 / np.pi * f * pw * (np.euler_gamma - h)
        j1 += 0.5 * x * f / (i + 1.0) * pw
        w1 -= 0.5 * x / np.pi * f / (i + 1.0) * pw * (2.0 * h + 1.0 / (i + 1.0) - 2.0 * np.euler_gamma)
        f, h, pw = f / (i + 1.0) ** 2, h + 1.0 / (i + 1.0), -pw * z
    far, t = x >= 2.0, 0.2 * (np.arange(34) + 0.5)
    y = x[far, None]
    r = np.sqrt(1.0 + 0.5j * t * t / y)
    e = 0.4 * np.exp(-t * t) * np.sqrt(2.0 / np.pi / y)
    h0 = np.exp(1j * (x[far] - np.pi / 4)) * (e / r).sum(1) / np.sqrt(np.pi)
    h1 = np.exp(1j * (x[far] - 3 * np.pi / 4)) * (e * t * t * r).sum(1) * 2.0 / np.sqrt(np.pi)
    j0[far], j1[far] = h0.real, h1.real
    w0[far], w1[far] = h0.imag - lg[far] * h0.real, h1.imag - lg[far] * h1.real + 2.0 / np.pi / x[far]
    C = np.polynomial.chebyshev
    to = np.stack([np.pad(C.cheb2poly(np.eye(16)[k]), (0, 15 - k)) for k in range(16)])
    vander = np.linalg.inv(C.chebvander(node, 15))
    tab = np.stack([v.reshape(m, 16) @ vander.T @ to for v in (j0, w0, j1, w1)])
    return torch.from_numpy(tab).cuda()


def _bessel_at(tab, x, order):
    """(J, Y) of the order at x > 0."""
    at = x.to(torch.int64).clamp_(max=tab.shape[1] - 1)
    t = 2.0 * (x - at) - 1.0
    out = []
    for f in tab[2 * order:2 * order + 2]:
        v = f[:, 15][at]
        for i in range(14, -1, -1):
            v = v * t + f[:, i][at]
        out.append(v)
    j, w = out
    w = w + (2.0 / math.pi) * torch.log(0.5 * x) * j
    return j, (w - (2.0 / math.pi) / x if order else w)


def _free(k, x, y, q, grad):
    """sum over j != i of (i/4) H0(k r) q_j, with its target gradient when grad."""
    n = x.numel()
    out = [torch.zeros(q.shape[0], n, dtype=torch.complex128, device="cuda") for _ in range(3 if grad else 1)]
    tab = _bessel(k * math.hypot(float(x.max() - x.min()), float(y.max() - y.min())) + 1.0)
    rows = max(1, 40_000_000 // n)
    for i in range(0, n, rows):
        dx, dy = x[i:i + rows, None] - x[None, :], y[i:i + rows, None] - y[None, :]
        r = torch.hypot(dx, dy)
        same = r == 0
        r = torch.where(same, torch.ones_like(r), r)
        jv, yv = _bessel_at(tab, k * r, 0)
        g = torch.complex(-0.25 * yv, 0.25 * jv)
        g[same] = 0
        out[0][:, i:i + rows] = q @ g.T
        if grad:
            jv, yv = _bessel_at(tab, k * r, 1)
            h = torch.complex(-0.25 * yv, 0.25 * jv) * (-k / r)
            h[same] = 0
            out[1][:, i:i + rows] = q @ (h * dx).T
            out[2][:, i:i + rows] = q @ (h * dy).T
    return out


def _reflected(c, x, y, q, grad, ddd):
    """The four image terms: on a fixed contour each is a product of a source and a target factor."""
    d, n = c["d"], x.numel()
    hmin = 2.0 * min(float((-y).min()), float((y + d).min()))
    crowd = hmin < 0.05  # pairs at the interface y = 0: their tails are added pair by pair
    span = max(float(x.max() - x.min()), 1.0)
    lam, w, top = _contour([c["k1"], c["k2"], c["k3"]], span, 0.1 if crowd else hmin)
    s2, tt, bb, tb = _densities(c, lam, ddd)
    base = w / (4.0 * math.pi * s2)
    out = [torch.zeros(q.shape[0], n, dtype=torch.complex128, device="cuda") for _ in range(3 if grad else 1)]
    step = max(16, 60_000_000 // n)
    xm = x - 0.5 * (x.max() + x.min())
    for j in range(0, lam.numel(), step):
        l, s, b = lam[j:j + step], s2[j:j + step], base[j:j + step]
        up = torch.exp(s[:, None] * y[None, :])            # source or target seen from y = 0
        dn = torch.exp(-s[:, None] * (y + d)[None, :])     # and from y = -d
        ed = torch.exp(-d * s)
        for sign in (1.0, -1.0):
            px = torch.exp(sign * 1j * l[:, None] * xm[None, :])
            a, e = (q @ (up / px).T) * b, (q @ (dn / px).T) * b
            ct = a * tt[j:j + step] + e * (tb[j:j + step] * ed)
            cb = e * bb[j:j + step] + a * (tb[j:j + step] * ed)
            tu, td = up * px, dn * px
            out[0] += ct @ tu + cb @ td
            if grad:
                il = sign * 1j * l
                out[1] += (ct * il) @ tu + (cb * il) @ td
                out[2] += (ct * s) @ tu - (cb * s) @ td
    if crowd:
        at = torch.nonzero(y > -0.1).reshape(-1)
        xc, yc, qc = x[at], y[at], q[:, at]
        # from `top` on along the direction of steepest descent; of the order 1e-6 of the field, so
        # single precision keeps it to 1e-13
        v, wv = _gl(24)
        v, wv = 0.5 * (v + 1.0), 0.5 * wv
        rows = max(1, 30_000_000 // xc.numel())
        for i in range(0, xc.numel(), rows):
            X, h = (xc[i:i + rows, None] - xc[None, :]).abs().float(), -(yc[i:i + rows, None] + yc[None, :]).float()
            rho = torch.hypot(X, h)
            e = torch.complex(h / rho, X / rho)  # e^{i phi}: i lambda X - lambda h falls as e^{-t rho}
            g = torch.zeros_like(rho)
            start = torch.exp(torch.complex(-top * h, (top * X.double()).remainder(2.0 * math.pi).float()))
            for vv, ww in zip(v.tolist(), wv.tolist()):
                t = top * vv / (1.0 - vv)
                ln = top + t * e
                # R_t e^{-s2 h} / s2 to second order in k / lambda
                more = 1.0 + (c["k2"] ** 2 + 0.5 * c["k1"] ** 2) / (ln * ln) + 0.5 * c["k2"] ** 2 * h / ln
                dens = (c["k1"] ** 2 - c["k2"] ** 2) / (4.0 * ln * ln * ln) * more
                g += (start * torch.exp(-t * rho) * dens * e).real * (ww * top / (1.0 - vv) ** 2)
            g = g.double() * (2.0 / (4.0 * math.pi))
            out[0][:, at[i:i + rows]] += qc @ g.T.to(torch.complex128)
    return out


def _fields(c, x, y, q, grad=False, ddd=False):
    out = _reflected(c, x, y, q, grad, ddd)
    return out if ddd else [a + b for a, b in zip(out, _free(c["k2"], x, y, q, grad))]


def _cross_field(c, xs, ys, xt, yt, q):
    """Layer-1 sources, middle-layer targets: u and its y-derivative continuous at y = 0 and y = -d."""
    d, hmin = c["d"], float(ys.min() - yt.max())
    span = max(float(torch.cat([xs, xt]).max() - torch.cat([xs, xt]).min()), 1.0)
    lam, w, _ = _contour([c["k1"], c["k2"], c["k3"]], span, hmin)
    s1, s2, s3 = (_s(lam, c[k]) for k in ("k1", "k2", "k3"))
    r = (s2 - s3) / (s2 + s3)
    e2 = torch.exp(-2.0 * d * s2)
    a = 2.0 / ((s1 + s2) + e2 * r * (s1 - s2)) * w / (4.0 * math.pi)
    u = torch.zeros(q.shape[0], xt.numel(), dtype=torch.complex128, device="cuda")
    step = max(16, 60_000_000 // max(xs.numel(), xt.numel()))
    for j in range(0, lam.numel(), step):
        k = slice(j, j + step)
        src = torch.exp(-s1[k, None] * ys[None, :])
        tgt = torch.exp(s2[k, None] * yt[None, :]) + r[k, None] * torch.exp(-s2[k, None] * (yt + 2.0 * d)[None, :])
        for sign in (1.0, -1.0):
            il = sign * 1j * lam[k, None]
            u += ((q @ (src * torch.exp(-il * xs[None, :])).T) * a[k]) @ (tgt * torch.exp(il * xt[None, :]))
    return u


def exact(case, seed):
    c, kind = case, case["kind"]
    inp = _inputs(c, seed)
    if kind == "batch":
        return [_fields(m, x, y, q.to(torch.complex128))[0] if m["n"] <= 30_000 else None for m, x, y, q in inp]
    if c["n"] ** 2 * (4 if kind == "gradient" else 1) > EXACT_PAIRS:
        return None
    if kind == "cross":
        return _cross_field(c, *inp)
    x, y, q = inp[0], inp[1], inp[2].to(torch.complex128)
    if kind == "adjoint":
        return _fields(c, x, y, q.conj())[0].conj().resolve_conj()
    if kind != "gradient":
        return _fields(c, x, y, q)[0]
    nv = c["nvec"]
    u, ux, uy = _fields(c, x, y, q, grad=True)
    g = 2.0 * (u - inp[3])  # of the sum of |u - u_obs|^2
    w, wx, wy = _fields(c, x, y, g.conj(), grad=True)
    ud = _fields(c, x, y, q, ddd=True)[0]
    gx, gy = ((g.conj() * a + q * b).real.sum(0) for a, b in ((ux, wx), (uy, wy)))
    return dict(u=u.reshape(nv, -1), gq=w.conj().resolve_conj(), gx=gx, gy=gy, gd=(g.conj() * ud).real.sum())
