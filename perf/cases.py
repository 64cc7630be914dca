"""Cases whose speed counts for a user of the reverse ray tracer.

Every case is a call (or a short chain of calls) of the public entry points on
seeded particle sets of the three kinds that the repository's workloads, tests
and benchmark use, built here on the GPU:

* ``lattice``: side^3 jittered lattice in a periodic 1 Mpc box, nearly uniform gas;
* ``halo``: n particles sampling n_H = 10 (r/kpc)^-2 cm^-3 on 1..100 kpc,
  isolated, with a self-shielded core;
* ``box``: side^3 particles sampling a log-normal density field (periodic,
  31.25 kpc mean spacing, rays of 100 kpc): clumps, filaments and voids.

Smoothing lengths hold 32 (lattice, box) or 48 (halo) neighbours of the local
density, with the few per cent of scatter that a neighbour count has.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1304_4235_gb300 as pkg
from paper_1304_4235_gb300 import autograd as AG
from paper_1304_4235_gb300 import urchin as U

DEV = "cuda"
KPC = 3.0856775814913673e21
GAMMA_THIN = 1.0e-12
L_RAY = {"lattice": 500.0, "halo": 200.0, "box": 100.0}
SIGMA_TH = 512.0 * math.pi / (3.0 * math.exp(4.0)) * 7.2973525693e-3 * math.pi * 5.29177210903e-9 ** 2


def listed():
    return [
        # one small periodic box, every origin: launches and latency count
        dict(name="columns-lattice", op="columns", kind="lattice", size=16, nside=1, origins=0, kernel="m4", f64=False),
        # columns of a whole resolved halo (long rays through a dense core)
        dict(name="columns-halo", op="columns", kind="halo", size=262144, nside=1, origins=0, kernel="m4", f64=False),
        # double-precision columns towards 48 directions from a ragged sample of origins
        dict(name="columns-box-f64", op="columns", kind="box", size=48, nside=2, origins=9973, kernel="gt", f64=True),
        # near/far split of the columns and the slab-corrected rate
        dict(name="nearfar-halo", op="nearfar", kind="halo", size=50021, nside=1, F=100, f64=False),
        # columns and their transpose (a gradient with respect to the neutral fractions)
        dict(name="columns-backward", op="columns_vjp", kind="halo", size=65536, nside=1, kernel="m4", f64=False),
        # shielded rate and ionisation equilibrium of given columns
        dict(name="rate", op="rate", rows=400003, nside=1, F=100, f64=False),
        # rate with its gradients in the columns and in the spectrum
        dict(name="rate-backward", op="rate_vjp", rows=65536, nside=1, F=200, f64=False),
        # a whole solve in double precision on the small box
        dict(name="solve-lattice-f64", op="solve", kind="lattice", size=16, nside=1, F=50, f64=True, helium=False),
        # a self-shielding halo to the paper's stopping test: hundreds of sweeps
        dict(name="solve-halo", op="solve", kind="halo", size=65536, nside=1, F=100, f64=False, helium=False),
        # fixed helium columns, 48 rays, hard spectrum
        dict(name="solve-helium", op="solve", kind="box", size=64, nside=2, F=200, f64=False, helium=True),
        # Newton-Krylov solve and the gradient of the converged state in the spectrum
        dict(name="converged-gradient", op="gradient", kind="halo", size=32768, nside=1, F=200, f64=False),
        # the benchmark box: tree build and solve of 2^24 particles
        dict(name="solve-box", op="solve", kind="box", size=256, nside=1, F=400, f64=False, helium=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["columns", "columns", "columns", "nearfar", "columns_vjp", "rate", "rate_vjp", "solve", "solve",
                     "solve", "gradient"])
    f64 = rng.random() < 0.25
    F = rng.choice([50, 100, 200, 400, 37, 141])
    if op in ("rate", "rate_vjp"):
        nside = rng.choice([1, 1, 2])
        rows = _log_int(rng, 500, (60000 if f64 or op == "rate_vjp" else 400000) // (nside * nside))
        return dict(op=op, rows=rows, nside=nside, F=F, f64=f64)
    kind = "halo" if op == "gradient" else rng.choice(["lattice", "halo", "box"])
    if kind == "halo":
        size = _log_int(rng, 1000, 24000 if f64 else (65536 if op in ("gradient", "solve", "nearfar") else 262144))
    elif kind == "lattice":
        size = rng.randint(7, 16 if f64 else 30)
    else:
        size = _log_int(rng, 12, 32 if f64 else 160)
    if op == "nearfar":
        if kind == "box":
            size = min(size, 48)
        return dict(op=op, kind=kind, size=size, nside=1, F=F, f64=f64)
    if op == "gradient":
        return dict(op=op, kind=kind, size=min(size, 8000 if f64 else size), nside=1, F=F, f64=f64)
    n = size if kind == "halo" else size ** 3
    if op == "columns_vjp":
        return dict(op=op, kind=kind, size=min(size, 120) if kind == "box" else size, nside=1,
                    kernel=rng.choice(["m4", "m4", "gt"]), f64=f64)
    if op == "columns":
        nside = rng.choice([1, 1, 2, 4]) if n < 40000 else 1
        origins = 0 if rng.random() < 0.5 else min(_log_int(rng, 1, 30000), n)
        return dict(op=op, kind=kind, size=size, nside=nside, origins=origins, kernel=rng.choice(["m4", "m4", "gt"]),
                    f64=f64)
    helium = kind != "halo" and rng.random() < 0.3
    if helium:
        size = min(size, 80)
    return dict(op=op, kind=kind, size=size, nside=1, F=F, f64=f64, helium=helium)


# ---- inputs ---------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1304 + 7919 * int(seed))


def _lattice(side, g):
    dx = 1000.0 / side
    a = (torch.arange(side, device=DEV, dtype=torch.float64) + 0.5) * dx
    p = torch.stack([v.reshape(-1) for v in torch.meshgrid(a, a, a, indexing="ij")], 1)
    p = p + (torch.rand(p.shape, generator=g, device=DEV, dtype=torch.float64) * 0.2 - 0.1) * dx
    p = torch.remainder(p, 1000.0).float()
    p[p >= 1000.0] = 0.0
    n = side ** 3
    h = dx * (3 * 32 / (4 * math.pi)) ** (1 / 3) * torch.exp(0.02 * torch.randn(n, generator=g, device=DEV))
    # moderately shielded: x_thin gives tau of a few tenths along a ray
    nH = 3.0e-4 * torch.exp(0.3 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    T = 1.0e4 * torch.exp(0.1 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    mass = nH * (1000.0 * KPC) ** 3 / n
    return p, h, mass, nH, T, True, 1000.0


def _halo(n, g):
    u = torch.rand(n, 3, generator=g, device=DEV, dtype=torch.float64)
    r = 1.0 + 99.0 * u[:, 0]
    c = 2 * u[:, 1] - 1
    s = torch.sqrt(1 - c * c)
    phi = 2 * math.pi * u[:, 2]
    p = torch.stack([r * s * torch.cos(phi), r * s * torch.sin(phi), r * c], 1).float()
    # 48 neighbours at the local number density n / (4 pi 99 r^2)
    h = (3 * 48 * 99.0 * r * r / n) ** (1 / 3) * torch.exp(0.05 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    mass = torch.full((n,), 10.0 * 4 * math.pi * 99.0 * KPC ** 3 / n, device=DEV, dtype=torch.float64)
    nH = 10.0 / (r * r)
    return p, h.float(), mass, nH, torch.full_like(nH, 1.0e4), False, 0.0


def _box(side, g):
    L = 31.25 * side
    f = torch.fft.fftfreq(side, device=DEV) * side
    z = torch.fft.rfftfreq(side, device=DEV) * side
    k2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + z[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2.clamp_min(1e-30) ** -0.625, torch.zeros_like(k2))
    d = torch.fft.irfftn(torch.fft.rfftn(torch.randn(side, side, side, generator=g, device=DEV)) * amp, s=(side,) * 3)
    d = (d - d.mean()) / d.std()
    rho = torch.exp(2.5 * d.double())
    rho = (rho / rho.mean()).reshape(-1)
    n = side ** 3
    cdf = torch.cumsum(rho, 0)
    u = torch.sort(torch.rand(n, generator=g, device=DEV, dtype=torch.float64))[0] * cdf[-1]
    cell = torch.searchsorted(cdf, u).clamp_max(n - 1)
    ci = torch.stack([cell // (side * side), (cell // side) % side, cell % side], 1)
    dx = L / side
    p = ((ci + torch.rand(n, 3, generator=g, device=DEV, dtype=torch.float64)) * dx).float()
    p[p >= L] = 0.0
    # radius holding 33 particles, from the counts in cubes of growing width
    cnt = torch.bincount(cell, minlength=n).reshape(side, side, side).float()
    h = torch.zeros(side, side, side, device=DEV)
    prev_n = prev_r = None
    for w in range(1, 16, 2):
        if w > side:
            break
        b = cnt
        for ax in range(3):
            b = sum(torch.roll(b, sh, ax) for sh in range(-(w // 2), w // 2 + 1))
        r = dx * w * (3 / (4 * math.pi)) ** (1 / 3)
        b = b.clamp_min(0.5)
        if prev_n is None:
            est = r * (33.0 / b) ** (1 / 3)
        else:
            t = (math.log(33.0) - torch.log(prev_n)) / (torch.log(b) - torch.log(prev_n)).clamp_min(1e-3)
            est = prev_r * torch.exp(t.clamp(0.0, 1.0) * math.log(r / prev_r))
        h = torch.where((h == 0) & (b >= 33), est, h)
        prev_n, prev_r = b, r
    h = torch.where(h == 0, torch.full_like(h, prev_r), h).reshape(-1)[cell]
    h = h * torch.exp(0.05 * torch.randn(n, generator=g, device=DEV))
    rc = rho[cell]
    mass = torch.full((n,), 1.0e-5 * (L * KPC) ** 3 / n, device=DEV, dtype=torch.float64)
    return p, h, mass, 1.0e-5 * rc, 1.0e4 * rc ** 0.6, True, L


def _spectrum(F, e_hi):
    edges = np.exp(np.linspace(math.log(13.6), math.log(e_hi), F + 1))
    mid = np.sqrt(edges[:-1] * edges[1:])
    s, w = U.urchin_spectrum_weights(edges, (mid / 13.6) ** -1.5, GAMMA_THIN)
    return edges, mid, torch.from_numpy(s).to(DEV), torch.from_numpy(w).to(DEV)


def _particles(case, g):
    make = {"lattice": _lattice, "halo": _halo, "box": _box}[case["kind"]]
    p, h, mass, nH, T, per, L = make(case["size"], g)
    return dict(px=p[:, 0].contiguous(), py=p[:, 1].contiguous(), pz=p[:, 2].contiguous(), h=h.contiguous(), mass=mass,
                nH=nH.contiguous(), T=T.contiguous(), periodic=per, L=L)


def _inputs(case, seed):
    """The arrays of a case, without any plan of the library."""
    g = _gen(seed)
    st = dict(case=case)
    f64 = bool(case.get("f64"))
    if "F" in case:
        st["edges"], st["mid"], st["s"], st["w"] = _spectrum(case["F"], 136.0 if case.get("helium") else 54.4)
    if case["op"] in ("rate", "rate_vjp"):
        R, m = 12 * case["nside"] ** 2, case["rows"]
        # thin to deeply shielded particles, the rays of one particle within a few dex
        c = torch.rand(m, 1, generator=g, device=DEV, dtype=torch.float64) * 8 - 5
        t = 10.0 ** (c + 0.7 * torch.randn(m, R, generator=g, device=DEV, dtype=torch.float64)).clamp(-8, 4.3)
        st["tau"] = t if f64 else t.float()
        st["nH"] = 10.0 ** (torch.rand(m, generator=g, device=DEV, dtype=torch.float64) * 6 - 5)
        st["T"] = 10.0 ** (torch.rand(m, generator=g, device=DEV, dtype=torch.float64) * 1.5 + 3.7)
        st["g_bar"] = torch.randn(m, generator=g, device=DEV, dtype=torch.float64)
        return st
    st.update(_particles(case, g))
    n = st["nH"].numel()
    st["n"], st["l"] = n, L_RAY[case["kind"]]
    st["dirs"] = U.urchin_healpix_dirs(case["nside"])
    # neutral fractions from ionised to neutral gas
    st["x"] = torch.exp(torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * math.log(1e4) - math.log(1e4))
    if case.get("origins"):
        st["org"] = torch.randperm(n, generator=g, device=DEV)[:case["origins"]].sort()[0].to(torch.int32)
    if case["op"] == "columns_vjp":
        tb = torch.randn(n, 12 * case["nside"] ** 2, generator=g, device=DEV, dtype=torch.float64)
        st["tau_bar"] = tb if f64 else tb.float()
    if case["op"] == "gradient":
        st["x_bar"] = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if case.get("helium"):
        mid = st["mid"]
        st["s1"] = torch.from_numpy(np.where(mid >= 24.59, 1.2 * (24.59 / mid) ** 2, 0.0)).to(DEV)
        st["s2"] = torch.from_numpy(U.urchin_cross_section_ratio(st["edges"], U.XSEC_HEII)).to(DEV)
        f1 = 0.3 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
        f2 = 0.5 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (1 - f1)
        st["he1"], st["he2"] = 0.079 * f1, 0.079 * f2
    return st


def _build(st):
    return U.urchin_build_bvh(st["px"], st["py"], st["pz"], st["h"], st["mass"], st["periodic"], st["L"], KPC)


def prepare(case, seed):
    st = _inputs(case, seed)
    # a solve is a step of its own and builds its tree; the other calls trace a tree in hand
    if "px" in st and case["op"] != "solve":
        st["bvh"] = _build(st)
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    prec = U.F64 if case.get("f64") else U.F32
    kern = U.KERNEL_GT if case.get("kernel") == "gt" else U.KERNEL_M4
    if op == "columns":
        return pkg.urchin_trace_columns(st["bvh"], st["x"], st["dirs"], st["l"], origins=st.get("org"), kernel=kern,
                                        precision=prec)
    if op == "nearfar":
        tf, tn = pkg.urchin_trace_columns_nearfar(st["bvh"], st["x"], st["dirs"], st["l"], precision=prec)
        g, te = pkg.urchin_gamma_nearfar(tf, tn, st["s"], st["w"], st["nH"], st["T"], slab=U.SLAB_SPECTRUM)
        return [tf, tn, g, te]
    if op == "columns_vjp":
        x = st["x"].clone().requires_grad_(True)
        tau = AG.columns(x, st["bvh"], st["dirs"], st["l"], kernel=kern, precision=prec)
        tau.backward(st["tau_bar"])
        return [tau.detach(), x.grad]
    if op == "rate":
        g, te = pkg.urchin_gamma(st["tau"], st["s"], st["w"])
        return [g, te, pkg.urchin_equilibrium(g, te, st["nH"], st["T"])]
    if op == "rate_vjp":
        tau, w = st["tau"].clone().requires_grad_(True), st["w"].clone().requires_grad_(True)
        g, te = AG.shielded_rate(tau, w, st["s"])
        g.backward(st["g_bar"])
        return [g.detach(), te, tau.grad, w.grad]
    if op == "solve":
        bvh = _build(st)
        he = dict(s_he1=st["s1"], s_he2=st["s2"], he1=st["he1"], he2=st["he2"]) if case.get("helium") else {}
        x, _ = pkg.urchin_solve(bvh, st["dirs"], st["l"], st["s"], st["w"], st["nH"], st["T"], tol=1e-3, max_iter=600,
                                segments=U.SEG_AUTO, precision=prec, raise_not_converged=False, **he)
        bvh.close()
        return x
    w = st["w"].clone().requires_grad_(True)
    x = AG.converged_x(w, st["bvh"], st["dirs"], st["l"], st["s"], st["nH"], st["T"],
                       solve_kw=dict(tol=1e-5, max_iter=400, method=U.METHOD_NEWTON, segments=U.SEG_AUTO, precision=prec,
                                     raise_not_converged=False),
                       vjp_kw=dict(tol=1e-8, max_iter=400, raise_not_converged=False))
    x.backward(st["x_bar"])
    return [x.detach(), w.grad]


# ---- work -----------------------------------------------------------------
def _hits(case):
    """Spheres crossed per ray, roughly: (number density) pi h^2 (length + 4/3 h) of a typical ray."""
    if case["kind"] == "lattice":
        return math.pi * (3 * 32 / (4 * math.pi)) ** (2 / 3) * (0.5 * case["size"] + 2.6)
    if case["kind"] == "halo":
        return 10.0 * case["size"] ** (1 / 3)
    return 85.0


def work(case):
    R = 12 * case["nside"] ** 2
    rsz = 8 if case.get("f64") else 4
    F = case.get("F", 0)
    if case["op"] in ("rate", "rate_vjp"):
        rays = case["rows"] * R
        back = case["op"] == "rate_vjp"
        # the columns in, (their gradient out,) the per-row rates; a multiply and an exponential per ray and bin
        return dict(bytes=rays * rsz * (2 if back else 1) + case["rows"] * (20 if back else 36) + 24 * F,
                    flops=rays * F * (12 if back else 4))
    n = case["size"] if case["kind"] == "halo" else case["size"] ** 3
    no = case.get("origins") or n
    rays = no * R
    # particles in (positions, h, weight), columns out; a chord integral (about 30 operations) per crossing
    b, f = n * 28 + rays * rsz, rays * _hits(case) * 30
    if case["op"] == "nearfar":
        return dict(bytes=b + rays * rsz + no * 28, flops=f + rays * F * 4)
    if case["op"] == "columns_vjp":
        return dict(bytes=2 * b + n * 8, flops=2 * f)
    if case["op"] == "columns":
        return dict(bytes=b, flops=f)
    # a solve: one pass over the crossings, two products and two folds at least
    species = 3 if case.get("helium") else 1
    return dict(bytes=n * 56 + rays * rsz * species, flops=f * species + 2 * rays * (F * 4 * species + 2 * _hits(case)))


# ---- the same outputs in 64 bits, without the library ---------------------
def _m4(b2, a1, a2):
    """int_{a1}^{a2} of the dimensionless M4 kernel at impact b2 = (b/h)^2 < 1, in closed form."""
    lb = 0.5 * torch.log(b2.clamp_min(1e-300))
    s = torch.sqrt((0.25 - b2).clamp_min(0))

    def H(a):
        m = a.abs()
        q = torch.sqrt(b2 + m * m)
        La = torch.where(b2 > 0, torch.log(m + q) - lb, torch.zeros_like(b2))
        Ls = torch.where(b2 > 0, torch.log(s + 0.5) - lb, torch.zeros_like(b2))
        inner = m * (1 - 6 * b2 - 2 * m * m) + 1.5 * m * q ** 3 + 2.25 * b2 * m * q + 2.25 * b2 * b2 * La
        outer = m * (2 + 6 * b2 + 2 * m * m) - 3 * m * q - 0.5 * m * q ** 3 - 0.75 * b2 * m * q - (3 * b2 + 0.75 * b2 * b2) * La
        join = -s * (0.25 + 6.5 * b2) + (3 * b2 + 3 * b2 * b2) * Ls
        v = torch.where(b2 < 0.25, torch.where(m <= s, inner, outer + join), outer)
        return torch.where(a >= 0, v, -v)
    return H(a2) - H(a1)


def _gt(b2, a1, a2):
    t = 2 * math.pi ** (1 / 6)
    D = math.erf(t) - 2 * t * math.exp(-t * t) / math.sqrt(math.pi)
    return math.sqrt(math.pi) / (2 * t * D) * torch.exp(-t * t * b2) * (torch.erf(t * a2) - torch.erf(t * a1))


def _pairs(st, rows, dirs, gt, split):
    """Chord integrals times A_j of origins `rows` along every direction: yields (k, row, col, value, near) of the crossings."""
    P = torch.stack([st["px"], st["py"], st["pz"]], 1).double()
    h, L, per, l = st["h"].double(), st["L"], st["periodic"], st["l"]
    A = SIGMA_TH * st["mass"] * 8 / math.pi / (h * KPC) ** 2
    O = P[rows]
    for k in range(dirs.shape[0]):
        d = torch.from_numpy(dirs[k]).to(DEV)
        mid = O + 0.5 * l * d
        t2 = tc = None
        for a in range(3):
            e = P[None, :, a] - mid[:, a, None]
            if per:
                e = e - L * torch.round(e / L)
            t2 = e * e if t2 is None else t2 + e * e
            tc = e * d[a] if tc is None else tc + e * d[a]
        i, j = torch.nonzero(t2 - tc * tc < (h * h * 1.0001)[None, :], as_tuple=True)
        e = P[j] - mid[i]
        if per:
            e = e - L * torch.round(e / L)
        c = torch.linalg.cross(e, d.expand_as(e))
        b2, t, hj = (c * c).sum(1), (e * d).sum(1) + 0.5 * l, h[j]
        ch = torch.sqrt((hj * hj - b2).clamp_min(0))
        ok = (b2 < hj * hj) & (t + ch > 0) & (t - ch < l)
        i, j, b2, t, hj, ch = (v[ok] for v in (i, j, b2, t, hj, ch))
        near = (b2 + t * t < hj * hj) if split else None
        u1, u2 = (torch.clamp_min(t - ch, 0) - t) / hj, (torch.clamp_max(t + ch, l) - t) / hj
        val = A[j] * (_gt if gt else _m4)(b2 / (hj * hj), u1, u2)
        yield k, i, j, val, near


def _fits(st, R, rows):
    n = st["n"]
    wrap = st["periodic"] and 0.5 * st["l"] + float(st["h"].max()) * 1.01 >= 0.5 * st["L"]
    return not wrap and float(rows) * R * n <= 6.0e10


def _exact_columns(st, weights, rows, gt=False, split=False, transpose=None):
    """sum_j weights_j (columns, and the near part with x = 1 when split) and, with `transpose`, the transposed product."""
    dirs = st["dirs"]
    R, m, n = dirs.shape[0], rows.numel(), st["n"]
    tau = [torch.zeros(m, R, device=DEV, dtype=torch.float64) for _ in weights]
    tn = torch.zeros(m, R, device=DEV, dtype=torch.float64)
    xb = torch.zeros(n, device=DEV, dtype=torch.float64)
    step = max(1, int(1.0e8) // n)
    for lo in range(0, m, step):
        for k, i, j, v, near in _pairs(st, rows[lo:lo + step], dirs, gt, split):
            far = v if near is None else torch.where(near, torch.zeros_like(v), v)
            for t, x in zip(tau, weights):
                t[:, k].index_add_(0, i + lo, far * x[j])
            if near is not None:
                tn[:, k].index_add_(0, i + lo, v - far)
            if transpose is not None:
                xb.index_add_(0, j, v * transpose[i + lo, k])
    return tau, tn, xb


def _exact_rate(tau, s, w, extra=()):
    """Gamma, tau_eff of columns [m, R] (and helium columns with their cross sections), rows a few thousand at a time."""
    m, R = tau.shape
    F, tot = s.numel(), float(w.sum())
    lw = torch.log(w / tot)
    G, te = torch.empty(m, device=DEV, dtype=torch.float64), torch.empty(m, device=DEV, dtype=torch.float64)
    step = max(1, int(1.0e8) // (R * F))
    for lo in range(0, m, step):
        E = tau[lo:lo + step].double()[:, :, None] * s
        for t, sx in extra:
            E = E + t[lo:lo + step, :, None] * sx
        ln = torch.logsumexp((lw - E).reshape(E.shape[0], -1), 1) - math.log(R)
        G[lo:lo + step], te[lo:lo + step] = tot * torch.exp(ln), -ln
    return G, te


def _exact_rates(T):
    lam = 315614.0 / T
    aA = 1.269e-13 * lam ** 1.503 / (1 + (lam / 0.522) ** 0.470) ** 1.923
    aB = 2.753e-14 * lam ** 1.500 / (1 + (lam / 2.740) ** 0.407) ** 2.242
    gc = 21.11 * T ** -1.5 * torch.exp(-0.5 * lam) * lam ** -1.089 / (1 + (lam / 0.354) ** 0.874) ** 1.101
    return aA, aB, gc


def _exact_x(G, nH, alpha, gc):
    an, e = alpha * nH, gc * nH
    return 2 * an / (G + 2 * an + e + torch.sqrt((G + e) ** 2 + 4 * G * an))


def _exact_solve(st, case):
    n, dirs = st["n"], st["dirs"]
    R = dirs.shape[0]
    if float(n) * R * n > 6.0e8 or not _fits(st, R, n):
        return None
    M = torch.zeros(R, n, n, device=DEV, dtype=torch.float64)
    for k, i, j, v, _ in _pairs(st, torch.arange(n, device=DEV), dirs, False, False):
        M[k, i, j] = v
    col = lambda x: torch.matmul(M, x).T  # noqa: E731
    extra = [(col(st["he1"]), st["s1"]), (col(st["he2"]), st["s2"])] if case.get("helium") else ()
    aA, aB, gc = _exact_rates(st["T"])
    x = _exact_x(torch.tensor(float(st["w"].sum()), device=DEV, dtype=torch.float64), st["nH"], aA, gc)
    act = torch.ones(n, dtype=torch.bool, device=DEV)
    latch = torch.zeros(n, dtype=torch.bool, device=DEV)
    for it in range(600):
        G, te = _exact_rate(col(x), st["s"], st["w"], extra)
        if it == 0:
            act = ~(te < 1e-4)
        latch |= act & (te >= 1)
        xn = torch.where(act, _exact_x(G, st["nH"], torch.where(latch, aB, aA), gc), x)
        rel = ((xn - x).abs() / x).max()
        x = xn
        if float(rel) < 1e-3:
            break
        if it > 60:
            return None
    return x


def exact(case, seed):
    st = _inputs(case, seed)
    op = case["op"]
    if op in ("rate", "rate_vjp"):
        if float(case["rows"]) * 12 * case["nside"] ** 2 * case["F"] > 2.0e9:
            return None
        tau, s, w = st["tau"].double(), st["s"], st["w"]
        G, te = _exact_rate(tau, s, w)
        if op == "rate":
            aA, aB, gc = _exact_rates(st["T"])
            return [G, te, _exact_x(G, st["nH"], torch.where(te >= 1, aB, aA), gc)]
        tb, wb = torch.empty_like(tau), torch.zeros_like(w)
        c = st["g_bar"][:, None] / tau.shape[1]
        step = max(1, int(1.0e8) // (tau.shape[1] * s.numel()))
        for lo in range(0, tau.shape[0], step):
            e = torch.exp(-tau[lo:lo + step, :, None] * s)
            tb[lo:lo + step] = -c[lo:lo + step] * (e * (w * s)).sum(2)
            wb += (e * c[lo:lo + step, :, None]).sum((0, 1))
        return [G, te, tb, wb]
    R = st["dirs"].shape[0]
    gt = case.get("kernel") == "gt"
    rows = st["org"].long() if "org" in st else torch.arange(st["n"], device=DEV)
    if op == "solve":
        return _exact_solve(st, case)
    if op == "gradient" or not _fits(st, R, rows.numel()):
        return None
    if op == "columns":
        return _exact_columns(st, [st["x"]], rows, gt)[0][0]
    if op == "columns_vjp":
        tau, _, xb = _exact_columns(st, [st["x"]], rows, gt, transpose=st["tau_bar"].double())
        return [tau[0], xb]
    tau, tn, _ = _exact_columns(st, [st["x"]], rows, gt, split=True)
    return [tau[0], tn, None, None]
