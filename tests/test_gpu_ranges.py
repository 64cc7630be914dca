"""Calls at the ends of their ranges and beside one another."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import workloads as W
from gpu_helpers import build, lnrate_sensitivity, small_halo, spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1304_4235_gb300 import urchin as U  # noqa: E402


def _dev(a, dt=np.float64):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).cuda()


def test_adjoint_rows_keep_the_high_bytes():
    # 6000 particles: the solve's rows take 6 bytes per segment, the adjoint's 7
    # (the order of the transposed product's additions hangs on its loads)
    w = small_halo(n=6000, seed=5)
    bvh, d = build(w, torch)
    (s, wts), _ = spectra(w, torch)
    dirs = U.urchin_healpix_dirs(1)
    state = torch.empty(w.n, dtype=torch.uint8, device="cuda")
    kw = dict(segments=U.SEG_STORE, raise_not_converged=False, profile=True)
    x, f = U.urchin_solve(bvh, dirs, w.l_ray, s, wts, d["nH"], d["T"], tol=1e-300, max_iter=2, tau_skip=0.0,
                          state=state, **kw)
    _, a = U.urchin_solve_vjp(bvh, dirs, w.l_ray, s, wts, d["nH"], d["T"], x, state, torch.ones_like(x),
                              tau_skip=0.0, max_iter=1, **kw)
    for st, per in ((f, 6), (a, 7)):
        # one product over every row: its segments, a column per ray and x
        assert st["n_active"] == w.n and st["nnz"] > 0
        assert st["spmv_bytes"] == st["nnz"] * per + w.n * 12 * 4 + w.n * 4


@pytest.mark.parametrize("decades", [20, 30, 60, 250])
def test_rate_transpose_fp32_of_wide_spectra(decades):
    # weights over many decades, the hard bins the faint ones: behind deep
    # columns those carry all of the rate, and the FP32 form stays the rounded
    # double one (to 7e-8, as over ordinary spectra)
    rng = np.random.default_rng(decades)
    F, n, R = 40, 800, 12
    E = np.exp(np.linspace(0.0, np.log(10.0), F))
    s = E ** -3
    wts = 1e-12 * 10.0 ** (-decades * (E - 1) / 9)
    tau = (10.0 ** rng.uniform(-3, 4.0, (n, R))).astype(np.float32)
    tau[0, :3] = [0.0, 1e30, np.inf]
    # cotangents that bring the result into the range of float
    gb = np.where(rng.random(n) < 0.5, -1.0, 1.0) * 10.0 ** rng.uniform(0, decades + 12, n)
    a, _ = U.urchin_gamma_vjp(_dev(tau, np.float32), _dev(s), _dev(wts), _dev(gb), want_w=False)
    b, _ = U.urchin_gamma_vjp(_dev(tau), _dev(s), _dev(wts), _dev(gb), want_w=False)
    a, b = a.cpu().numpy().astype(np.float64), b.cpu().numpy()
    with np.errstate(over="ignore"):
        over = ~np.isfinite(b.astype(np.float32))
    ok = (np.abs(b) > 1.2e-38) & ~over
    assert ok.mean() > 0.2
    assert (np.abs(a[ok] - b[ok]) <= 7e-8 * np.abs(b[ok])).all()
    assert np.array_equal(np.isinf(a), over)
    # two bins: the faint one alone is left behind a column of 2000
    t = np.full((1, 1), 2000.0)
    g, _ = U.urchin_gamma_vjp(_dev(t, np.float32), _dev([1.0, 0.02]), _dev([1e-12, 1e-60]), _dev([1e50]), want_w=False)
    want = -1e50 * 1e-60 * 0.02 * np.exp(-40.0)
    assert abs(float(g[0, 0]) - want) <= 1e-6 * abs(want)


def test_bins_that_fill_the_default_shared_memory():
    # dynamic sizes within a block's static ones of 48 KB, in a process whose
    # earlier calls have not raised the limit (24 B per bin in the fold, with
    # the log rates of a block's rows, and 16 B in the rate transpose)
    code = """
import numpy as np, torch
import workloads as W
from gpu_helpers import build, small_halo
from paper_1304_4235_gb300 import urchin as U
def spec(F):
    e, J = W.powerlaw_spectrum(F, 13.6, 54.4)
    return [torch.from_numpy(a).cuda() for a in U.urchin_spectrum_weights(e, J, 1e-12)]
g = torch.Generator(device="cuda").manual_seed(1)
tau = lambda n, R: 10.0 ** (6 * torch.rand(n, R, generator=g, device="cuda") - 4)
for n, R, F in ((130000, 12, 2048), (65536, 12, 1536), (40000, 48, 1024), (9000, 192, 1024)):
    s, w = spec(F)
    t = tau(n, R)
    a = U.urchin_gamma(t, s, w)[0]
    b = torch.exp(-t[:64, :, None].double() * s) @ w
    assert float((a[:64] / b.mean(1) - 1).abs().max()) < 1e-5
for F in (3040, 3072):
    s, w = spec(F)
    t = tau(300, 12)
    one = torch.ones(300, dtype=torch.float64, device="cuda")
    a = U.urchin_gamma_vjp(t, s, w, one, want_w=True)
    b = U.urchin_gamma_vjp(t.double(), s, w, one, want_w=True)
    assert float((a[0] / b[0] - 1).abs().max()) < 1e-6 and float((a[1] / b[1] - 1).abs().max()) < 1e-6
for n, F in ((65536, 1536), (4096, 4093)):
    w = small_halo(n=n, seed=2)
    bvh, d = build(w, torch)
    s, wt = spec(F)
    state = torch.empty(n, dtype=torch.uint8, device="cuda")
    x, _ = U.urchin_solve(bvh, U.urchin_healpix_dirs(1), w.l_ray, s, wt, d["nH"], d["T"], tol=1e-300, max_iter=1,
                          state=state, raise_not_converged=False)
    assert bool(torch.isfinite(x).all())
    if n < 10000:
        wb, _ = U.urchin_solve_vjp(bvh, U.urchin_healpix_dirs(1), w.l_ray, s, wt, d["nH"], d["T"], x, state,
                                   torch.ones_like(x), max_iter=1, raise_not_converged=False)
        assert bool(torch.isfinite(wb).all())
print("done")
"""
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(here), here]))
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stderr[-2000:]


def test_threads_with_different_sizes():
    # calls of one kernel with different amounts of shared memory from six threads
    # at once: none is refused, and each gives what it gives alone
    w = small_halo(n=600, seed=8)
    bvh, _ = build(w, torch)
    x = _dev(np.exp(np.random.default_rng(1).uniform(np.log(1e-4), 0.0, w.n)))
    tau = torch.rand(64, 12, device="cuda") * 10

    def columns(nside):
        return lambda: U.urchin_trace_columns(bvh, x, U.urchin_healpix_dirs(nside), w.l_ray)

    def rate(F):
        e, J = W.powerlaw_spectrum(F, 13.6, 54.4)
        s, wt = (_dev(a) for a in U.urchin_spectrum_weights(e, J, 1e-12))
        return lambda: U.urchin_gamma(tau, s, wt)[0]

    for fa, fb, times in ((columns(1), columns(4), 300), (rate(2100), rate(4096), 3000)):
        want, bad = [fa(), fb()], []

        def work(f, ref):
            try:
                for _ in range(times):
                    if not torch.equal(f(), ref):
                        bad.append("differs")
            except Exception as e:      # noqa: BLE001
                bad.append(repr(e))

        th = [threading.Thread(target=work, args=a) for a in 3 * list(zip((fa, fb), want))]
        for t in th:
            t.start()
        for t in th:
            t.join()
        assert not bad, bad[:3]


@pytest.mark.parametrize("precision", [U.F32, U.F64])
def test_192_directions_in_every_form(precision):
    w = small_halo(n=1500, seed=9)
    bvh, d = build(w, torch)
    x = _dev(np.exp(np.random.default_rng(2).uniform(np.log(1e-4), 0.0, w.n)))
    dirs = U.urchin_healpix_dirs(4)
    pick = np.arange(0, 192, 17)
    kw = dict(precision=precision)
    # a ray does not depend on the other directions
    full = U.urchin_trace_columns(bvh, x, dirs, w.l_ray, **kw)
    part = U.urchin_trace_columns(bvh, x, dirs[pick], w.l_ray, **kw)
    assert torch.equal(full[:, _dev(pick, np.int64)], part)
    nf, np_ = (U.urchin_trace_columns_nearfar(bvh, x, q, w.l_ray, **kw) for q in (dirs, dirs[pick]))
    # (near columns to 2 ulp in FP32: their few full chords are added between the
    # partial ones as the packet's queue fills)
    assert torch.equal(nf[0][:, _dev(pick, np.int64)], np_[0])
    near = nf[1][:, _dev(pick, np.int64)]
    assert float(((near - np_[1]).abs() / np_[1]).max()) <= (2.4e-7 if precision == U.F32 else 0.0)
    # the transpose is linear in the rays: the two halves of the directions add
    # up (FP64 sums in any order of values rounded alike)
    tb = torch.rand(w.n, 192, device="cuda", dtype=torch.float64)
    tb = tb.float() if precision == U.F32 else tb
    xb = U.urchin_trace_columns_vjp(bvh, dirs, w.l_ray, tb, **kw)
    parts = sum(U.urchin_trace_columns_vjp(bvh, dirs[a:a + 96], w.l_ray, tb[:, a:a + 96].contiguous(), **kw)
                for a in (0, 96))
    assert float(((xb - parts).abs() / parts.clamp_min(1e-300)).max()) < 1e-12
    # lists kept while tracing (FP32), counted and filled, and no lists: sweep 0
    # has the same columns
    (s, wts), _ = spectra(w, torch)
    for near_far in (False, True):
        xs = [U.urchin_solve(bvh, dirs, w.l_ray, s, wts, d["nH"], d["T"], tol=1e-300, max_iter=1, segments=g,
                             near_far=near_far, raise_not_converged=False, **kw)[0]
              for g in (U.SEG_RECOMPUTE, U.SEG_AUTO, U.SEG_STORE)]
        assert torch.equal(xs[0], xs[1]) and torch.equal(xs[0], xs[2])


@pytest.mark.parametrize("precision", [U.F32, U.F64])
def test_rays_longer_than_the_particle_set(precision):
    # isolated particles: beyond the far side of the set there is nothing, so
    # longer rays have the same columns (bit for bit: the same chords) and are
    # filtered against no more spheres
    w = small_halo(n=6000, seed=12)
    bvh, d = build(w, torch)
    x = _dev(np.exp(np.random.default_rng(3).uniform(np.log(1e-4), 0.0, w.n)))
    (s, wts), _ = spectra(w, torch)
    dirs = U.urchin_healpix_dirs(1)
    ref, tests = None, None
    for l in (1e3, 1e6, 1e9, 1e20, 1e30, 1e300):
        tau = U.urchin_trace_columns(bvh, x, dirs, l, precision=precision)
        _, st = U.urchin_solve(bvh, dirs, l, s, wts, d["nH"], d["T"], tol=1e-300, max_iter=1, profile=True,
                               precision=precision, raise_not_converged=False)
        if ref is None:
            ref, tests = tau, st["sphere_tests"]
        assert torch.equal(tau, ref)
        assert st["sphere_tests"] <= 1.01 * tests


def test_rays_over_many_periodic_images():
    # along an axis a shift by a multiple of the box is a symmetry: 700 boxes are
    # seven times 100 (1401 images a side, more than 2^31 in all)
    w = W.lattice_box(n_side=6, seed=4)
    bvh, _ = build(w, torch)
    x = _dev(np.full(w.n, 0.5))
    for a in range(3):
        d = np.zeros((1, 3))
        d[0, a] = 1.0 if a < 2 else -1.0
        one, many = (U.urchin_trace_columns(bvh, x, d, k * w.box, origins=_dev([0, 40, 215], np.int32),
                                            precision=U.F64) for k in (100, 700))
        assert float(one.min()) > 0.0
        assert float((many / one / 7.0 - 1.0).abs().max()) < 1e-9


def test_ray_order_of_a_list_shorter_than_the_particles():
    # the sort of fewer than 2^21 keys takes smaller tiles, and so more work
    # space per key: a list just below that of 2^21 particles, one direction
    n = 1 << 21
    g = torch.Generator(device="cuda").manual_seed(7)
    p = torch.rand(3, n, generator=g, device="cuda") * 1000.0
    h = torch.full((n,), 6.0, device="cuda")
    bvh = U.urchin_build_bvh(p[0].contiguous(), p[1].contiguous(), p[2].contiguous(), h,
                             torch.full((n,), 1e60, dtype=torch.float64, device="cuda"), False, 0.0, 3.0857e21)
    one = torch.ones(n, dtype=torch.float64, device="cuda")
    state = torch.zeros(n, dtype=torch.uint8, device="cuda")
    state[::2048] = 2                                    # 1024 frozen particles
    wb, st = U.urchin_solve_vjp(bvh, np.array([[0.0, 0.6, 0.8]]), 10.0, one[:1].clone(), one[:1] * 1e-12, one * 1e-4,
                                one * 1e4, one * 1e-3, state, one, max_iter=2, raise_not_converged=False)
    assert st["n_active"] == n - 1024 and bool(torch.isfinite(wb).all())


def test_traversals_are_those_made():
    # helium columns traced along with the hydrogen columns are one traversal
    w = W.lattice_box(n_side=8, seed=3)
    bvh, d = build(w, torch)
    edges = np.exp(np.linspace(np.log(13.6), np.log(136.0), 31))
    mid = np.sqrt(edges[:-1] * edges[1:])
    s, wts = U.urchin_spectrum_weights(edges, (mid / 13.6) ** -1.5, w.gamma_thin)
    f1, f2 = W.helium_fractions(w, 9)
    for g, traces in ((U.SEG_AUTO, 1), (U.SEG_RECOMPUTE, 1), (U.SEG_STORE, 4)):
        _, st = U.urchin_solve(bvh, U.urchin_healpix_dirs(1), w.l_ray, _dev(s), _dev(wts), d["nH"], d["T"], tol=1e-300,
                               max_iter=1, segments=g, s_he1=_dev(W.hei_cross_section_standin(edges)),
                               s_he2=_dev(U.urchin_cross_section_ratio(edges, U.XSEC_HEII)), he1=_dev(f1),
                               he2=_dev(f2), raise_not_converged=False)
        assert st["trace_launches"] == traces and st["traversals"] == traces


@pytest.mark.parametrize("dtype,R,F", [(np.float32, 12, 1400), (np.float32, 12, 1401), (np.float32, 5, 3),
                                       (np.float64, 48, 47), (np.float64, 48, 48)])
def test_rates_by_rays_and_by_rows(dtype, R, F):
    # many rows are folded with several rays to a thread (FP32 up to 1400 bins,
    # FP64 with fewer bins than rays), few by a thread per ray: the same bits
    n = 960000 // R
    g = torch.Generator(device="cuda").manual_seed(F)
    tau = 10.0 ** (9 * torch.rand(n, R, generator=g, device="cuda", dtype=torch.float64) - 5)
    tau = tau.to(torch.from_numpy(np.zeros(1, dtype)).dtype)
    e, J = W.powerlaw_spectrum(F, 13.6, 54.4)
    s, wts = (_dev(a) for a in U.urchin_spectrum_weights(e, J, 1e-12))
    many = U.urchin_gamma(tau, s, wts)
    for a in (0, n // 2):
        few = U.urchin_gamma(tau[a:a + 100].contiguous(), s, wts)
        assert torch.equal(few[0], many[0][a:a + 100]) and torch.equal(few[1], many[1][a:a + 100])


@pytest.mark.parametrize("n,R", [(1, 12), (1023, 48), (2049, 5), (1500, 192), (270001, 3)])
def test_spectrum_gradient_of_the_rate(n, R):
    # the coefficients' blocks take one row up to 256 rows; w_bar in FP64 is the
    # sum of its terms to their rounding (1e-16 each, about 1e6 of them)
    g = torch.Generator(device="cuda").manual_seed(n)
    tau = 10.0 ** (6 * torch.rand(n, R, generator=g, device="cuda", dtype=torch.float64) - 5)
    gb = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    gb[::7] = 0.0
    s, wts = _dev([1.0, 0.3, 0.02]), _dev([1e-12, 3e-13, 1e-13])
    _, wb = U.urchin_gamma_vjp(tau, s, wts, gb, want_tau=False)
    for b in range(3):
        e = torch.exp(-float(s[b]) * tau) * (gb / R)[:, None]
        assert abs(float(wb[b] - e.sum())) <= 1e-12 * float(e.abs().sum())


@pytest.mark.parametrize("n,per", [(65536, 6), (65537, 7), (80000, 7)])
def test_products_of_6_and_7_byte_rows(n, per):
    # one sweep over rows (written by the filling traversal, and copied from the
    # chunks before the fourth sweep) against the same sweep with traced columns.
    # These differ by their order of summation, 2e-6, which moves a rate by D times
    # that (D = sum tau |d ln Gamma / d tau|), and x by no more; the fold rounds its
    # sums to 1e-6.  At 80000 particles 14464 indices need their high byte; without
    # it they would be those of particles on the other side of the halo.
    w = small_halo(n=n, seed=29)
    bvh, d = build(w, torch)
    (s, wts), (so, wo) = spectra(w, torch)
    dirs = U.urchin_healpix_dirs(1)

    def solve(seg, sweeps, x=None, **kw):
        return U.urchin_solve(bvh, dirs, w.l_ray, s, wts, d["nH"], d["T"], x, tol=1e-300, max_iter=sweeps, segments=seg,
                              tau_skip=0.0, case_rule=U.CASE_A, raise_not_converged=False, **kw)

    pick = W.random_origins(n, 2500, 31)
    for seg, before in ((U.SEG_STORE, 1), (U.SEG_AUTO, 4)):
        x0, _ = solve(seg, before)
        x1, st = solve(seg, before + 1, profile=True)
        assert st["segments_stored"]
        if seg == U.SEG_STORE:
            assert st["n_active"] == n and st["spmv_bytes"] == st["nnz"] * per + n * 12 * 4 + n * 4
        tau = U.urchin_trace_columns(bvh, x0, dirs, w.l_ray, origins=_dev(pick, np.int32)).cpu().numpy()
        want, _ = solve(U.SEG_RECOMPUTE, 1, x0.clone(), warm_start=True)
        dx = ((x1 - want).abs() / want).cpu().numpy()[pick]
        assert (dx <= 2e-6 * lnrate_sensitivity(tau, so, wo) + 2e-6).all()


@pytest.mark.parametrize("R,F", [(3, 100), (7, 20), (15, 33)])
def test_rates_of_odd_ray_counts(R, F):
    # the last ray of an odd number is folded by itself: the same bits as a thread
    # per ray gives, also where bins underflow and for columns out of range
    n = 1000000 // R + 1
    g = torch.Generator(device="cuda").manual_seed(R)
    tau = 10.0 ** (9 * torch.rand(n, R, generator=g, device="cuda") - 4)
    tau[1] = float("nan")
    tau[2, R - 1] = float("inf")
    tau[3] = 0.0
    e, J = W.powerlaw_spectrum(F, 13.6, 54.4)
    s, wts = (_dev(a) for a in U.urchin_spectrum_weights(e, J, 1e-12))
    many = U.urchin_gamma(tau, s, wts)
    for a in (0, n // 2, n - 100):
        few = U.urchin_gamma(tau[a:a + 100].contiguous(), s, wts)
        for p, q in zip(few, many):
            assert torch.equal(p.nan_to_num(-1.0), q[a:a + 100].nan_to_num(-1.0))


@pytest.mark.parametrize("slab", [U.SLAB_THRESHOLD, U.SLAB_SPECTRUM])
@pytest.mark.parametrize("R", [1, 2, 3, 48, 192])
def test_near_far_rate_is_the_mean_of_its_rays(R, slab):
    # a row whose rays all equal ray k has that ray's rate, and rows add up to the
    # mean of those (a sum of R doubles: R roundings, and some in each exponential);
    # a row does not depend on the others
    n = 1300 if R <= 3 else 20
    g = torch.Generator(device="cuda").manual_seed(R)
    tf = 10.0 ** (5 * torch.rand(n, R, generator=g, device="cuda", dtype=torch.float64) - 4)
    tn = 10.0 ** (5 * torch.rand(n, R, generator=g, device="cuda", dtype=torch.float64) - 4)
    tf[1, R // 2] = tf[2] = float("inf") if slab == U.SLAB_SPECTRUM else 1e5
    nH = torch.full((n,), 1e-2, dtype=torch.float64, device="cuda")
    e, J = W.powerlaw_spectrum(30, 13.6, 54.4)
    s, wts = (_dev(a) for a in U.urchin_spectrum_weights(e, J, 1e-12))

    def rate(a, b):
        m = a.shape[0]
        return U.urchin_gamma_nearfar(a.contiguous(), b.contiguous(), s, wts, nH[:m], nH[:m] * 1e6, slab=slab)

    gam, te = rate(tf, tn)
    want = sum(rate(tf[:, k:k + 1].expand(n, R), tn[:, k:k + 1].expand(n, R))[0] for k in range(R)) / R
    ok = want > 0
    assert float(gam[~ok].abs().sum()) == 0.0
    assert float(((gam - want).abs()[ok] / want[ok]).max()) < 1e-13 + 3e-16 * R
    part = rate(tf[:7], tn[:7])
    assert torch.equal(part[0], gam[:7]) and torch.equal(part[1], te[:7])
