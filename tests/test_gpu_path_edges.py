"""The forms that the kernels take by size, at the sizes where they change:
tree levels and blocks of 32 spheres, full pair lists, narrow and wide packets,
ray order, rows folded by several threads, stored lists with 16-bit indices,
batches of sweeps, helium traced along, and the FP32 rate transpose.

Columns are held to the bounds of the parity tests (FP64 rel 1e-11, FP32 rel
1e-5 of the oracle).  A ray's columns do not depend on the rays that share its
packet, nor a row's rate on the threads that share the row, so calls of
different sizes on the same rays or rows are compared bit for bit."""
import dataclasses

import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import build, rel_err, small_halo, spectra

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1304_4235_gb300 import urchin as U  # noqa: E402


def _dev(a, dt=np.float64):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).cuda()


def _x(n, seed=0):
    return np.exp(np.random.default_rng(seed).uniform(np.log(1e-4), 0.0, n))


# one particle, one block and its neighbours, one and two entries of level 1
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 1023, 1025, 1057])
@pytest.mark.parametrize("periodic", [False, True])
def test_columns_tree_and_pair_list_edges(n, periodic):
    w = W.subset(W.lattice_box(n_side=11, seed=91), np.arange(n))
    # spheres of 300 kpc in a 1 Mpc box: every ray of a packet meets nearly
    # every sphere of a block, 1024 pairs where a list holds 128 to 256
    rng = np.random.default_rng(n)
    w = dataclasses.replace(w, h=(300.0 * rng.uniform(0.9, 1.1, n)).astype(np.float32), periodic=periodic,
                            box=w.box if periodic else 0.0)
    bvh, _ = build(w, torch)
    x = _x(n)
    ref = O.columns(w, x, O.healpix(1))
    for kernel in (U.KERNEL_M4, U.KERNEL_GT):
        if kernel == U.KERNEL_GT:
            ref = O.columns(w, x, O.healpix(1), kernel=U.KERNEL_GT)
        for prec, tol in ((U.F64, 1e-11), (U.F32, 1e-5)):
            tau = U.urchin_trace_columns(bvh, _dev(x), U.urchin_healpix_dirs(1), w.l_ray, kernel=kernel, precision=prec)
            assert rel_err(tau.cpu().numpy(), ref, floor=1e-300).max() < tol
    # every mode of the traversal over the same lists: near + far = all, and
    # the transpose
    tf, tn = U.urchin_trace_columns_nearfar(bvh, _dev(np.ones(n)), U.urchin_healpix_dirs(1), w.l_ray, precision=U.F64)
    tau1 = U.urchin_trace_columns(bvh, _dev(np.ones(n)), U.urchin_healpix_dirs(1), w.l_ray, precision=U.F64)
    assert rel_err((tf + tn).cpu().numpy(), tau1.cpu().numpy(), floor=1e-300).max() < 1e-11
    for prec, tol in ((U.F64, 1e-10), (U.F32, 1e-5)):
        tb = torch.rand(n, 12, dtype=torch.float64, device="cuda")
        tb = tb if prec == U.F64 else tb.float()
        xb = U.urchin_trace_columns_vjp(bvh, U.urchin_healpix_dirs(1), w.l_ray, tb, precision=prec)
        lhs, rhs = float((tau1 * tb.double()).sum()), float(xb.sum())
        assert abs(lhs - rhs) <= tol * abs(lhs)


# below and above the thresholds of the ray order (16384 particles, a list of
# 1024 origins), of the wide form (8512 packets on 152 SMs) and of 16 and 8
# origins per packet; in any order
@pytest.mark.parametrize("precision", [U.F32, U.F64])
@pytest.mark.parametrize("n", [9000, 16383, 24001])
def test_columns_do_not_depend_on_the_packet(n, precision):
    if precision == U.F64 and n > 16383:
        n = 16385
    w = small_halo(n=n, seed=17)
    bvh, _ = build(w, torch)
    x, dirs = _dev(_x(n)), U.urchin_healpix_dirs(1)
    full = U.urchin_trace_columns(bvh, x, dirs, w.l_ray, precision=precision)
    fullnf = U.urchin_trace_columns_nearfar(bvh, x, dirs, w.l_ray, precision=precision)
    for m in (1, 33, 1023, 1024, 5000):
        org = np.random.default_rng(m).permutation(n)[:m].astype(np.int32)
        part = U.urchin_trace_columns(bvh, x, dirs, w.l_ray, origins=_dev(org, np.int32), precision=precision)
        assert torch.equal(part, full[torch.from_numpy(org).long().cuda()])
        nf = U.urchin_trace_columns_nearfar(bvh, x, dirs, w.l_ray, origins=_dev(org, np.int32), precision=precision)
        assert torch.equal(nf[0], fullnf[0][torch.from_numpy(org).long().cuda()])


@pytest.mark.parametrize("R", [1, 5, 12, 48, 192])
@pytest.mark.parametrize("F", [1, 37])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_gamma_rows_shared_by_threads(R, F, dtype):
    # few rows are folded by many threads each, 130000 by one: the same bits
    rng = np.random.default_rng(R + F)
    n = 130000 if R <= 12 else 9000
    tau = 10.0 ** rng.uniform(-6, 4.4, (n, R))
    tau[0] = 0.0
    tau[1, 0] = np.nan
    e, J = W.powerlaw_spectrum(F, 13.6, 54.4)
    s, wts = U.urchin_spectrum_weights(e, J, 1e-12)
    sg, wg = _dev(s), _dev(wts)
    g, te = U.urchin_gamma(_dev(tau, dtype), sg, wg)
    for m in (1, 2, 500, 7001):
        gs, ts = U.urchin_gamma(_dev(tau[:m], dtype), sg, wg)
        assert torch.equal(torch.nan_to_num(gs, nan=-1.0), torch.nan_to_num(g[:m], nan=-1.0))
        assert torch.equal(torch.nan_to_num(ts, nan=-1.0), torch.nan_to_num(te[:m], nan=-1.0))
    assert torch.isnan(g[1]) and abs(float(g[0]) - wts.sum()) <= 1e-6 * wts.sum()


@pytest.mark.parametrize("F", [1, 64, 401])
def test_rate_transpose_fp32_is_the_rounded_double(F):
    # the float-pair sum is within about 1e-9 of the double one, so the FP32
    # result is its rounding (2^-24 = 6e-8) to 7e-8; outside [0, 1e30) both take
    # the double loop
    rng = np.random.default_rng(F)
    n, R = 1500, 12
    tau = (10.0 ** rng.uniform(-9, 4.3, (n, R))).astype(np.float32)
    tau[0], tau[1, :4] = 0.0, [np.nan, np.inf, 1e30, 1e29]
    e, J = W.powerlaw_spectrum(F, 13.6, 54.4)
    s, wts = U.urchin_spectrum_weights(e, J, 1e-12)
    if F > 1:
        wts[-1] = 0.0                     # the smallest cross section without a weight
    gb = rng.normal(size=n) * 10.0 ** rng.uniform(-30, 40, n)
    gb[2] = 0.0
    a, _ = U.urchin_gamma_vjp(_dev(tau, np.float32), _dev(s), _dev(wts), _dev(gb), want_w=False)
    b, _ = U.urchin_gamma_vjp(_dev(tau.astype(np.float64)), _dev(s), _dev(wts), _dev(gb), want_w=False)
    a, b = a.cpu().numpy().astype(np.float64), b.cpu().numpy()
    big = np.abs(b) > 1.2e-38
    with np.errstate(over="ignore"):
        ovf = ~np.isfinite(b.astype(np.float32))
    assert np.array_equal(np.isinf(a), ovf)
    ok = big & ~ovf
    assert (np.abs(a[ok] - b[ok]) <= 7e-8 * np.abs(b[ok])).all()
    assert np.abs(a[~big]).max(initial=0.0) <= 1.2e-38


def _solve(w, bvh, d, sp, **kw):
    kw.setdefault("precision", U.F32)
    return U.urchin_solve(bvh, U.urchin_healpix_dirs(w.nside), w.l_ray, sp[0], sp[1], d["nH"], d["T"],
                          raise_not_converged=False, **kw)


def test_sweep_batches_and_16_bit_lists():
    # profile mode times every sweep and launches them one by one; the batches
    # stop where it stops, with the same history and the same bits, also when
    # the limit cuts a batch short
    w = small_halo(n=6000, seed=5)
    bvh, d = build(w, torch)
    sg, _ = spectra(w, torch)
    for kw in (dict(tol=1e-3, max_iter=300), dict(tol=1e-300, max_iter=4), dict(tol=1e-300, max_iter=12),
               dict(tol=1e-6, max_iter=200, method=U.METHOD_NEWTON), dict(tol=1e-3, max_iter=60, precision=U.F64)):
        xa, sa = _solve(w, bvh, d, sg, segments=U.SEG_AUTO, history=True, **kw)
        xb, sb = _solve(w, bvh, d, sg, segments=U.SEG_AUTO, history=True, profile=True, **kw)
        assert torch.equal(xa, xb)
        for k in ("iterations", "converged", "traversals", "rays", "particle_updates", "history_maxrel",
                  "history_unconverged", "spmv_launches", "sweep_launches"):
            assert sa[k] == sb[k], k


@pytest.mark.parametrize("n", [65536, 65537])
def test_stored_indices_at_the_16_bit_edge(n):
    # the first n slots of the same particles: lists written by the filling
    # traversal (SEG_STORE) and copied from the chunks (SEG_AUTO, sweep 3 on)
    # hold the same entries in the same order
    w = small_halo(n=n, seed=23)
    bvh, d = build(w, torch)
    sg, _ = spectra(w, torch)
    xa, sa = _solve(w, bvh, d, sg, segments=U.SEG_AUTO, tol=1e-300, max_iter=5, profile=True)
    xs, ss = _solve(w, bvh, d, sg, segments=U.SEG_STORE, tol=1e-300, max_iter=5)
    assert sa["segments_stored"] and ss["segments_stored"]
    # the products group a ray's entries otherwise than the traversal does, which
    # moves a column by up to 1e-6 and x by up to its sensitivity (about 1e3 at a
    # front) times that in a sweep; a wrong particle moves it by far more
    assert float(((xa - xs).abs() / xs).max()) < 5e-2
    xr, _ = _solve(w, bvh, d, sg, segments=U.SEG_RECOMPUTE, tol=1e-300, max_iter=5)
    assert float(((xs - xr).abs() / xr).max()) < 5e-2


def test_helium_traced_along_is_the_same_columns():
    # SEG_STORE traces every species by itself, SEG_AUTO and SEG_RECOMPUTE all
    # three at once: sweep 0 has the same columns bit for bit
    w = W.lattice_box(n_side=9, seed=3)
    bvh, d = build(w, torch)
    edges = np.exp(np.linspace(np.log(13.6), np.log(136.0), 31))
    mid = np.sqrt(edges[:-1] * edges[1:])
    s, wts = U.urchin_spectrum_weights(edges, (mid / 13.6) ** -1.5, w.gamma_thin)
    f1, f2 = W.helium_fractions(w, 9)
    kw = dict(s_he1=_dev(W.hei_cross_section_standin(edges)), s_he2=_dev(U.urchin_cross_section_ratio(edges, U.XSEC_HEII)),
              he1=_dev(f1), he2=_dev(f2), tol=1e-300, max_iter=1)
    for kernel in (U.KERNEL_M4, U.KERNEL_GT):
        x = [_solve(w, bvh, d, (_dev(s), _dev(wts)), segments=g, kernel=kernel, **kw)[0]
             for g in (U.SEG_STORE, U.SEG_AUTO, U.SEG_RECOMPUTE)]
        assert torch.equal(x[0], x[1]) and torch.equal(x[0], x[2])
