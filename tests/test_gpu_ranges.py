"""Calls at the ends of their ranges and beside one another."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import build, small_halo, spectra

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
