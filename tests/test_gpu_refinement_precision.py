"""When a refinement pass of the panel solver may take S c and the residual in FP32.
df panels: behind a first sweep whose residual is below engine_light() inner tolerances,
0.05 over the error of an FP32 residual: with inner_tol 1e-12 3.3e-7 ||rt|| at hi / lo = 1.6,
which a first sweep reaches (it ends near 2e-7, FP32 rounding), and 1e-7 at hi / lo near 19,
which it does not: there the pass is a df one.
G agrees with dense LU: tol 1e-10, eta 0.3, lambda_min 0.13: 1e-8 of the largest entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl
from oracle import dense, systems

DEV = "cuda:0"


def _solve(scale, prec, **kw):
    o = systems.build_system(wl.scaled(wl.C2_SYSTEM, L=6), 1234)
    H, S = o.H, o.S
    br = np.repeat(np.arange(S.n_brows), np.diff(S.row_ptr))
    S.val[br != S.col_idx] *= scale
    lam = np.linalg.eigvalsh(S.to_dense())
    cols = np.array([0, 101, 500], np.int64)
    ptr = np.arange(4, dtype=np.int64)
    z = wl.midpoint_shifts(4, -8.0, 6.0, 0.3)
    dev = lambda a: tb.Bsr(a.n_brows, a.bdim, a.row_ptr, a.col_idx, a.val).to(DEV)
    with tb.Context() as ctx:
        r = tb.solve(ctx, dev(H), dev(S), z, cols, ptr, cols, precision=prec, **kw)
    assert r.rc == 0
    ex = dense.green_lu(H.to_dense(), S.to_dense(), z, cols)
    for c, j in enumerate(cols):
        e = ex[j, c, :]
        assert np.abs(r.G.cpu().numpy()[c] - e).max() < 1e-8 * np.abs(ex).max()
    return r, lam[-1] / lam[0]


def test_df_passes_in_fp32_only_where_the_spectrum_allows_it():
    r, kappa = _solve(1.0, tb.TB_PREC_DF64)
    assert kappa < 1.6 and r.light_refinements > 0
    r, kappa = _solve(4.0, tb.TB_PREC_DF64)
    assert 9 < kappa < 11                  # 19 between the bounds, which are 5 % of the width outside
    assert r.refinements > 0 and r.light_refinements < 0.1 * r.refinements


def test_fp64_passes_are_fp64():
    """Also where a residual is below the df panels' bound (inner_tol 1e-9: 1.6e-5 after the first sweep)."""
    r, _ = _solve(1.0, tb.TB_PREC_FP64, inner_tol=1e-9)
    assert r.refinements > 0 and r.light_refinements == 0
    r, _ = _solve(1.0, tb.TB_PREC_FP64)
    assert r.refinements > 0 and r.light_refinements == 0
