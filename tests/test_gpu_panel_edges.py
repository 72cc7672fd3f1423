"""The persistent panel solver at its edges, against dense LU: numbers of columns
that do not divide a CTA (1, 3, 33), more columns than slots (refill), block edges
1, 4 and 9, one row a thread and (df, larger systems) the rows of a block, whole
solution vectors without overlap (the kept rows are updated while other CTAs
change the residual), QMR, and an overlap whose spectrum is too wide for Chebyshev
sweeps (conjugate gradients).

tol 1e-11: a recurrence residual of 1e-11 leaves G within 1e-11 / eta of the exact
one, eta >= 0.1; max|G| is above 0.1 in all these systems, so 1e-8 of the largest
entry bounds every entry with a margin of ten.  QMR's quasi-residual bounds the
residual up to sqrt(iterations) < 40.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl
from oracle import dense, systems
from tests.helpers import out_layout

DEV = "cuda:0"
F, D = tb.TB_PREC_FP64, tb.TB_PREC_DF64
COCG, QMR = tb.TB_SOLVER_COCG, tb.TB_SOLVER_QMR


def _bsr(b):
    return tb.Bsr(b.n_brows, b.bdim, b.row_ptr, b.col_idx, b.val).to(DEV)


def _check(H, S, n_cols, prec, solver=COCG, full=False, panel_w=0, seed_shift=-1, tol=1e-11, inner_max=0):
    M = H.n_brows * H.bdim
    cols = np.unique(np.linspace(0, M - 1, n_cols).astype(np.int64))
    rl = [np.arange(M) if full else systems.block_pattern_rows(H, j) for j in cols]
    ptr, rows = out_layout(rl)
    z = wl.midpoint_shifts(7, -8.0, 6.0, 0.2)
    with tb.Context() as ctx:
        r = tb.solve(ctx, _bsr(H), None if S is None else _bsr(S), z, cols, ptr, rows, tol=tol, precision=prec,
                     solver=solver, panel_w=panel_w, seed_shift=seed_shift, inner_max=inner_max)
        assert r.rc == 0 and np.all(r.status.cpu().numpy() == tb.TB_COL_CONVERGED)
        G = r.G.cpu().numpy()
    ex = dense.green_lu(H.to_dense(), None if S is None else S.to_dense(), z, cols)
    bound = (40 if solver == QMR else 1) * 1e-8
    for c in range(len(cols)):
        e = ex[rl[c], c, :]
        assert np.abs(G[ptr[c]:ptr[c + 1]] - e).max() < bound * np.abs(ex).max(), c
    return r


@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
@pytest.mark.parametrize("n_cols,panel_w", [(1, 0), (3, 0), (33, 0), (20, 8)])
@pytest.mark.parametrize("spec", [wl.scaled(wl.C1_SYSTEM, L=5), wl.scaled(wl.C2_SYSTEM, L=4),
                                  wl.scaled(wl.C3_SYSTEM, n_sites=43), wl.scaled(wl.C5_SYSTEM, L=4)],
                         ids=["b1", "b4-overlap", "b9", "b4-subst"])
def test_columns_and_blocks(spec, n_cols, panel_w, prec):
    o = systems.build_system(spec, 11)
    _check(o.H, o.S, n_cols, prec, panel_w=panel_w)


@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
@pytest.mark.parametrize("solver", [COCG, QMR], ids=["cocg", "qmr"])
@pytest.mark.parametrize("spec", [wl.scaled(wl.C1_SYSTEM, L=7), wl.scaled(wl.C2_SYSTEM, L=4)], ids=["b1", "b4-overlap"])
def test_whole_vectors(spec, solver, prec):
    o = systems.build_system(spec, 5)
    _check(o.H, o.S, 6, prec, solver=solver, full=True, panel_w=8 if solver == QMR else 0)


def test_rows_of_a_block_per_thread():
    """df with overlap, 64 slots and 2048 rows per slot: the kernel whose threads hold a block row."""
    o = systems.build_system(wl.scaled(wl.C2_SYSTEM, L=9), 3)   # 729 block rows x 64 slots > 152 SMs x 256
    r = _check(o.H, o.S, 64, D)
    assert r.refinements > 0


@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
def test_wide_overlap_spectrum_takes_conjugate_gradients(prec):
    """S = D S0 D with D from 0.3 to 2 keeps S positive definite but spreads its spectrum."""
    o = systems.build_system(wl.scaled(wl.C2_SYSTEM, L=3), 3)
    S = o.S
    d = np.random.default_rng(1).uniform(0.3, 2.0, (S.n_brows, S.bdim))
    br = np.repeat(np.arange(S.n_brows), np.diff(S.row_ptr))
    S.val[:] = S.val * d[br][:, :, None] * d[S.col_idx][:, None, :]
    _check(o.H, S, 5, prec, inner_max=200)   # a condition number near 100: more steps than the default 40


def test_seed_at_the_edge_of_the_spectrum_leaves_fp32_range():
    """The residual of a seed far from the spectrum falls below what FP32 numbers hold long before the other shifts
    converge; the sweeps work on scaled residuals."""
    o = systems.build_system(wl.scaled(wl.C2_SYSTEM, L=3), 21)
    _check(o.H, o.S, 4, F, seed_shift=0, tol=1e-12)
