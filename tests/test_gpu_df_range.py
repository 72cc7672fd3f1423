"""Seeds that converge long before another shift: between two bands (the substitution
system at its median shift) and outside the spectrum (seed_shift = 0 of a window that
starts far below the band).  The seed's residual then falls below what the exponents of
df and FP32 vectors (and, far enough, the squares of FP64 ones) hold while other shifts
are still at work; columns are kept in range by powers of two.

Every column converges and agrees with dense LU.  A residual of tol leaves G within
tol / (eta lambda_min(S)) of the exact one, eta >= 0.05; with the
largest entry of a column above 0.1, 1e-8 of it bounds tol = 1e-11 (1e-10 where eta and
lambda_min(S) allow it) with a margin.  FP32 panels: 2e-3, the bound that tests/test_gpu_local.py holds them to.
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
F, D, M = tb.TB_PREC_FP64, tb.TB_PREC_DF64, tb.TB_PREC_MIXED


def _principal(A, atoms):
    b, n = A.bdim, len(atoms)
    loc = {int(a): i for i, a in enumerate(atoms)}
    out = np.zeros((n * b, n * b))
    for a, i in loc.items():
        for k in range(A.row_ptr[a], A.row_ptr[a + 1]):
            j = loc.get(int(A.col_idx[k]))
            if j is not None:
                out[i * b:(i + 1) * b, j * b:(j + 1) * b] = A.val[k]
    return out


def _local(H, S, n, radii, z, prec, tol, bound, seed_shift=-1):
    rng = np.random.default_rng(5)
    rows = np.sort(rng.choice(H.n_rows, n, replace=False)).astype(np.int64)
    rad = rng.choice(np.asarray(radii), n).astype(np.int32)
    sptr, satoms = tb.local_subspaces(H, rows, rad)
    optr = np.arange(n + 1, dtype=np.int64)
    with tb.Context() as ctx:
        r = tb.solve_local(ctx, H.to(DEV), None if S is None else S.to(DEV), z, rows, sptr, satoms, optr, rows, tol=tol,
                           precision=prec, seed_shift=seed_shift)
        status, G = r.status.cpu().numpy(), r.G.cpu().numpy()
    assert r.rc == 0 and np.all(status == tb.TB_COL_CONVERGED), np.bincount(status)
    b = H.bdim
    for c, j in enumerate(rows):
        at = satoms[sptr[c]:sptr[c + 1]].astype(np.int64)
        Hd, Sd = _principal(H, at), None if S is None else _principal(S, at)
        jl = int(np.searchsorted(at, j // b)) * b + int(j % b)
        L = np.eye(len(Hd)) if Sd is None else np.linalg.cholesky(Sd)
        lam, Y = np.linalg.eigh(np.linalg.solve(L, np.linalg.solve(L, Hd).T))
        y = np.linalg.solve(L.T, Y)[jl]
        ex = (y * y) @ (1.0 / (z[None, :] - lam[:, None]))
        assert np.abs(G[c] - ex).max() < bound * np.abs(ex).max(), (c, np.abs(G[c] - ex).max() / np.abs(ex).max())


@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
@pytest.mark.parametrize("nz", [17, 64])
def test_local_median_shift_between_the_bands(nz, prec):
    """255 columns: df64 columns broke down (rho = 0) or stopped with a wrong G."""
    H, S, _ = tb.build_system(wl.scaled(wl.C5_SYSTEM, L=24), 1234)
    _local(H, S, 255, (2, 3, 4), wl.midpoint_shifts(nz, -10.0, 6.0, 0.1), prec, 1e-10, 1e-8)


@pytest.mark.parametrize("prec,tol,bound", [(F, 1e-11, 1e-8), (D, 1e-11, 1e-8), (M, 1e-5, 2e-3)], ids=["fp64", "df64", "mixed"])
@pytest.mark.parametrize("spec", [wl.scaled(wl.C1_SYSTEM, L=7), wl.scaled(wl.C2_SYSTEM, L=6)], ids=["b1", "b4-overlap"])
def test_local_seed_outside_the_spectrum(spec, prec, tol, bound):
    H, S, _ = tb.build_system(spec, 3)
    _local(H, S, 20, (2, 3), wl.midpoint_shifts(9, -60.0, 6.0, 0.1), prec, tol, bound, seed_shift=0)


def _panel(H, S, n_cols, z, prec, tol, bound, **kw):
    cols = np.unique(np.linspace(0, H.n_brows * H.bdim - 1, n_cols).astype(np.int64))
    rl = [systems.block_pattern_rows(H, j) for j in cols]
    ptr, rows = out_layout(rl)
    bsr = lambda a: tb.Bsr(a.n_brows, a.bdim, a.row_ptr, a.col_idx, a.val).to(DEV)
    with tb.Context() as ctx:
        r = tb.solve(ctx, bsr(H), None if S is None else bsr(S), z, cols, ptr, rows, tol=tol, precision=prec, seed_shift=0, **kw)
        status, G = r.status.cpu().numpy(), r.G.cpu().numpy()
    assert r.rc == 0 and np.all(status == tb.TB_COL_CONVERGED), np.bincount(status)
    ex = dense.green_lu(H.to_dense(), None if S is None else S.to_dense(), z, cols)
    for c in range(len(cols)):
        e = ex[rl[c], c, :]
        assert np.abs(G[ptr[c]:ptr[c + 1]] - e).max() < bound * np.abs(e).max(), c


@pytest.mark.parametrize("prec,tol,bound", [(F, 1e-11, 1e-8), (D, 1e-11, 1e-8), (M, 1e-5, 2e-3)], ids=["fp64", "df64", "mixed"])
@pytest.mark.parametrize("spec", [wl.scaled(wl.C1_SYSTEM, L=7), wl.scaled(wl.C2_SYSTEM, L=5), wl.scaled(wl.C3_SYSTEM, n_sites=60)],
                         ids=["b1", "b4-overlap", "b9"])
def test_panel_seed_outside_the_spectrum(spec, prec, tol, bound):
    o = systems.build_system(spec, 11)
    _panel(o.H, o.S, 6, wl.midpoint_shifts(9, -60.0, 6.0, 0.2), prec, tol, bound)


def test_panel_seed_far_outside_the_spectrum_fp64():
    """The squares of the seed's residual leave FP64's range too (below 1e-154)."""
    o = systems.build_system(wl.scaled(wl.C1_SYSTEM, L=9), 11)
    _panel(o.H, o.S, 4, np.concatenate([[-60.0 + 0.1j], wl.midpoint_shifts(8, -6.0, 6.0, 0.05)]), F, 1e-11, 1e-8)


@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
def test_panel_seed_outside_the_spectrum_with_a_wide_overlap(prec):
    """The conjugate-gradient path (S = D S0 D, D from 0.3 to 2)."""
    o = systems.build_system(wl.scaled(wl.C2_SYSTEM, L=3), 3)
    S = o.S
    d = np.random.default_rng(1).uniform(0.3, 2.0, (S.n_brows, S.bdim))
    br = np.repeat(np.arange(S.n_brows), np.diff(S.row_ptr))
    S.val[:] = S.val * d[br][:, :, None] * d[S.col_idx][:, None, :]
    _panel(o.H, S, 5, wl.midpoint_shifts(7, -60.0, 6.0, 0.2), prec, 1e-11, 1e-8, inner_max=200)


@pytest.mark.parametrize("solver", [tb.TB_SOLVER_QMR])
@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
def test_panel_qmr_seed_outside_the_spectrum(solver, prec):
    """The quasi-residual bounds the residual up to sqrt(iterations) < 40."""
    o = systems.build_system(wl.scaled(wl.C2_SYSTEM, L=4), 11)
    _panel(o.H, o.S, 5, wl.midpoint_shifts(9, -60.0, 6.0, 0.2), prec, 1e-11, 4e-7, solver=solver)
