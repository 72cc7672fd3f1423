"""The local solver's launch shapes against dense LU of the principal submatrices:
subspaces of one atom, sizes that leave threads idle, block edges 1, 4 and 9 (blocks
of 9 are stored transposed), own-row vectors in shared and in global memory (a
subspace too large for the first), several kept rows, more columns than CTAs, and
an overlap whose spectrum is too wide for Chebyshev sweeps.

tol 1e-11 leaves G within 1e-11 / eta = 1e-10 of the exact one; entries below the
largest by 1e-2 are compared on the largest one's scale, so 1e-8 of max|G| has a
margin of ten.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"
F, D = tb.TB_PREC_FP64, tb.TB_PREC_DF64


def _dense(A, atoms):
    b, n = A.bdim, len(atoms)
    loc = {int(a): i for i, a in enumerate(atoms)}
    out = np.zeros((n * b, n * b))
    for a, i in loc.items():
        for k in range(A.row_ptr[a], A.row_ptr[a + 1]):
            j = loc.get(int(A.col_idx[k]))
            if j is not None:
                out[i * b:(i + 1) * b, j * b:(j + 1) * b] = A.val[k]
    return out


def _check(H, S, radii, n, prec, keep=1, inner_max=0):
    rng = np.random.default_rng(5)
    rows = np.sort(rng.choice(H.n_rows, n, replace=False)).astype(np.int64)
    rad = rng.choice(np.asarray(radii), n).astype(np.int32)
    sptr, satoms = tb.local_subspaces(H, rows, rad)
    b = H.bdim
    kept = []
    for c, j in enumerate(rows):
        sub = satoms[sptr[c]:sptr[c + 1]].astype(np.int64)
        other = (sub[:, None] * b + np.arange(b)).ravel()[: keep - 1]
        kept.append(np.concatenate([[j], other]).astype(np.int64))
    optr = np.concatenate([[0], np.cumsum([len(k) for k in kept])]).astype(np.int64)
    z = wl.midpoint_shifts(5, -6.0, 6.0, 0.1)
    with tb.Context() as ctx:
        r = tb.solve_local(ctx, H.to(DEV), None if S is None else S.to(DEV), z, rows, sptr, satoms, optr,
                           np.concatenate(kept), tol=1e-11, precision=prec, inner_max=inner_max)
        assert r.rc == 0 and np.all(r.status.cpu().numpy() == tb.TB_COL_CONVERGED)
        G = r.G.cpu().numpy()
    for c in range(0, n, max(1, n // 12)):
        at = satoms[sptr[c]:sptr[c + 1]].astype(np.int64)
        Hd = _dense(H, at)
        Sd = np.eye(len(Hd)) if S is None else _dense(S, at)
        loc = lambda rr: np.searchsorted(at, rr // b) * b + rr % b
        e = np.zeros(len(Hd), complex)
        e[loc(rows[c])] = 1.0
        x = np.stack([np.linalg.solve(zz * Sd - Hd, e) for zz in z], axis=1)
        err = np.abs(G[optr[c]:optr[c + 1]] - x[loc(kept[c])]).max()
        assert err < 1e-8 * np.abs(x).max(), (c, err)


@pytest.mark.parametrize("prec", [F, D], ids=["fp64", "df64"])
@pytest.mark.parametrize("spec,radii,n,keep", [
    (wl.scaled(wl.C1_SYSTEM, L=7), (0, 1, 2), 30, 1),
    (wl.scaled(wl.C4_SYSTEM, n_sites=900), (0, 1, 2, 3), 40, 3),
    (wl.scaled(wl.C3_SYSTEM, n_sites=300), (0, 1, 2), 20, 1),
    (wl.scaled(wl.C2_SYSTEM, L=6), (1,), 700, 1),
], ids=["b1", "b4-overlap", "b9", "b4-many"])
def test_subspace_sizes(spec, radii, n, keep, prec):
    H, S, _ = tb.build_system(spec, 3)
    _check(H, S, radii, n, prec, keep)


@pytest.mark.parametrize("spec,radii,n", [
    (wl.scaled(wl.C3_SYSTEM, n_sites=2000), (5,), 3),     # 561 atoms of 9: p and u in global memory, 1024 threads
    (wl.scaled(wl.C5_SYSTEM, L=10), (5,), 4),             # 231 atoms of 4 with overlap
], ids=["b9-large", "b4-large"])
def test_large_subspaces(spec, radii, n):
    H, S, _ = tb.build_system(spec, 3)
    _check(H, S, radii, n, D)


def test_wide_overlap_spectrum_takes_conjugate_gradients():
    H, S, _ = tb.build_system(wl.scaled(wl.C4_SYSTEM, n_sites=600), 3)
    d = np.random.default_rng(1).uniform(0.3, 2.0, (S.n_brows, S.bdim))
    br = np.repeat(np.arange(S.n_brows), np.diff(S.row_ptr))
    S.val[:] = S.val * d[br][:, :, None] * d[S.col_idx][:, None, :]
    _check(H, S, (1, 2), 20, F, inner_max=300)
