"""An eigenvalue of S that the Lanczos bounds cannot see.  Row R0 is coupled to no other
row by S, and its entry of the bounds' fixed start vector is exactly zero (the
hash of that row), so no Krylov vector has a part there.  A sweep on those bounds grows
on that row, to a large residual (S_rr = 4) or until FP32 overflows (1e6); the solve
then has to take conjugate gradients, as if the spectrum were known to be wide.

Oracle: dense FP64 solutions of the seven rows that H couples R0 to (all else is decoupled
from them).  tol 1e-10, eta 0.5, entries of G up to 2: 1e-8 of the largest, a margin of 50.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"
R0, N = 2354591, 2354600


def _start_value(r):
    h = (r * 2654435761) % 2 ** 32
    h ^= h >> 15
    h = h * 0x85ebca6b % 2 ** 32
    h ^= h >> 13
    return (h & 0xffffff) / 8388608.0 - 1.0


def _system(srr):
    """b = 1: rows R0 - 3 .. R0 + 3 a chain in H (not in S); all other rows pairs with overlap 0.1."""
    assert _start_value(R0) == 0.0
    lo, hi = R0 - 3, R0 + 4
    r = np.arange(N)
    partner = r ^ 1
    inside = (r >= lo) & (r < hi)
    paired = ~inside & (partner < N) & ~((partner >= lo) & (partner < hi))
    i = np.concatenate([r, r[paired], r[lo:hi - 1], r[lo + 1:hi]])
    j = np.concatenate([r, partner[paired], r[lo + 1:hi], r[lo:hi - 1]])
    h = np.concatenate([0.3 * np.cos(r), np.full(paired.sum(), -0.5), np.full(2 * (hi - lo - 1), 0.7)])
    s = np.concatenate([np.where(r == R0, srr, 1.0), np.full(paired.sum(), 0.1), np.zeros(2 * (hi - lo - 1))])
    o = np.lexsort((j, i))
    rp = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=N))]).astype(np.int64)
    mat = lambda v: tb.Bsr(N, 1, rp, j[o].astype(np.int32), v[o].reshape(-1, 1, 1).copy())
    return mat(h), mat(s)


@pytest.mark.parametrize("local", [False, True], ids=["panel", "local"])
@pytest.mark.parametrize("prec", [tb.TB_PREC_FP64, tb.TB_PREC_DF64], ids=["fp64", "df64"])
@pytest.mark.parametrize("srr", [4.0, 1e6])
def test_outlier_falls_back_to_conjugate_gradients(srr, prec, local):
    H, S = _system(srr)
    frag = np.arange(R0 - 3, R0 + 4)
    rows = np.array([R0, R0 - 1, 10], np.int64)
    kept = [frag, frag, np.array([10, 11])]
    optr = np.array([0, 7, 14, 16], np.int64)
    z = wl.midpoint_shifts(3, -1.5, 1.5, 0.5)
    with tb.Context() as ctx:
        if local:
            sub = np.concatenate(kept).astype(np.int32)
            res = tb.solve_local(ctx, H.to(DEV), S.to(DEV), z, rows, optr, sub, optr, np.concatenate(kept), precision=prec)
        else:
            res = tb.solve(ctx, H.to(DEV), S.to(DEV), z, rows, optr, np.concatenate(kept), precision=prec)
        G, status = res.G.cpu().numpy(), res.status.cpu().numpy()
    assert res.rc == 0 and np.all(status == tb.TB_COL_CONVERGED), status
    if prec == tb.TB_PREC_FP64:
        assert res.refinements == 0                      # the rerun's counts: conjugate gradients alone

    def dense(A, at):
        out = np.zeros((len(at), len(at)))
        for a, q in enumerate(at):
            for k in range(A.row_ptr[q], A.row_ptr[q + 1]):
                b = np.searchsorted(at, A.col_idx[k])
                if b < len(at) and at[b] == A.col_idx[k]:
                    out[a, b] = A.val[k, 0, 0]
        return out

    for c, j in enumerate(rows):
        at = kept[c]
        e = (at == j).astype(float)
        x = np.stack([np.linalg.solve(zz * dense(S, at) - dense(H, at), e) for zz in z], axis=1)
        err = np.abs(G[optr[c]:optr[c + 1]] - x).max()
        assert err < 1e-8 * np.abs(x).max(), (c, err)
