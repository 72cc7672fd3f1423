"""One context on two streams: a product returns with work queued, and a call on another
stream must leave that work's operands and its fault word alone.  The product's X is
not 16-byte aligned (FP64: it is copied first, 2 GB, so that the product starts long
after the call returned) or the product itself takes longer than the solve that
follows; the solve's S has diagonal blocks that are not the identity, and it takes
spectral bounds.  Same arrays, same kernels: the bits are those of the product alone.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"


def _solve_args():
    H, S, _ = tb.build_system(wl.scaled(wl.C2_SYSTEM, L=4), 3)
    d = np.random.default_rng(1).uniform(0.9, 1.1, (S.n_brows, S.bdim))
    br = np.repeat(np.arange(S.n_brows), np.diff(S.row_ptr))
    S.val[:] = S.val * d[br][:, :, None] * d[S.col_idx][:, None, :]
    rows = np.array([5], np.int64)
    return H.to(DEV), S.to(DEV), wl.midpoint_shifts(3, -8.0, 6.0, 0.5), rows, np.array([0, 1], np.int64), rows


@pytest.mark.parametrize("other", ["solve", "solve_local", "malformed_product"])
@pytest.mark.parametrize("prec", [tb.TB_PREC_FP64, tb.TB_PREC_DF64, tb.TB_PREC_MIXED], ids=["fp64", "df64", "mixed"])
def test_a_queued_product_and_a_call_on_another_stream(prec, other):
    H, _, _ = tb.build_system(wl.scaled(wl.C1_SYSTEM, L=128), 7)
    ncols = 64
    A = H.to(DEV)
    n = 2 * H.n_rows * ncols
    buf = torch.randn(n + 1, dtype=torch.float64, device=DEV)
    y, ref = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(2))
    h, s, z, rows, ptr, out = _solve_args()
    sub = np.arange(h.n_brows, dtype=np.int32)
    bad = tb.Bsr(h.n_brows, h.bdim, h.row_ptr, h.col_idx.clone(), h.val)
    bad.col_idx[3] = h.n_brows + 5
    small = torch.zeros(2 * h.n_rows * ncols, dtype=torch.float64, device=DEV)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with tb.Context() as ctx:
        def product(mat, px, py, stream):
            c = mat.c_struct()
            return ctx.lib.tb_bsr_spmm(ctx.h, ctypes.byref(c), px, ncols, py, prec, stream.cuda_stream)

        x = buf[1:].data_ptr()
        assert product(A, x, ref.data_ptr(), a) == 0
        torch.cuda.synchronize()
        with torch.cuda.stream(b):                       # every workspace has its size
            tb.solve(ctx, h, s, z, rows, ptr, out)
            tb.solve_local(ctx, h, s, z, rows, np.array([0, len(sub)], np.int64), sub, ptr, out)
        torch.cuda.synchronize()
        for _ in range(3):
            y.zero_()
            torch.cuda.synchronize()
            assert product(A, x, y.data_ptr(), a) == 0   # still at work when it returns
            if other == "malformed_product":
                assert product(bad, small.data_ptr(), small.data_ptr(), b) == tb.TB_ERR_STRUCTURE
            else:
                with torch.cuda.stream(b):
                    if other == "solve":
                        tb.solve(ctx, h, s, z, rows, ptr, out)
                    else:
                        tb.solve_local(ctx, h, s, z, rows, np.array([0, len(sub)], np.int64), sub, ptr, out)
            torch.cuda.synchronize()
            assert torch.equal(y, ref)
