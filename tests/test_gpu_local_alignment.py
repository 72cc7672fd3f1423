"""The local solver's S values in device memory need no 16-byte boundary (H's do): the
same bits as from aligned ones, for every precision and block edge."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"


def _shifted(A):
    n = A.val.numel()
    buf = torch.empty(n + 1, dtype=torch.float64, device=DEV)
    buf[1:] = A.val.reshape(-1)
    val = buf[1:].view(A.val.shape)
    assert val.data_ptr() % 16 == 8
    return tb.Bsr(A.n_brows, A.bdim, A.row_ptr, A.col_idx, val)


@pytest.mark.parametrize("prec", [tb.TB_PREC_FP64, tb.TB_PREC_DF64, tb.TB_PREC_MIXED], ids=["fp64", "df64", "mixed"])
@pytest.mark.parametrize("spec", [wl.scaled(wl.C4_SYSTEM, n_sites=400), wl.scaled(wl.C2_SYSTEM, L=5)], ids=["fcc4", "sc4"])
def test_overlap_values_on_an_8_byte_boundary(spec, prec):
    H, S, _ = tb.build_system(spec, 3)
    rows = np.arange(3, H.n_rows, H.n_rows // 9).astype(np.int64)
    rad = np.full(len(rows), 2, np.int32)
    sptr, satoms = tb.local_subspaces(H, rows, rad)
    optr = np.arange(len(rows) + 1, dtype=np.int64)
    z = wl.midpoint_shifts(4, -6.0, 6.0, 0.2)
    Hd, Sd = H.to(DEV), S.to(DEV)
    tol = 1e-5 if prec == tb.TB_PREC_MIXED else 1e-10
    with tb.Context() as ctx:
        a = tb.solve_local(ctx, Hd, Sd, z, rows, sptr, satoms, optr, rows, tol=tol, precision=prec)
        b = tb.solve_local(ctx, Hd, _shifted(Sd), z, rows, sptr, satoms, optr, rows, tol=tol, precision=prec)
        assert a.rc == 0 and b.rc == 0
        assert torch.equal(torch.view_as_real(a.G), torch.view_as_real(b.G))
        with pytest.raises(tb.TbError):                  # H's values, as before
            tb.solve_local(ctx, _shifted(Hd), Sd, z, rows, sptr, satoms, optr, rows, tol=tol, precision=prec)
