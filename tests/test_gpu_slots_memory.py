"""FP64 and df panels of 33 to 64 columns take as many slots as columns, and 32 where the
memory does not hold the arrays of 64, whichever array that is: with whole solution
vectors the kept-row solutions are the largest by far."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"


@pytest.mark.parametrize("prec", [tb.TB_PREC_FP64, tb.TB_PREC_DF64], ids=["fp64", "df64"])
def test_whole_vectors_in_little_memory(prec):
    H, S, _ = tb.build_system(wl.scaled(wl.C1_SYSTEM, L=20), 3)
    n, nz = 64, 32                                   # 8000 rows x 32 shifts x 32 bytes a slot: 8.2 MB
    slot = H.n_rows * nz * 32
    cols = np.arange(0, H.n_rows, H.n_rows // n)[:n].astype(np.int64)
    kept = np.concatenate([np.arange(H.n_rows) if c == 0 else np.array([j]) for c, j in enumerate(cols)]).astype(np.int64)
    ptr = np.concatenate([[0, H.n_rows], H.n_rows + np.arange(1, n)]).astype(np.int64)
    z = wl.midpoint_shifts(nz, -7.0, 7.0, 1.0)
    Hd = H.to(DEV)
    with tb.Context() as ctx:
        ref = tb.solve(ctx, Hd, None, z, cols, ptr, kept, precision=prec, panel_w=32)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with tb.Context() as ctx:
        tb.solve(ctx, Hd, None, z, cols[:1], np.array([0, 1], np.int64), cols[:1], precision=prec)  # modules, small arrays
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        # 32 slots' solutions and vectors (16 bytes x 3 a row) with room for the rest, half of 64 slots' short
        want = 32 * slot + 32 * H.n_rows * 48 + (128 << 20)
        assert want < 64 * slot
        fill = torch.empty(free - want, dtype=torch.uint8, device=DEV)
        try:
            r = tb.solve(ctx, Hd, None, z, cols, ptr, kept, precision=prec)
            with pytest.raises(tb.TbError, match="-3"):  # asked for, they are refused
                tb.solve(ctx, Hd, None, z, cols, ptr, kept, precision=prec, panel_w=64)
        finally:
            del fill
            torch.cuda.empty_cache()
    assert r.rc == 0 and ref.rc == 0
    assert torch.equal(torch.view_as_real(r.G), torch.view_as_real(ref.G))
