"""Local solves with many kept rows in little memory: the solutions of a CTA's column on its
kept rows are the workspace's largest part, and eight CTAs to an SM (small subspaces)
would need four times what two do.  Where the memory does not hold them, fewer CTAs run:
the same bits, as a column's arithmetic is its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"


@pytest.mark.parametrize("overlap", [True, False], ids=["overlap", "identity"])
@pytest.mark.parametrize("prec", [tb.TB_PREC_FP64, tb.TB_PREC_DF64], ids=["fp64", "df64"])
def test_many_kept_rows_in_little_memory(prec, overlap):
    H, S, _ = tb.build_system(wl.scaled(wl.C2_SYSTEM, L=11), 3)
    n, nz, keep = 1300, 64, 2000
    rows = (4 * np.arange(n)).astype(np.int64)
    sptr, satoms = tb.local_subspaces(H, rows, np.full(n, 1, np.int32))
    kept = np.concatenate([np.resize(np.arange(28), keep), rows[1:]]).astype(np.int64)  # column 0 keeps rows many times
    optr = np.concatenate([[0], keep + np.arange(n)]).astype(np.int64)
    z = wl.midpoint_shifts(nz, -8.0, 6.0, 0.5)
    Hd, Sd = H.to(DEV), S.to(DEV) if overlap else None
    args = lambda ctx: tb.solve_local(ctx, Hd, Sd, z, rows, sptr, satoms, optr, kept, precision=prec)
    with tb.Context() as ctx:
        ref = args(ctx)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    cta = 2 * keep * nz * 16                              # 4 MB
    with tb.Context() as ctx:
        tb.solve_local(ctx, Hd, Sd, z, rows[:1], sptr[:2], satoms[:sptr[1]], optr[:2], kept[:keep], precision=prec)
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        want = 304 * cta + (512 << 20)                    # two CTAs for each of 152 SMs, and the rest
        assert want < 1216 * cta
        fill = torch.empty(free - want, dtype=torch.uint8, device=DEV)
        try:
            r = args(ctx)
        finally:
            del fill
            torch.cuda.empty_cache()
    assert r.rc == 0 and ref.rc == 0
    assert torch.equal(torch.view_as_real(r.G), torch.view_as_real(ref.G))
