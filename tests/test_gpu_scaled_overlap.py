"""H and S scaled together leave G as it is divided by the scale; so do the spectral
bounds of S and the sweeps that use them: a small S takes as many refinement passes an
iteration as S itself (bounds from a Lanczos run that stopped at once take three times
as many, or fail and leave the solve to conjugate gradients, which count none).  Powers
of two scale every number of the solve exactly but those that meet a fixed bound: the
results agree to the bound of the solve, 1e-8."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"


@pytest.mark.parametrize("k", [-24, -40, 30])
def test_scaled_overlap_takes_sweeps(k):
    H, S, _ = tb.build_system(wl.scaled(wl.C2_SYSTEM, L=5), 3)
    z = wl.midpoint_shifts(4, -6.0, 6.0, 0.3)
    rows = np.array([0, 77, 300], np.int64)
    ptr = np.arange(4, dtype=np.int64)
    f = 2.0 ** k
    scaled = lambda A: tb.Bsr(A.n_brows, A.bdim, A.row_ptr, A.col_idx, A.val * f).to(DEV)
    with tb.Context() as ctx:
        a = tb.solve(ctx, H.to(DEV), S.to(DEV), z, rows, ptr, rows)
        b = tb.solve(ctx, scaled(H), scaled(S), z, rows, ptr, rows)
    assert a.rc == 0 and b.rc == 0
    per_iteration = lambda r: r.refinements / r.outer_iters
    assert 0 < per_iteration(a) and abs(per_iteration(b) / per_iteration(a) - 1) < 0.1
    Ga, Gb = a.G.cpu().numpy(), b.G.cpu().numpy() * f
    assert np.abs(Ga - Gb).max() < 1e-8 * np.abs(Ga).max()
