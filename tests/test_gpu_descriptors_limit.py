"""tb_descriptors at the largest subspaces that fit a CTA's 227 KB (b = 1, seven blocks a
row: 66 bytes an atom and 64 beside the kernel's own 208), against the FP64 oracle where a
number does not depend on the atoms beyond five hops, and numpy for the rest; one more
atom is TB_ERR_SIZE.  FP32 outputs: 1e-5 relative; sums of 3500 FP64 terms are below that."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl
from oracle import descriptors, systems
from oracle.subspace import hop_distances

DEV = "cuda:0"
LIMIT = 232448


def _run(n_atoms):
    spec = wl.scaled(wl.C1_SYSTEM, L=16)
    o = systems.build_system(spec, 3)
    H = tb.Bsr(o.H.n_brows, 1, o.H.row_ptr, o.H.col_idx, o.H.val)
    j = 2000
    dist = hop_distances(o.nbr_ptr, o.nbr, j, 64)
    sub = np.array(sorted(sorted(dist, key=lambda a: (dist[a], a))[:n_atoms]), np.int32)
    with tb.Context() as ctx:
        D = tb.descriptors(ctx, H.to(DEV), None, np.array([j], np.int64), np.array([6], np.int32),
                           np.array([0, n_atoms], np.int64), sub).cpu().numpy()[0]
    return o, j, sub, D


def test_largest_subspace():
    n = (LIMIT - 208 - 64) // 66
    o, j, sub, D = _run(n)
    ref = descriptors.descriptor(o, j, 6)
    same = [0, 2, 3, 4, 5, 6, 7, 8] + list(range(9, 17)) + [17, 22, 23]
    assert np.allclose(D[same], ref[same], rtol=1e-5, atol=1e-6)
    diag = np.array([o.H.val[k, 0, 0] for a in sub for k in range(o.H.row_ptr[a], o.H.row_ptr[a + 1]) if o.H.col_idx[k] == a])
    assert np.allclose(D[18:22], [diag.mean(), diag.std(), diag.min(), diag.max()], rtol=1e-5, atol=1e-6)
    assert np.allclose(D[[1, 24]], [np.log(n) / np.log(1000.0), n / 1000.0], rtol=1e-6)


def test_too_large_a_subspace():
    with pytest.raises(tb.TbError, match=str(tb.TB_ERR_SIZE)):
        _run((LIMIT - 64) // 66 + 1)


@pytest.mark.parametrize("n", [1, 2, 7])
def test_smallest_subspaces(n):
    """The sums that lie in the vectors' place need more than these vectors."""
    o, j, sub, D = _run(n)
    diag = np.array([o.H.val[k, 0, 0] for a in sub for k in range(o.H.row_ptr[a], o.H.row_ptr[a + 1]) if o.H.col_idx[k] == a])
    assert np.allclose(D[18:22], [diag.mean(), diag.std(), diag.min(), diag.max()], rtol=1e-5, atol=1e-5)
    if n == 7:
        hjj = float(D[8])
        assert np.isclose(D[9], np.sqrt(6.0), rtol=1e-5)  # m_2: six neighbours with hopping -1
