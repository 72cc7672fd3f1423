"""tb_bsr_spmm at the edges of its kernels: every way a team of threads divides a
CTA (1..64 columns, even and odd), matrices smaller than a wave, values outside
the range of the integer conversions, X and Y that are not 16-byte aligned or
are the same array, and a malformed structure (Y stays as it was).

Bounds, relative to sum_k |a_ik| |x_kj|: FP64 products of at most 117 terms
117 * 2^-53 < 2e-14; df 117 * 2^-46 < 2e-12 and FP32 119 * 2^-24 < 1e-5, each
plus the smallest FP32 subnormal per term where operands underflow.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import paper_1402_7285_gb300 as tb
import workloads as wl

DEV = "cuda:0"
BOUND = {tb.TB_PREC_FP64: 2e-14, tb.TB_PREC_DF64: 2e-12, tb.TB_PREC_MIXED: 1e-5}
SPECS = [wl.scaled(wl.C1_SYSTEM, L=5), wl.scaled(wl.C2_SYSTEM, L=3), wl.scaled(wl.C3_SYSTEM, n_sites=40),
         wl.scaled(wl.C2_SYSTEM, L=22)]


def _dense_rows(H, X):
    b = H.bdim
    br = np.repeat(np.arange(H.n_brows), np.diff(H.row_ptr))
    Xb = X.reshape(H.n_brows, b, -1)
    Y, mag = np.zeros_like(Xb), np.zeros(Xb.shape)
    np.add.at(Y, br, np.einsum("kij,kjc->kic", H.val, Xb[H.col_idx]))
    ax = np.abs(Xb.real) + np.abs(Xb.imag)
    np.add.at(mag, br, np.einsum("kij,kjc->kic", np.abs(H.val), ax[H.col_idx]))
    return Y.reshape(X.shape), mag.reshape(X.shape)


@pytest.mark.parametrize("prec", list(BOUND))
@pytest.mark.parametrize("spec", SPECS, ids=["b1", "b4", "b9", "b4-wave"])
def test_spmm_column_counts_and_value_ranges(spec, prec):
    H, _, _ = tb.build_system(spec, 7)
    Hd = H.to(DEV)
    rng = np.random.default_rng(3)
    with tb.Context() as ctx:
        for ncols in (1, 2, 3, 7, 31, 33, 48, 63, 64):
            X = rng.standard_normal((H.n_rows, ncols)) + 1j * rng.standard_normal((H.n_rows, ncols))
            X[::3] *= 10.0 ** rng.integers(-60, 30, (len(X[::3]), 1))
            X[::5, 0] = 0.0
            X[1::7, 0] = 2.0 ** rng.integers(-160, 100, len(X[1::7]))
            Y = tb.bsr_spmm(ctx, Hd, torch.as_tensor(X, device=DEV), prec).cpu().numpy()
            ref, mag = _dense_rows(H, X)
            floor = 0.0 if prec == tb.TB_PREC_FP64 else 120 * 2.0 ** -149 * np.abs(H.val).max() * 4
            assert np.all(np.abs(Y - ref) <= BOUND[prec] * mag + floor), (ncols, prec)


@pytest.mark.parametrize("prec", list(BOUND))
def test_spmm_unaligned_in_place_and_malformed(prec):
    H, _, _ = tb.build_system(wl.scaled(wl.C2_SYSTEM, L=3), 7)
    Hd, ncols = H.to(DEV), 5
    n = H.n_rows * ncols * 2
    g = torch.Generator(device=DEV).manual_seed(1)
    x = torch.randn(n, dtype=torch.float64, device=DEV, generator=g)
    with tb.Context() as ctx:
        X = torch.view_as_complex(x.reshape(H.n_rows, ncols, 2))
        ref = tb.bsr_spmm(ctx, Hd, X, prec)
        stream = torch.cuda.current_stream().cuda_stream
        A = Hd.c_struct()

        def call(px, py):
            return ctx.lib.tb_bsr_spmm(ctx.h, ctypes.byref(A), px, ncols, py, prec, stream)

        buf = torch.zeros(2 * n + 3, dtype=torch.float64, device=DEV)
        buf[1:n + 1] = x
        assert call(buf[1:].data_ptr(), buf[n + 2:].data_ptr()) == 0   # the second is aligned or not, as n is even
        assert torch.equal(buf[n + 2:2 * n + 2], torch.view_as_real(ref).reshape(-1))
        assert call(buf[1:].data_ptr(), buf[n + 1:].data_ptr()) == 0
        assert torch.equal(buf[n + 1:2 * n + 1], torch.view_as_real(ref).reshape(-1))
        y = x.clone()
        assert call(y.data_ptr(), y.data_ptr()) == 0
        assert torch.equal(y, torch.view_as_real(ref).reshape(-1))
        ci = Hd.col_idx.clone()
        ci[3] = H.n_brows + 5
        bad = tb.Bsr(H.n_brows, H.bdim, Hd.row_ptr, ci, Hd.val)
        A = bad.c_struct()
        y.fill_(3.0)
        assert call(x.data_ptr(), y.data_ptr()) == tb.TB_ERR_STRUCTURE
        torch.cuda.synchronize()
        assert torch.all(y == 3.0)
        A = Hd.c_struct()                                               # the next check starts clean
        assert call(x.data_ptr(), y.data_ptr()) == 0
        assert torch.equal(y, torch.view_as_real(ref).reshape(-1))
