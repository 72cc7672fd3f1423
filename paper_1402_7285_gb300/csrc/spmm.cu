// tb_bsr_spmm: Y = A X for a real BSR matrix and a complex panel (FP64, FP32 or df).
#include "spmm.cuh"
#include "dispatch.cuh"

namespace {

using tbgf::bsr_row_fault;

constexpr int SNT = 256;

// ------------------------------------------------------------- conversions
// FP64 <-> FP32 and FP64 <-> df conversions on the integer and FP32 pipes: GB300
// converts to and from 64-bit types at its FP64 rate (about 2 per clock and SM),
// which made the conversions of an sp+d df panel (180,000 x 33) take 237 us, 3.5
// times what their bytes need.  Each gives the bits of the conversion it stands
// for; numbers outside the range where the integer form holds (zeros, values
// whose FP32 parts are not normal numbers, infinities, NaN) take the conversion
// itself.
// (Calls, not selects: inlined, both forms run for every value.)
__device__ __noinline__ float cast_f32(double v) { return (float)v; }
__device__ __noinline__ double cast_f64(float v) { return (double)v; }
__device__ __noinline__ double cast_f64(df v) { return (double)v.hi + (double)v.lo; }
__device__ __noinline__ df cast_df(double v) { return df(v); }

__device__ __forceinline__ float cvt_f32(double v) {
    const uint64_t w = (uint64_t)__double_as_longlong(v), u = w & 0x7fffffffffffffffull;
    // round to nearest even at bit 29, then rebias the exponent (1023 - 127 = 896)
    const uint64_t r = u + 0x0fffffffull + ((u >> 29) & 1);
    const uint32_t f = (uint32_t)(r >> 29) - (896u << 23);
    if (u - (897ull << 52) < ((1150ull - 897ull) << 52)) // result in the normal range, with room for the carry
        return __uint_as_float(f | ((uint32_t)(w >> 32) & 0x80000000u));
    return cast_f32(v);
}

__device__ __forceinline__ double cvt_f64(float x) {
    const uint32_t w = __float_as_uint(x), u = w & 0x7fffffffu;
    if (u - 0x00800000u < 0x7f000000u) // a normal number
        return __longlong_as_double((long long)(((uint64_t)(w & 0x80000000u) << 32) | (((uint64_t)u << 29) + (896ull << 52))));
    return cast_f64(x);
}

// v = hi + lo: hi the rounded FP32 value; what is left of the mantissa is an
// integer below 2^29 in units of 2^(e - 52), rounded to FP32 as (float)(v - hi) is
__device__ __forceinline__ df cvt_df(double v) {
    const uint64_t w = (uint64_t)__double_as_longlong(v), u = w & 0x7fffffffffffffffull;
    const uint64_t r = u + 0x0fffffffull + ((u >> 29) & 1);
    // exponents for which hi, 2^(e - 52) and every non-zero lo are normal numbers
    if (u == 0) return df(0.f, 0.f); // onsite blocks hold many
    if (u - (960ull << 52) < ((1149ull - 960ull) << 52)) {
        const uint32_t sg = (uint32_t)(w >> 32) & 0x80000000u;
        const uint32_t f = (uint32_t)(r >> 29) - (896u << 23);
        const int rem = (int)(uint32_t)(u - ((r >> 29) << 29)); // |rem| <= 2^28
        const float unit = __uint_as_float(((uint32_t)(u >> 52) - (896u + 52u)) << 23);
        const float lo = __fmul_rn((float)rem, unit);
        return df(__uint_as_float(f | sg), sg ? -lo : lo);
    }
    return cast_df(v);
}

// hi + lo rounded to FP64: lo counts in units of hi's last FP64 bit
__device__ __forceinline__ double cvt_f64(df x) {
    const uint32_t w = __float_as_uint(x.hi), u = w & 0x7fffffffu, e = u >> 23;
    // hi normal and large enough for its FP64 unit's reciprocal to be an FP32 number; not a power
    // of two (below one the unit halves); |lo| at most an ulp of hi (2^29 units)
    if (e >= 54u && e <= 250u && (u & 0x7fffffu)) {
        const float q = __fmul_rn(w >> 31 ? -x.lo : x.lo, __uint_as_float((127u + 52u + 127u - e) << 23));
        if (fabsf(q) <= 268435456.f) {
            const uint64_t m = ((uint64_t)u << 29) + (896ull << 52) + (uint64_t)(int64_t)__float2int_rn(q);
            return __longlong_as_double((long long)(((uint64_t)(w & 0x80000000u) << 32) | m));
        }
    }
    return cast_f64(x);
}
__device__ __forceinline__ double cvt_f64(double x) { return x; }

__device__ __forceinline__ void cvt_to(double v, float &x) { x = cvt_f32(v); }
__device__ __forceinline__ void cvt_to(double v, df &x) { x = cvt_df(v); }

// dst[t] = src[t] for n doubles; two a thread where src and dst allow the wide accesses
template <typename T>
__device__ void convert_span(const double *__restrict__ src, T *__restrict__ dst, int64_t n) {
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const bool wide = ((uintptr_t)src & 15) == 0; // dst is the library's own, 256-byte aligned
    const int64_t n2 = wide ? n / 2 : 0;
#pragma unroll 4
    for (int64_t t = tid; t < n2; t += stride) {
        const double2 v = __ldcs(reinterpret_cast<const double2 *>(src) + t);
        T a, b;
        cvt_to(v.x, a);
        cvt_to(v.y, b);
        if constexpr (sizeof(T) == 4)
            reinterpret_cast<float2 *>(dst)[t] = make_float2(a, b);
        else
            reinterpret_cast<float4 *>(dst)[t] = make_float4(a.hi, a.lo, b.hi, b.lo);
    }
    for (int64_t t = 2 * n2 + tid; t < n; t += stride) cvt_to(src[t], dst[t]);
}

template <typename T>
__global__ void __launch_bounds__(SNT) k_convert(const double *src, T *dst, int64_t n) {
    convert_span(src, dst, n);
}

// dst block (j, i) = src block (i, j), b x b blocks: the rows of a block become neighbours
template <typename T>
__global__ void __launch_bounds__(SNT) k_convert_t(const double *__restrict__ src, T *__restrict__ dst, int64_t n, int b) {
    const int bb = b * b;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / bb;
        const int r = (int)(t - k * bb), j = r / b, i = r - j * b;
        cvt_to(src[k * bb + i * b + j], dst[t]);
    }
}

// First launch of a product: the structure check of A and, for FP32 and df, the
// conversion of A's values and of X.
template <typename T>
__global__ void __launch_bounds__(SNT) k_spmm_prep(const int64_t *rp, const int32_t *ci, int64_t n_brows, int64_t nnzb,
                                                   int *words, int *host, const double *val, T *vdst, int64_t nval,
                                                   const double *X, T *xdst, int64_t nx) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < n_brows; a += stride)
        if (const int f = bsr_row_fault(rp, ci, n_brows, nnzb, a)) atomicOr(words, f);
    if constexpr (!std::is_same<T, double>::value) {
        convert_span(val, vdst, nval);
        convert_span(X, xdst, nx);
    }
    publish_check(words, host, words + 2);
}

// ------------------------------------------------------------------ product
// CPT consecutive complex values at element e of a panel
template <typename T, int CPT>
__device__ __forceinline__ void ld_cpx(const T *__restrict__ base, int64_t e, cpx<T> (&x)[CPT]) {
    if constexpr (std::is_same<T, df>::value) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(base) + e);
        x[0] = mk(df(v.x, v.y), df(v.z, v.w));
    } else if constexpr (std::is_same<T, double>::value) {
        const double2 v = __ldg(reinterpret_cast<const double2 *>(base) + e);
        x[0] = mk(v.x, v.y);
    } else if constexpr (CPT == 2) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(base + 2 * e));
        x[0] = mk(v.x, v.y), x[1] = mk(v.z, v.w);
    } else {
        const float2 v = __ldg(reinterpret_cast<const float2 *>(base) + e);
        x[0] = mk(v.x, v.y);
    }
}

// the RPT x B values of rows i0.. of a block (16-byte loads where rows allow them)
template <typename T, int B, int RPT>
__device__ __forceinline__ void ld_rows(const T *__restrict__ blk, int i0, T (&a)[RPT * B]) {
    const T *r = blk + i0 * B;
    if constexpr ((B * sizeof(T)) % 16 == 0) {
        constexpr int PER = 16 / sizeof(T);
#pragma unroll
        for (int q = 0; q < RPT * B / PER; ++q) {
            if constexpr (std::is_same<T, df>::value) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(r) + q);
                a[2 * q] = df(v.x, v.y), a[2 * q + 1] = df(v.z, v.w);
            } else if constexpr (sizeof(T) == 4) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(r) + q);
                a[4 * q] = v.x, a[4 * q + 1] = v.y, a[4 * q + 2] = v.z, a[4 * q + 3] = v.w;
            } else {
                const double2 v = __ldg(reinterpret_cast<const double2 *>(r) + q);
                a[2 * q] = v.x, a[2 * q + 1] = v.y;
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < RPT * B; ++q) a[q] = ldg_val(r + q);
    }
}

// Y = A X.  A team of ncols / CPT threads owns RPT rows of one block row at a
// time (CPT columns a thread), so any number of columns runs without padding:
// FP64 reads X and writes Y in place of two padded copies, FP32 and df read
// the panel that k_spmm_prep converted and write Y in FP64.  Rows of a thread:
// FP64 one (the FP64 pipe sets the time, and one row a thread spreads a small
// matrix over all SMs), FP32 and df a block row of b = 4 (each x is read once
// per block), three of b = 9 (nine rows hold 81 values and spill).  Where the
// matrix does not fill the chip, one row each.  What bounds it: FP32 the loads of
// X from L2 (each neighbour row once per referencing block), FP64 its pipe, df
// the register reads of its 12 FP32 operations per term (issue 62-69 %, the rest
// dispatch stalls; packed f32x2 operations and loads a block ahead were measured
// and change nothing).  Whole calls, before (padded copies, allocated check flag)
// and now: 1331 x 3 FP64 260 -> 37 us; b = 4, 131072 x 64, FP32 258 -> 107 us (45 us at
// the copy rate; the product 61, the conversion 45); b = 9, 180099 x 33, df 1532 -> 822 us.
template <typename T, int B, int RPT, int CPT, typename OUT, int MINB>
__global__ void __launch_bounds__(SNT, MINB) k_spmm(const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                                    const T *__restrict__ val, int64_t n_brows,
                                                    const T *__restrict__ X, OUT *__restrict__ Y, int ncols,
                                                    const int *__restrict__ bad) {
    if (bad && *bad) return; // malformed structure: the host reports it
    constexpr int G = B / RPT;
    const int lanes = ncols / CPT, teams = SNT / lanes;
    const int team = threadIdx.x / lanes, c0 = (threadIdx.x % lanes) * CPT;
    if (team >= teams) return;
    const int64_t units = n_brows * G, step = (int64_t)gridDim.x * teams;
    for (int64_t w = (int64_t)blockIdx.x * teams + team; w < units; w += step) {
        const int64_t br = w / G;
        const int i0 = (int)(w % G) * RPT;
        const int64_t k0 = __ldg(rp + br), k1 = __ldg(rp + br + 1);
        typedef typename std::conditional<std::is_same<T, df>::value, DfSum, T>::type A;
        A sr[RPT][CPT], si[RPT][CPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i)
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                if constexpr (std::is_same<T, df>::value)
                    sr[i][c].zero(), si[i][c].zero();
                else
                    sr[i][c] = si[i][c] = 0;
            }
        int64_t col_n = k0 < k1 ? (int64_t)__ldg(ci + k0) : 0;
#pragma unroll(B <= 4 ? 2 : 1)
        for (int64_t k = k0; k < k1; ++k) {
            const int64_t col = col_n;
            if (k + 1 < k1) col_n = __ldg(ci + k + 1);
            cpx<T> x[B][CPT];
#pragma unroll
            for (int j = 0; j < B; ++j) ld_cpx<T, CPT>(X, (col * B + j) * ncols + c0, x[j]);
            T a[RPT * B];
            ld_rows<T, B, RPT>(val + k * (int64_t)(B * B), i0, a);
#pragma unroll
            for (int i = 0; i < RPT; ++i)
#pragma unroll
                for (int j = 0; j < B; ++j)
#pragma unroll
                    for (int c = 0; c < CPT; ++c) {
                        if constexpr (std::is_same<T, df>::value) {
                            sr[i][c].add_prod(a[i * B + j], x[j][c].re);
                            si[i][c].add_prod(a[i * B + j], x[j][c].im);
                        } else {
                            sr[i][c] = fma(a[i * B + j], x[j][c].re, sr[i][c]);
                            si[i][c] = fma(a[i * B + j], x[j][c].im, si[i][c]);
                        }
                    }
        }
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int64_t e = (br * B + i0 + i) * ncols + c0;
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                T re, im;
                if constexpr (std::is_same<T, df>::value)
                    re = sr[i][c].value(), im = si[i][c].value();
                else
                    re = sr[i][c], im = si[i][c];
                if constexpr (std::is_same<OUT, double>::value)
                    __stcs(reinterpret_cast<double2 *>(Y) + e + c, make_double2(cvt_f64(re), cvt_f64(im)));
                else if constexpr (std::is_same<OUT, df>::value)
                    reinterpret_cast<float4 *>(Y)[e + c] = make_float4(re.hi, re.lo, im.hi, im.lo);
                else
                    reinterpret_cast<float2 *>(Y)[e + c] = make_float2(re, im);
            }
        }
    }
}

// x(r, c) = deterministic test values in [-1, 1) (a cheap integer hash)
template <typename T>
__global__ void k_fill_panel(T *__restrict__ x, int64_t n2) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n2; t += (int64_t)gridDim.x * blockDim.x) {
        uint32_t h = (uint32_t)t * 2654435761u;
        h ^= h >> 15;
        x[t] = (T)((double)(h & 0xffffff) / 8388608.0 - 1.0);
    }
}

int sm_count();

struct SpmmLaunch {
    const int64_t *rp;
    const int32_t *ci;
    const void *val;
    int64_t n_brows;
    const void *X;
    void *Y;
    int ncols;
    const int *bad;
    cudaStream_t s;

    template <typename T, int B, int RPT, int CPT, typename OUT, int MINB>
    void go() {
        const int teams = SNT / (ncols / CPT);
        const int64_t need = (n_brows * (B / RPT) + teams - 1) / teams;
        // one wave of resident CTAs (FP32 on C2: 8 % faster than two waves)
        const int g = (int)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sm_count() * MINB));
        k_spmm<T, B, RPT, CPT, OUT, MINB><<<g, SNT, 0, s>>>(rp, ci, (const T *)val, n_brows, (const T *)X, (OUT *)Y, ncols, bad);
    }
    // rows of a thread: RPT, or one where RPT would leave SMs with less than two CTAs
    template <typename T, int B, int RPT, int CPT, typename OUT>
    void rows() {
        constexpr int MINB = std::is_same<T, df>::value ? 3 : 4;
        if (RPT > 1 && n_brows * (B / RPT) * (ncols / CPT) < (int64_t)sm_count() * 2 * SNT)
            go<T, B, 1, CPT, OUT, 4>();
        else
            go<T, B, RPT, CPT, OUT, MINB>();
    }
    template <typename T, int B, typename OUT>
    void cols() {
        if constexpr (std::is_same<T, float>::value) {
            if (ncols % 2 == 0) return rows<T, B, B == 9 ? 3 : B, 2, OUT>();
            return rows<T, B, B == 9 ? 3 : B, 1, OUT>();
        } else if constexpr (std::is_same<T, df>::value) {
            rows<T, B, B == 9 ? 3 : B, 1, OUT>();
        } else {
            rows<T, B, 1, 1, OUT>();
        }
    }
    template <typename T, typename OUT>
    void run(int b) {
        if (b == 1) cols<T, 1, OUT>();
        else if (b == 4) cols<T, 4, OUT>();
        else cols<T, 9, OUT>();
    }
};

int sm_count() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
    }
    return sms;
}

} // namespace

namespace tbgf {
void convert_values(int precision, const double *src, void *dst, int64_t n, cudaStream_t s) {
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n / 2 + SNT - 1) / SNT, 152 * 8));
    if (precision == TB_PREC_MIXED)
        k_convert<float><<<g, SNT, 0, s>>>(src, (float *)dst, n);
    else if (precision == TB_PREC_DF64)
        k_convert<df><<<g, SNT, 0, s>>>(src, (df *)dst, n);
}
void convert_values_t(int precision, const double *src, void *dst, int64_t n, int b, cudaStream_t s) {
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n + SNT - 1) / SNT, 152 * 8));
    if (precision == TB_PREC_MIXED)
        k_convert_t<float><<<g, SNT, 0, s>>>(src, (float *)dst, n, b);
    else
        k_convert_t<df><<<g, SNT, 0, s>>>(src, (df *)dst, n, b);
}
} // namespace tbgf

extern "C" int tb_bsr_spmm(tb_ctx *ctx, const tb_bsr *A, const double *X, int32_t ncols, double *Y,
                           int32_t precision, void *stream) {
    using namespace tbgf;
    if (!ctx) return TB_ERR_ARG;
    TB_CHECK(ctx, A && A->row_ptr && A->col_idx && A->val, TB_ERR_ARG, "tb_bsr_spmm: matrix arrays missing");
    TB_CHECK(ctx, X && Y && ncols >= 1 && ncols <= 64, TB_ERR_ARG, "tb_bsr_spmm: ncols must be 1..64");
    TB_CHECK(ctx, precision == TB_PREC_FP64 || precision == TB_PREC_MIXED || precision == TB_PREC_DF64, TB_ERR_ARG,
             "bad precision");
    TB_CHECK(ctx, supported_bdim(A->bdim), TB_ERR_UNSUPPORTED, "tb_bsr_spmm: bdim %d not built", A->bdim);
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n = A->n_brows * A->bdim;
    const int64_t bb = (int64_t)A->bdim * A->bdim;
    Stager st(ctx, WS_STAGE_IN, s);
    void *rp, *ci, *val, *x, *y;
    st.add(A->row_ptr, sizeof(int64_t) * (A->n_brows + 1), true, false, &rp);
    st.add(A->col_idx, sizeof(int32_t) * A->nnzb, true, false, &ci);
    st.add(A->val, sizeof(double) * A->nnzb * bb, true, false, &val);
    st.add(X, sizeof(double) * 2 * n * ncols, true, false, &x);
    st.add(Y, sizeof(double) * 2 * n * ncols, false, true, &y);
    int rc = st.commit();
    if (rc) return rc;
    TB_CHECK(ctx, ((uintptr_t)val & 15u) == 0, TB_ERR_ARG, "A values must be 16-byte aligned");
    TB_CHECK(ctx, A->n_brows > 0 && A->nnzb >= 0, TB_ERR_STRUCTURE, "A: bad sizes");
    const bool f32 = precision == TB_PREC_MIXED, dfp = precision == TB_PREC_DF64;
    const size_t esz = f32 ? 4 : 8;
    const int64_t nx = 2 * n * ncols;
    // FP32 and df work on converted copies of A's values and X.  FP64 works on the caller's arrays, unless X or Y
    // is not aligned for 16-byte accesses or they overlap: then on copies.
    const char *xb = (const char *)x, *yb = (const char *)y;
    const bool overlap = xb < yb + 8 * nx && yb < xb + 8 * nx;
    const bool copy_x = f32 || dfp || overlap || ((uintptr_t)x & 15u), copy_y = ((uintptr_t)y & 15u) != 0;
    const size_t off_x = (f32 || dfp) ? align_up(esz * A->nnzb * bb, 256) : 0;
    const size_t off_y = off_x + (copy_x ? align_up(esz * nx, 256) : 0);
    void *wsp;
    rc = ws_get(ctx, WS_SPMM_STAGE, off_y + (copy_y ? sizeof(double) * nx : 0), &wsp);
    if (rc) return rc;
    char *ws = (char *)wsp;
    int *words = nullptr, *host = nullptr, fault = 0;
    rc = check_words(ctx, &words, &host);
    if (rc) return rc;
    StageOrder order(ctx, s);
    if (order.rc) return order.rc;
    const int64_t items = std::max<int64_t>(A->n_brows, (f32 || dfp) ? nx / 4 : 0);
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((items + SNT - 1) / SNT, (int64_t)sm_count() * 8));
    const int64_t nv = A->nnzb * bb;
    if (f32)
        k_spmm_prep<float><<<g, SNT, 0, s>>>((const int64_t *)rp, (const int32_t *)ci, A->n_brows, A->nnzb, words, host,
                                             (const double *)val, (float *)ws, nv, (const double *)x,
                                             (float *)(ws + off_x), nx);
    else if (dfp)
        k_spmm_prep<df><<<g, SNT, 0, s>>>((const int64_t *)rp, (const int32_t *)ci, A->n_brows, A->nnzb, words, host,
                                          (const double *)val, (df *)ws, nv, (const double *)x, (df *)(ws + off_x), nx);
    else
        k_spmm_prep<double><<<g, SNT, 0, s>>>((const int64_t *)rp, (const int32_t *)ci, A->n_brows, A->nnzb, words,
                                              host, nullptr, nullptr, 0, nullptr, nullptr, 0);
    TB_CUDA_TRY(ctx, cudaGetLastError());
    TB_CUDA_TRY(ctx, cudaEventRecord(ctx->chk_ev, s));
    // the product is queued behind the check, and does nothing if that found a fault
    if (copy_x && !f32 && !dfp)
        TB_CUDA_TRY(ctx, cudaMemcpyAsync(ws + off_x, x, sizeof(double) * nx, cudaMemcpyDeviceToDevice, s));
    SpmmLaunch L{(const int64_t *)rp, (const int32_t *)ci, (f32 || dfp) ? ws : val, A->n_brows,
                 copy_x ? ws + off_x : x, copy_y ? ws + off_y : y, ncols, words + 2, s};
    if (f32)
        L.run<float, double>(A->bdim);
    else if (dfp)
        L.run<df, double>(A->bdim);
    else
        L.run<double, double>(A->bdim);
    TB_CUDA_TRY(ctx, cudaGetLastError());
    TB_CUDA_TRY(ctx, cudaEventSynchronize(ctx->chk_ev));
    fault = *ctx->chk_host;
    if (fault) {
        // staged host outputs are not copied back
        return set_error(ctx, TB_ERR_STRUCTURE, "A: malformed BSR structure (code %d)", fault);
    }
    if (copy_y) TB_CUDA_TRY(ctx, cudaMemcpyAsync(y, ws + off_y, sizeof(double) * nx, cudaMemcpyDeviceToDevice, s));
    return st.finish();
}

extern "C" int tb_bsr_spmm_profile(tb_ctx *ctx, const tb_bsr *A, int32_t ncols, int32_t precision, int32_t reps,
                                   void *stream, double *ms_per_launch) {
    using namespace tbgf;
    if (!ctx) return TB_ERR_ARG;
    TB_CHECK(ctx, A && A->row_ptr && A->col_idx && A->val, TB_ERR_ARG, "tb_bsr_spmm_profile: matrix arrays missing");
    TB_CHECK(ctx, ncols >= 1 && ncols <= 64 && reps >= 1 && ms_per_launch, TB_ERR_ARG,
             "tb_bsr_spmm_profile: ncols 1..64, reps >= 1, output required");
    TB_CHECK(ctx, precision == TB_PREC_FP64 || precision == TB_PREC_MIXED || precision == TB_PREC_DF64, TB_ERR_ARG,
             "bad precision");
    TB_CHECK(ctx, supported_bdim(A->bdim), TB_ERR_UNSUPPORTED, "tb_bsr_spmm_profile: bdim %d not built", A->bdim);
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n = A->n_brows * A->bdim;
    const int64_t bb = (int64_t)A->bdim * A->bdim;
    Stager st(ctx, WS_STAGE_IN, s);
    void *rp, *ci, *val;
    st.add(A->row_ptr, sizeof(int64_t) * (A->n_brows + 1), true, false, &rp);
    st.add(A->col_idx, sizeof(int32_t) * A->nnzb, true, false, &ci);
    st.add(A->val, sizeof(double) * A->nnzb * bb, true, false, &val);
    int rc = st.commit();
    if (rc) return rc;
    rc = validate_bsr(ctx, (const int64_t *)rp, (const int32_t *)ci, val, A->n_brows, A->nnzb, s, "A");
    if (rc) return rc;
    const int W = panel_width_for(ncols);
    const bool f32 = precision == TB_PREC_MIXED, dfp = precision == TB_PREC_DF64;
    const size_t esz = f32 ? 4 : 8;
    size_t off_val = 0, off_x = (f32 || dfp) ? align_up(esz * A->nnzb * bb, 256) : 0;
    size_t off_y = off_x + align_up(esz * 2 * n * W, 256);
    // a buffer twice the L2 size, written before every timed launch, so no
    // launch finds the previous launch's panel or matrix in L2
    const size_t flush_bytes = (size_t)256 << 20;
    const size_t off_flush = align_up(off_y + esz * 2 * n * W, 256);
    void *wsp;
    rc = ws_get(ctx, WS_SPMM_STAGE, off_flush + flush_bytes, &wsp);
    if (rc) return rc;
    char *ws = (char *)wsp;
    StageOrder order(ctx, s);
    if (order.rc) return order.rc;
    const void *mval = val;
    if (f32 || dfp) {
        convert_values(precision, (const double *)val, ws + off_val, A->nnzb * bb, s);
        mval = ws + off_val;
    }
    const int g = (int)std::min<int64_t>((2 * n * W + 255) / 256, 152 * 16);
    if (f32)
        k_fill_panel<float><<<g, 256, 0, s>>>((float *)(ws + off_x), 2 * n * W);
    else if (dfp)
        k_fill_panel<df><<<g, 256, 0, s>>>((df *)(ws + off_x), 2 * n * W);
    else
        k_fill_panel<double><<<g, 256, 0, s>>>((double *)(ws + off_x), 2 * n * W);
    SpmmLaunch L{(const int64_t *)rp, (const int32_t *)ci, mval, A->n_brows, ws + off_x, ws + off_y, W, nullptr, s};
    auto launch = [&]() { // panel to panel, in the working precision
        if (f32)
            L.run<float, float>(A->bdim);
        else if (dfp)
            L.run<df, df>(A->bdim);
        else
            L.run<double, double>(A->bdim);
    };
    launch();
    cudaEvent_t e0, e1;
    TB_CUDA_TRY(ctx, cudaEventCreate(&e0));
    TB_CUDA_TRY(ctx, cudaEventCreate(&e1));
    double total = 0.0;
    cudaError_t e = cudaSuccess;
    for (int r = 0; r < reps && e == cudaSuccess; ++r) {
        cudaMemsetAsync(ws + off_flush, r & 0xff, flush_bytes, s);
        cudaEventRecord(e0, s);
        launch();
        cudaEventRecord(e1, s);
        e = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        total += ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) return set_error(ctx, TB_ERR_CUDA, "tb_bsr_spmm_profile: %s", cudaGetErrorString(e));
    *ms_per_launch = total / reps;
    TB_CUDA_TRY(ctx, cudaGetLastError());
    return st.finish();
}
