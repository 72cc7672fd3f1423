// tb_descriptors: 32 local-environment numbers per right-hand side, the input
// of the iteration-count predictor (the paper has no learned component; the
// definition is the project's own and is listed in include/tbgf.h).
//
// One CTA per column: the hop-shell subspace's block structure and two FP64
// vectors live in shared memory; hop distances come from a level-synchronous
// breadth-first search inside the subspace; the spectral moments
// m_k = e_j^T (H_OO - H_jj)^k e_j (k = 2..9) from v_{k+1} = (H_OO - H_jj) v_k
// with m_{2k} = v_k.v_k and m_{2k+1} = v_k.v_{k+1}.  Bound by the FP64 pipe and the
// barriers of the sums.
#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

constexpr int DNT = 256;
constexpr int NDESC = 32;

__device__ __forceinline__ int find_atom(const int32_t *atoms, int n, int64_t g) {
    int lo = 0, hi = n - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int64_t v = atoms[mid];
        if (v == g) return mid;
        if (v < g) lo = mid + 1; else hi = mid - 1;
    }
    return -1;
}

// CTA sums of K doubles, in v of every thread; two barriers for all K (a sum of its
// own for each of the 24 numbers cost 29 us a column)
template <int K>
__device__ __forceinline__ void cta_sums(double (&v)[K], double (*scratch)[DNT / 32 + 1]) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        v[k] = warp_sum(v[k]);
        if ((threadIdx.x & 31) == 0) scratch[k][threadIdx.x >> 5] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int w = 0; w < DNT / 32; ++w) s += scratch[threadIdx.x][w];
        scratch[threadIdx.x][DNT / 32] = s;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = scratch[k][DNT / 32];
}

// sum_j row[j] x[j] added to y in order
template <int B>
__device__ __forceinline__ double dot_row(const double *__restrict__ row, const double *x, double y) {
    if constexpr (B % 2 == 0) { // rows of such blocks are 16-byte aligned
#pragma unroll
        for (int q = 0; q < B; q += 2) {
            const double2 h = __ldg(reinterpret_cast<const double2 *>(row + q));
            y = fma(h.x, x[q], y);
            y = fma(h.y, x[q + 1], y);
        }
    } else {
#pragma unroll
        for (int q = 0; q < B; ++q) y = fma(__ldg(row + q), x[q], y);
    }
    return y;
}

// Shared memory of the two vectors, or of the sums in their place where those are larger.
constexpr int EARLY = 5 * (DNT / 32 + 1) + 2 * (DNT / 32); // doubles
__host__ __device__ constexpr size_t vector_bytes(int64_t maxr) { return 8 * (2 * maxr > EARLY ? 2 * maxr : EARLY); }

template <int B>
__global__ void __launch_bounds__(DNT) k_desc(const int64_t *__restrict__ h_rp, const int32_t *__restrict__ h_ci,
                                              const double *__restrict__ h_val, const double *__restrict__ s_val,
                                              const int64_t *__restrict__ rhs, const int32_t *__restrict__ radii,
                                              const int64_t *__restrict__ sub_ptr,
                                              const int32_t *__restrict__ sub_atoms, int64_t n, int maxa, int dmax,
                                              float *__restrict__ out) {
    // (no more static shared memory than the kernel ever had, or the largest subspaces would no longer fit: the sums
    // before the vectors are in use lie in their place)
    extern __shared__ __align__(16) unsigned char smem[];
    const int maxr = maxa * B;
    double *v0 = reinterpret_cast<double *>(smem);
    double *v1 = v0 + maxr;
    int32_t *atoms = reinterpret_cast<int32_t *>(smem + vector_bytes(maxr));
    int32_t *nbk = atoms + maxa;
    int16_t *nbl = reinterpret_cast<int16_t *>(nbk + maxa * dmax);
    int16_t *cnt = nbl + maxa * dmax;
    int16_t *dist = cnt + maxa;
    typedef double Scratch[DNT / 32 + 1];
    __shared__ Scratch scratch[2];
    __shared__ int s_shell[6], s_max, s_surf;
    Scratch *early = reinterpret_cast<Scratch *>(smem);        // [5], then the warps' minima and maxima
    double *s_mn = reinterpret_cast<double *>(early + 5), *s_mx = s_mn + DNT / 32;
    const int tid = threadIdx.x;
    for (int64_t c = blockIdx.x; c < n; c += gridDim.x) {
        const int64_t a0 = sub_ptr[c];
        const int nat = (int)(sub_ptr[c + 1] - a0);
        const int64_t j = rhs[c];
        const int R = radii[c];
        for (int l = tid; l < nat; l += DNT) atoms[l] = sub_atoms[a0 + l];
        __syncthreads();
        for (int l = tid; l < nat; l += DNT) {
            const int64_t g = atoms[l];
            int k2 = 0;
            for (int64_t k = h_rp[g]; k < h_rp[g + 1] && k2 < dmax; ++k) {
                const int lc = find_atom(atoms, nat, h_ci[k]);
                if (lc >= 0) {
                    nbl[l * dmax + k2] = (int16_t)lc;
                    nbk[l * dmax + k2] = (int32_t)k;
                    ++k2;
                }
            }
            cnt[l] = (int16_t)k2;
            dist[l] = -1;
        }
        __syncthreads();
        const int la = find_atom(atoms, nat, j / B);
        const int jl = la * B + (int)(j % B);
        if (tid == 0) dist[la] = 0;
        __syncthreads();
        for (int d = 0; d < R; ++d) {
            for (int l = tid; l < nat; l += DNT) {
                if (dist[l] != d) continue;
                for (int s = 0; s < cnt[l]; ++s) {
                    const int lc = nbl[l * dmax + s];
                    if (dist[lc] < 0) dist[lc] = (int16_t)(d + 1); // every writer stores the same value
                }
            }
            __syncthreads();
        }
        const int nrows = nat * B;
        // --- shell counts, largest hop distance
        if (tid < 6) s_shell[tid] = 0;
        if (tid == 6) s_max = 0, s_surf = 0;
        __syncthreads();
        for (int l = tid; l < nat; l += DNT) {
            const int dd = dist[l];
            if (dd >= 1 && dd <= 5) atomicAdd(&s_shell[dd], 1);
            if (dd > 0) atomicMax(&s_max, dd);
        }
        // --- diagonal statistics and row-j sums (dsum, dsq, hjj, hrow, srow)
        double st[5] = {0, 0, 0, 0, 0}, dmin = 1e300, dmaxv = -1e300;
        for (int l = tid; l < nrows; l += DNT) {
            const int lat = l / B, i = l % B;
            for (int s = 0; s < cnt[lat]; ++s) {
                if (nbl[lat * dmax + s] != lat) continue;
                const double h = h_val[(int64_t)nbk[lat * dmax + s] * B * B + i * B + i];
                st[0] += h;
                st[1] += h * h;
                dmin = fmin(dmin, h);
                dmaxv = fmax(dmaxv, h);
            }
        }
        const int jo = jl % B;
        for (int e = tid; e < cnt[la] * B; e += DNT) { // row j, an entry a thread
            const int s = e / B, q = e - s * B, lc = nbl[la * dmax + s];
            const int64_t at = (int64_t)nbk[la * dmax + s] * B * B + jo * B + q;
            const double h = h_val[at];
            if (lc == la && q == jo) {
                st[2] += h;
                continue;
            }
            st[3] += h * h;
            if (s_val) {
                const double sv = s_val[at];
                st[4] += sv * sv;
            }
        }
        // min / max through warp reductions of the negated / plain values
        double mn = dmin, mx = dmaxv;
        for (int o = 16; o > 0; o >>= 1) {
            mn = fmin(mn, __shfl_xor_sync(TB_FULL_MASK, mn, o));
            mx = fmax(mx, __shfl_xor_sync(TB_FULL_MASK, mx, o));
        }
        if ((tid & 31) == 0) s_mn[tid >> 5] = mn, s_mx[tid >> 5] = mx;
        cta_sums(st, early);
        if (tid == 0)
            for (int w = 1; w < DNT / 32; ++w) mn = fmin(mn, s_mn[w]), mx = fmax(mx, s_mx[w]);
        const double dmean = st[0] / nrows, dvar = st[1] / nrows - dmean * dmean, hjj = st[2], hrow = st[3], srow = st[4];
        const int dmax_reached = s_max;
        for (int l = tid; l < nat; l += DNT)
            if (dist[l] == dmax_reached) atomicAdd(&s_surf, 1);
        // --- mean Frobenius norm of the in-subspace neighbour blocks of atom a
        double fs[2] = {0, 0};
        for (int s = tid; s < cnt[la]; s += DNT) {
            const int lc = nbl[la * dmax + s];
            if (lc == la) continue;
            const int64_t kb = nbk[la * dmax + s];
            double f = 0.0;
            for (int q = 0; q < B * B; ++q) f += h_val[kb * B * B + q] * h_val[kb * B * B + q];
            fs[0] += sqrt(f);
            fs[1] += 1.0;
        }
        // --- spectral moments; v_k is zero beyond k hops, so step k takes the rows up to
        // k + 1 hops away and the neighbours up to k (under half of the FP64 products)
        cta_sums(fs, scratch);
        for (int l = tid; l < nrows; l += DNT) v0[l] = (l == jl) ? 1.0 : 0.0; // (behind the sums in its place)
        __syncthreads();
        const double fsum = fs[0], fcnt = fs[1];
        double mom[10];
        double *cur = v0, *nxt = v1;
        for (int k = 0; k < 5; ++k) {
            double d[2] = {0, 0};
            const int reach = k < 4 ? k + 1 : k; // the last vector is only needed where v_4 is not zero
            for (int l = tid; l < nrows; l += DNT) {
                const int lat = l / B, i = l - lat * B;
                double y = 0.0;
                if (dist[lat] <= reach) {
                    const double x = cur[l];
                    y = -hjj * x;
                    for (int s = 0; s < cnt[lat]; ++s) {
                        const int lc = nbl[lat * dmax + s];
                        if (dist[lc] > k) continue;
                        y = dot_row<B>(h_val + (int64_t)nbk[lat * dmax + s] * B * B + i * B, cur + lc * B, y);
                    }
                    d[0] += x * x;
                    d[1] += x * y;
                }
                nxt[l] = y;
            }
            // v_k . v_k = m_{2k},  v_k . v_{k+1} = m_{2k+1}
            cta_sums(d, scratch);
            mom[2 * k] = d[0];
            mom[2 * k + 1] = d[1];
            double *t = cur;
            cur = nxt;
            nxt = t;
        }
        if (tid == 0) {
            float *o = out + c * NDESC;
            for (int q = 0; q < NDESC; ++q) o[q] = 0.f;
            o[0] = (float)(R / 5.0);
            o[1] = (float)(log((double)nat) / log(1000.0));
            for (int s = 1; s <= 5; ++s) o[1 + s] = (float)(s_shell[s] / 100.0);
            o[7] = (float)((double)(h_rp[j / B + 1] - h_rp[j / B] - 1) / 12.0);
            o[8] = (float)hjj;
            for (int k = 2; k <= 9; ++k) {
                const double m = mom[k];
                o[9 + k - 2] = (float)((m < 0 ? -1.0 : 1.0) * pow(fabs(m), 1.0 / k));
            }
            o[17] = (float)srow;
            o[18] = (float)dmean;
            o[19] = (float)sqrt(fmax(dvar, 0.0));
            o[20] = (float)mn;
            o[21] = (float)mx;
            o[22] = (float)hrow;
            o[23] = (float)(fcnt > 0 ? fsum / fcnt : 0.0);
            o[24] = (float)(nrows / 1000.0);
            o[25] = (float)((double)s_surf / nat);
        }
        __syncthreads();
    }
}

} // namespace

extern "C" int tb_descriptors(tb_ctx *ctx, const tb_bsr *H, const tb_bsr *S, const int64_t *rhs_rows,
                              const int32_t *radii, int64_t n_rhs, const int64_t *sub_ptr, const int32_t *sub_atoms,
                              float *out, void *stream) {
    using namespace tbgf;
    if (!ctx) return TB_ERR_ARG;
    TB_CHECK(ctx, H && H->row_ptr && H->col_idx && H->val && n_rhs >= 0, TB_ERR_ARG, "tb_descriptors: bad arguments");
    TB_CHECK(ctx, H->bdim == 1 || H->bdim == 4 || H->bdim == 9, TB_ERR_UNSUPPORTED, "bdim %d", H->bdim);
    TB_CHECK(ctx, !S || (S->nnzb == H->nnzb && S->bdim == H->bdim), TB_ERR_ARG, "S must have H's block pattern");
    if (n_rhs == 0) return TB_OK;
    TB_CHECK(ctx, rhs_rows && radii && sub_ptr && sub_atoms && out, TB_ERR_ARG, "tb_descriptors: arrays missing");
    cudaStream_t s = (cudaStream_t)stream;
    const int b = H->bdim;
    std::vector<int64_t> h_sptr(n_rhs + 1), h_rp(H->n_brows + 1), h_rhs(n_rhs);
    std::vector<int32_t> h_rad(n_rhs);
    auto fetch = [&](void *dst, const void *src, size_t bytes) -> int {
        if (is_device_ptr(src)) {
            TB_CUDA_TRY(ctx, cudaMemcpy(dst, src, bytes, cudaMemcpyDeviceToHost));
        } else {
            std::memcpy(dst, src, bytes);
        }
        return TB_OK;
    };
    int rc = fetch(h_sptr.data(), sub_ptr, 8 * (n_rhs + 1));
    if (!rc) rc = fetch(h_rp.data(), H->row_ptr, 8 * (H->n_brows + 1));
    if (!rc) rc = fetch(h_rhs.data(), rhs_rows, 8 * n_rhs);
    if (!rc) rc = fetch(h_rad.data(), radii, 4 * n_rhs);
    if (rc) return rc;
    int maxa = 1, dmax = 1;
    for (int64_t a = 0; a < H->n_brows; ++a) dmax = std::max<int64_t>(dmax, h_rp[a + 1] - h_rp[a]);
    for (int64_t c = 0; c < n_rhs; ++c) {
        const int64_t na = h_sptr[c + 1] - h_sptr[c];
        TB_CHECK(ctx, na >= 1 && na <= 32767 && h_rad[c] >= 0 && h_rad[c] <= 64 && h_rhs[c] >= 0 &&
                          h_rhs[c] < H->n_brows * b,
                 TB_ERR_ARG, "tb_descriptors: column %lld out of range", (long long)c);
        maxa = std::max<int64_t>(maxa, na);
    }
    const int64_t n_sub = h_sptr[n_rhs];
    Stager st(ctx, WS_STAGE_IN, s);
    void *drp, *dci, *dval, *dsval = nullptr, *drhs, *drad, *dsptr, *datoms, *dout;
    const int64_t bb = (int64_t)b * b;
    st.add(H->row_ptr, 8 * (H->n_brows + 1), true, false, &drp);
    st.add(H->col_idx, 4 * H->nnzb, true, false, &dci);
    st.add(H->val, 8 * H->nnzb * bb, true, false, &dval);
    if (S) st.add(S->val, 8 * S->nnzb * bb, true, false, &dsval);
    st.add(rhs_rows, 8 * n_rhs, true, false, &drhs);
    st.add(radii, 4 * n_rhs, true, false, &drad);
    st.add(sub_ptr, 8 * (n_rhs + 1), true, false, &dsptr);
    st.add(sub_atoms, 4 * n_sub, true, false, &datoms);
    st.add(out, 4 * 32 * n_rhs, false, true, &dout);
    rc = st.commit();
    if (rc) return rc;
    rc = validate_bsr(ctx, (const int64_t *)drp, (const int32_t *)dci, dval, H->n_brows, H->nnzb, s, "H");
    if (rc) return rc;
    const size_t sm = vector_bytes((int64_t)maxa * b) + (size_t)maxa * 4 + (size_t)maxa * dmax * 6 + (size_t)maxa * 4 + 64;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const void *fn = b == 1 ? (const void *)k_desc<1> : b == 4 ? (const void *)k_desc<4> : (const void *)k_desc<9>;
    cudaFuncAttributes at;
    TB_CUDA_TRY(ctx, cudaFuncGetAttributes(&at, fn));
    TB_CHECK(ctx, sm + at.sharedSizeBytes <= (size_t)optin, TB_ERR_SIZE, "descriptor subspace needs %zu bytes of shared memory",
             sm + at.sharedSizeBytes);
    TB_CUDA_TRY(ctx, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    const int grid = (int)std::min<int64_t>(n_rhs, 152 * 4);
#define TB_DESC_ARGS                                                                                          \
    (const int64_t *)drp, (const int32_t *)dci, (const double *)dval, (const double *)dsval, (const int64_t *)drhs, \
        (const int32_t *)drad, (const int64_t *)dsptr, (const int32_t *)datoms, n_rhs, maxa, dmax, (float *)dout
    if (b == 1)
        k_desc<1><<<grid, DNT, sm, s>>>(TB_DESC_ARGS);
    else if (b == 4)
        k_desc<4><<<grid, DNT, sm, s>>>(TB_DESC_ARGS);
    else
        k_desc<9><<<grid, DNT, sm, s>>>(TB_DESC_ARGS);
#undef TB_DESC_ARGS
    TB_CUDA_TRY(ctx, cudaGetLastError());
    return st.finish();
}
