// Spectral bounds of the overlap matrix for the Chebyshev sweeps of the panel
// solver (engine.cuh): a short Lanczos run on S from a fixed pseudo-random vector,
// one cooperative launch with two grid barriers per step.
//
// Step k: t_k = w - alpha_{k-1} v_{k-1} with its norm beta_k, then w = S v_k - beta_k
// v_{k-1} and alpha_k = v_k.w for v_k = t_k / beta_k (beta_k from ||w||^2 - alpha_k^2
// instead loses ||v|| = 1 within four steps).  FP32 vectors, FP64 sums of per-thread
// FP32 sums: the bounds need two digits.  The alpha and beta
// go to pinned host memory; the host takes the extreme eigenvalues of the tridiagonal
// matrix and widens the interval by 5 % on each side (the Ritz values lie inside
// the spectrum; what sticks out still converges, only more slowly).
#include <cmath>

#include "engine.cuh"

namespace tbgf {

namespace {

constexpr int LZ_STEPS = 12;

struct LzArgs {
    const int64_t *rp;
    const int32_t *ci;
    const double *val;
    int64_t n_brows;
    int b;
    float *u[3];          // w, and v of even and odd steps
    double *part;         // [grid]
    GridBarrier *bar;
    double *ab;           // device: [0] steps made, then alpha, beta pairs; beta_0 = ||u_0||
    double *host;
};

__device__ __forceinline__ float lz_hash(int64_t r) {
    uint32_t h = (uint32_t)r * 2654435761u ^ (uint32_t)(r >> 32);
    h ^= h >> 15;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    return (float)(h & 0xffffff) / 8388608.f - 1.f;
}

// barrier whose last arriver adds up the CTAs' partial sums and runs `last`
template <class F>
__device__ bool lz_step(const LzArgs &a, unsigned &gen, float s0, F last) {
    __shared__ double sh[NT / 32];
    __shared__ int ok;
    const double d = warp_sum((double)s0);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x / 32] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < NT / 32; ++w) t += sh[w];
        a.part[blockIdx.x] = t;
    }
    gen = (gen + 1) & 0xffffffu;
    if (group_arrival(&a.bar->arrive, gridDim.x)) {
        double t = 0;
        for (int q = threadIdx.x; q < (int)gridDim.x; q += NT) t += __ldcg(a.part + q);
        t = warp_sum(t);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x / 32] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            t = 0;
            for (int w = 0; w < NT / 32; ++w) t += sh[w];
            last(t);
            ok = 1;
            __threadfence();
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&a.bar->word), "r"(gen << 8) : "memory");
        }
    } else if (threadIdx.x == 0) {
        unsigned w, spins = 0;
        const unsigned long long t0 = global_ns();
        ok = 1;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(&a.bar->word) : "memory");
            if ((w >> 8) == gen) break;
            if ((++spins & 1023u) == 0 && (*(volatile int32_t *)&a.bar->err || global_ns() - t0 > 20000000000ull)) {
                *(volatile int32_t *)&a.bar->err = 1;
                ok = 0;
                break;
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

__device__ void timed_out(const LzArgs &a) {
    if (threadIdx.x == 0) {
        *reinterpret_cast<volatile double *>(a.host) = -1.0;
        __threadfence_system();
    }
}

__global__ void __launch_bounds__(NT, 2) k_lanczos(const __grid_constant__ LzArgs a) {
    const int64_t tid = blockIdx.x * (int64_t)NT + threadIdx.x, stride = (int64_t)gridDim.x * NT;
    const int b = a.b;
    const int64_t n = a.n_brows * b;
    unsigned gen = 0;
    float *w = a.u[0], s0 = 0.f;
    for (int64_t r = tid; r < n; r += stride) {
        const float h = lz_hash(r);
        w[r] = h;
        a.u[1][r] = a.u[2][r] = 0.f;
    }
    float alpha = 0.f, bi_prev = 0.f;
    double size = 0; // of S: |alpha_0| + beta_1
    for (int k = 0; k < LZ_STEPS; ++k) {
        // t_k = w - alpha_{k-1} v_{k-1} and its norm (t_0: the start vector)
        float *t = a.u[1 + (k & 1)], *tp = a.u[2 - (k & 1)];
        const float ab = alpha * bi_prev;
        s0 = 0.f;
        for (int64_t r = tid; r < n; r += stride) {
            const float x = w[r] - ab * tp[r];
            t[r] = x;
            s0 += x * x;
        }
        if (!lz_step(a, gen, s0, [&](double t0) { a.ab[2 + 2 * k] = t0 > 0 ? sqrt(t0) : 0; })) return timed_out(a);
        // the scalars of the last CTA: __ldcg, they change while the kernel runs
        const double beta = __ldcg(a.ab + 2 + 2 * k);
        if (k == 1) size = fabsf(alpha) + beta;
        if (!(beta > 1e-5 * size)) break; // the Krylov space is exhausted
        const float bi = (float)(1.0 / beta), bp = (float)beta * bi_prev;
        s0 = 0.f;
        for (int64_t r = tid; r < n; r += stride) {
            const int64_t br = r / b;
            const int i = (int)(r - br * b);
            float y = 0.f;
            for (int64_t q = a.rp[br]; q < a.rp[br + 1]; ++q) {
                const int64_t c = (int64_t)a.ci[q] * b;
                const double *row = a.val + (q * b + i) * b;
                for (int j = 0; j < b; ++j) y = fmaf((float)row[j], t[c + j], y);
            }
            y = y * bi - bp * tp[r];
            w[r] = y;
            s0 += t[r] * bi * y;
        }
        if (!lz_step(a, gen, s0, [&](double t0) {
                a.ab[0] = k + 1;
                a.ab[3 + 2 * k] = t0;
            }))
            return timed_out(a);
        alpha = (float)__ldcg(a.ab + 3 + 2 * k);
        bi_prev = bi;
    }
    if (tid < 3 + 2 * LZ_STEPS) {
        *reinterpret_cast<volatile double *>(a.host + tid) = __ldcg(a.ab + tid);
        __threadfence_system();
    }
}

// Number of eigenvalues of the symmetric tridiagonal (d, e) below x (Sturm sequence).
int below(const double *d, const double *e, int n, double x) {
    int c = 0;
    double q = 1;
    for (int i = 0; i < n; ++i) {
        const double off = i ? e[i - 1] * e[i - 1] : 0;
        q = d[i] - x - (q != 0 ? off / q : off / 1e-300);
        c += q < 0;
    }
    return c;
}

} // namespace

// *lo and *hi: bounds of the spectrum of S; *lo > *hi when there are none (not finite).
int spectral_bounds(tb_ctx *ctx, const int64_t *rp, const int32_t *ci, const double *val, int64_t n_brows, int b,
                    int sms, cudaStream_t s, double *lo, double *hi) {
    *lo = 1, *hi = 0;
    const int64_t n = n_brows * b;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + NT - 1) / NT, sms));
    const size_t vb = align_up(sizeof(float) * n, 256), pb = align_up(sizeof(double) * 2 * grid, 256);
    void *wsp = nullptr;
    int rc = ws_get(ctx, WS_LANCZOS, 3 * vb + pb + 4096, &wsp);
    if (rc) return rc;
    char *ws = (char *)wsp;
    int *words = nullptr, *host = nullptr;
    rc = check_words(ctx, &words, &host);
    if (rc) return rc;
    LzArgs a;
    a.rp = rp, a.ci = ci, a.val = val, a.n_brows = n_brows, a.b = b;
    for (int q = 0; q < 3; ++q) a.u[q] = (float *)(ws + q * vb);
    a.part = (double *)(ws + 3 * vb);
    a.bar = (GridBarrier *)(ws + 3 * vb + pb);
    a.ab = (double *)(ws + 3 * vb + pb + 3584);
    a.host = (double *)host + 8;
    static_assert(sizeof(GridBarrier) <= 3584, "workspace layout");
    *(volatile double *)a.host = 0.0; // nothing of an earlier call
    TB_CUDA_TRY(ctx, cudaMemsetAsync(a.bar, 0, 4096, s));
    void *args[] = {&a};
    TB_CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void *)k_lanczos, dim3(grid), dim3(NT), args, 0, s));
    int dummy = 0;
    rc = check_wait(ctx, s, &dummy);
    if (rc) return rc;
    const volatile double *h = (const volatile double *)host + 8;
    const int k = (int)h[0]; // steps made; -1: a grid barrier timed out
    TB_CHECK(ctx, k >= 0, TB_ERR_CUDA, "spectral bounds of S: a grid barrier timed out");
    if (k < 1 || k > LZ_STEPS) return TB_OK;
    double d[LZ_STEPS], e[LZ_STEPS], r = 0;
    for (int i = 0; i < k; ++i) {
        d[i] = h[3 + 2 * i];
        e[i] = i + 1 < k ? h[4 + 2 * i] : 0.0; // beta_{i+1}
        if (!std::isfinite(d[i]) || !std::isfinite(e[i])) return TB_OK;
        r = std::max(r, std::fabs(d[i]) + 2 * std::fabs(e[i]) + (i ? std::fabs(e[i - 1]) : 0));
    }
    double x0 = -2 * r, x1 = 2 * r, y0 = -2 * r, y1 = 2 * r; // smallest in (x0, x1], largest in (y0, y1]
    for (int it = 0; it < 60; ++it) {
        const double x = 0.5 * (x0 + x1), y = 0.5 * (y0 + y1);
        (below(d, e, k, x) >= 1 ? x1 : x0) = x;
        (below(d, e, k, y) >= k ? y1 : y0) = y;
    }
    const double w = 0.05 * (y1 - x0);
    *lo = x0 - w;
    *hi = y1 + w;
    return TB_OK;
}

} // namespace tbgf
