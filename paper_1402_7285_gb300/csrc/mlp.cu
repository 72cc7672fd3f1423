// Iteration-count predictor: MLP 32 -> 64 -> 64 -> 1 (tanh), FP16 weights in
// the forward pass, FP32 accumulation, FP32 master weights updated by Adam
// (Kingma & Ba, 2015), mean squared error loss.  The paper has no learned
// component: this is the project's scheduler model (predicts each column's
// iterations to tolerance so columns can be ordered / binned).
//
// Kernels: forward (+ backward deltas) per (sample, hidden unit); gradient of the
// minibatch per parameter (a fixed summation order: deterministic) with the Adam step.
// Parameter layout (floats): W1[64][32] | b1[64] | W2[64][64] | b2[64] | w3[64] | b3.
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

constexpr int DI = 32, DH = 64;
constexpr int O_W1 = 0, O_B1 = O_W1 + DH * DI, O_W2 = O_B1 + DH, O_B2 = O_W2 + DH * DH, O_W3 = O_B2 + DH,
              O_B3 = O_W3 + DH, NPARAM = O_B3 + 1;
constexpr int SPC = 4;        // samples of a CTA
constexpr int FNT = SPC * DH; // one thread per (sample, hidden unit)

// Forward (and, with DZ1 != nullptr, backward deltas) for samples [s0, s0 + n), one
// thread per (sample, hidden unit).  A minibatch of 256 samples with one thread per
// sample kept two SMs busy for 51 us a step (12,000 dependent FMAs a thread); here 64
// SMs work on it and a thread's chain is 160 FMAs.  W2 has rows of 65 in shared memory:
// units read it by rows in the forward pass and by columns in the backward pass.
constexpr int W2LD = DH + 1;
__global__ void __launch_bounds__(FNT) k_mlp_fwd(const __half *__restrict__ w16, const float *__restrict__ X,
                                                 const float *__restrict__ tgt, int64_t s0, int64_t n,
                                                 float inv_batch, float *__restrict__ pred,
                                                 float *__restrict__ H1, float *__restrict__ H2,
                                                 float *__restrict__ DZ1, float *__restrict__ DZ2,
                                                 float *__restrict__ DY, float *__restrict__ sqerr) {
    __shared__ float w1[DH * (DI + 1)], w2[DH * W2LD], wr[3 * DH + 1]; // rows padded by one; b1, b2, w3, b3
    __shared__ float x[SPC][DI], h1[SPC][DH], z2[SPC][DH], err[SPC];
    for (int i = threadIdx.x; i < NPARAM; i += FNT) {
        const float v = __half2float(w16[i]);
        if (i < O_B1) w1[(i / DI) * (DI + 1) + i % DI] = v;
        else if (i < O_W2) wr[i - O_B1] = v;
        else if (i < O_B2) w2[((i - O_W2) / DH) * W2LD + (i - O_W2) % DH] = v;
        else wr[DH + i - O_B2] = v;
    }
    const int q = threadIdx.x / DH, u = threadIdx.x % DH;
    const int64_t t0 = blockIdx.x * (int64_t)SPC, t = t0 + q, s = s0 + t;
    const bool on = t < n;
    for (int i = threadIdx.x; i < SPC * DI; i += FNT)
        x[i / DI][i % DI] = t0 + i / DI < n ? X[(s0 + t0) * DI + i] : 0.f;
    __syncthreads();
    float acc = wr[u];
#pragma unroll
    for (int k = 0; k < DI; ++k) acc = fmaf(w1[u * (DI + 1) + k], x[q][k], acc);
    const float a1 = tanhf(acc);
    h1[q][u] = a1;
    __syncthreads();
    acc = wr[DH + u];
#pragma unroll
    for (int k = 0; k < DH; ++k) acc = fmaf(w2[u * W2LD + k], h1[q][k], acc);
    const float a2 = tanhf(acc), w3 = wr[2 * DH + u];
    z2[q][u] = a2;
    __syncthreads();
    float y = wr[3 * DH]; // in order, in every thread of the sample
#pragma unroll
    for (int i = 0; i < DH; ++i) y = fmaf(wr[2 * DH + i], z2[q][i], y);
    __syncthreads();
    float err2 = 0.f;
    if (on && pred && u == 0) pred[s] = y;
    if (tgt) {
        const float e = on ? y - tgt[s] : 0.f;
        err2 = e * e;
        if (DZ1) {
            const float dy = 2.f * e * inv_batch;
            const float dz2 = dy * w3 * (1.f - a2 * a2);
            z2[q][u] = dz2;
            __syncthreads();
            acc = 0.f;
#pragma unroll
            for (int i = 0; i < DH; ++i) acc = fmaf(w2[i * W2LD + u], z2[q][i], acc);
            if (on) {
                if (u == 0) DY[t] = dy;
                DZ2[t * DH + u] = dz2;
                H2[t * DH + u] = a2;
                DZ1[t * DH + u] = acc * (1.f - a1 * a1);
                H1[t * DH + u] = a1;
            }
        }
    }
    if (sqerr) { // per-CTA part of the squared error
        if (u == 0) err[q] = err2;
        __syncthreads();
        if (threadIdx.x == 0) {
            float v = 0.f;
            for (int k = 0; k < SPC; ++k) v += err[k];
            sqerr[blockIdx.x] = v;
        }
    }
}

// The forward pass of many samples (predictions, losses), a thread a sample: one shared
// load for each FMA, the weights loaded once for 128 samples.  The kernel above loads
// them for four, and two numbers for each FMA: a prediction (with its launch of k_to_half)
// takes 14 us for 256 samples, 21 for 4096, 31 for 8192 and 2543 for 10^6 with it, and 24
// us up to a wave (19456 samples) and 504 for 10^6 with this one.  The same operations in
// the same order: the same bits.
constexpr int MNT = 128;
constexpr int64_t MANY = 5120;
__global__ void __launch_bounds__(MNT) k_mlp_many(const __half *__restrict__ w16, const float *__restrict__ X,
                                                  const float *__restrict__ tgt, int64_t n, float *__restrict__ pred,
                                                  float *__restrict__ sqerr) {
    __shared__ float w[NPARAM];
    for (int i = threadIdx.x; i < NPARAM; i += MNT) w[i] = __half2float(w16[i]);
    __syncthreads();
    const int64_t s = blockIdx.x * (int64_t)MNT + threadIdx.x;
    float err2 = 0.f;
    if (s < n) {
        float x[DI], h1[DH];
#pragma unroll
        for (int k = 0; k < DI; ++k) x[k] = X[s * DI + k];
#pragma unroll 4
        for (int i = 0; i < DH; ++i) {
            float acc = w[O_B1 + i];
#pragma unroll
            for (int k = 0; k < DI; ++k) acc = fmaf(w[O_W1 + i * DI + k], x[k], acc);
            h1[i] = tanhf(acc);
        }
        float y = w[O_B3];
#pragma unroll 4
        for (int i = 0; i < DH; ++i) {
            float acc = w[O_B2 + i];
#pragma unroll
            for (int k = 0; k < DH; ++k) acc = fmaf(w[O_W2 + i * DH + k], h1[k], acc);
            y = fmaf(w[O_W3 + i], tanhf(acc), y);
        }
        if (pred) pred[s] = y;
        if (tgt) {
            const float e = y - tgt[s];
            err2 = e * e;
        }
    }
    if (sqerr) { // per-CTA part of the squared error
        __shared__ float red[MNT];
        red[threadIdx.x] = err2;
        __syncthreads();
        for (int o = MNT / 2; o > 0; o >>= 1) {
            if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) sqerr[blockIdx.x] = red[0];
    }
}

// The forward pass alone; the parts of the squared error are mlp_parts(n).
inline int64_t mlp_parts(int64_t n) { return n > MANY ? (n + MNT - 1) / MNT : (n + SPC - 1) / SPC; }
void mlp_forward(const __half *w16, const float *X, const float *tgt, int64_t n, float *pred, float *sqerr, cudaStream_t s) {
    if (n > MANY)
        k_mlp_many<<<(int)mlp_parts(n), MNT, 0, s>>>(w16, X, tgt, n, pred, sqerr);
    else
        k_mlp_fwd<<<(int)mlp_parts(n), FNT, 0, s>>>(w16, X, tgt, 0, n, 0.f, pred, nullptr, nullptr, nullptr, nullptr,
                                                    nullptr, sqerr);
}

// Gradient of the minibatch and (w != nullptr) the Adam step.  CTA i owns hidden unit
// i of both layers (rows i of W1 and W2, b1, b2, w3; CTA 0 also b3), a thread a
// parameter; up to 1024 samples it adds them in order with 32 loads in flight, larger
// batches are split over 8 groups of threads whose parts are added in order.  (6337
// threads in 50 CTAs with one load in flight took 17 us a step of 256 samples, with
// the Adam step a launch of its own.)
constexpr int WCH = 8, WPC = 128; // groups at most, threads of a group (99 or 100 parameters)
struct AdamArgs {
    float *w, *m, *v;
    __half *w16;
    float lr, b1, b2, eps, t;
};
__device__ __forceinline__ void adam_step(const AdamArgs &A, int p, float gp) {
    const float mp = A.b1 * A.m[p] + (1.f - A.b1) * gp;
    const float vp = A.b2 * A.v[p] + (1.f - A.b2) * gp * gp;
    A.m[p] = mp;
    A.v[p] = vp;
    const float mh = mp / (1.f - powf(A.b1, A.t));
    const float vh = vp / (1.f - powf(A.b2, A.t));
    const float wp = A.w[p] - A.lr * mh / (sqrtf(vh) + A.eps);
    A.w[p] = wp;
    A.w16[p] = __float2half_rn(wp);
}
__global__ void __launch_bounds__(WCH *WPC) k_mlp_wgrad(const float *__restrict__ X, int64_t s0, int64_t n,
                                                        const float *__restrict__ H1, const float *__restrict__ H2,
                                                        const float *__restrict__ DZ1, const float *__restrict__ DZ2,
                                                        const float *__restrict__ DY, float *__restrict__ grad,
                                                        AdamArgs A) {
    __shared__ float sum[WCH][WPC];
    const int i = blockIdx.x, c = threadIdx.x % WPC, g = threadIdx.x / WPC;
    // column c of this unit's parameters: W2[i][c], W1[i][c - 64], b1, b2, w3, b3
    const float *fa = nullptr, *fb = nullptr; // factors at sample t: fa[t * la], fb[t * lb]
    int64_t la = DH, lb = DH;
    int p = -1;
    if (c < DH) p = O_W2 + i * DH + c, fa = DZ2 + i, fb = H1 + c;
    else if (c < DH + DI) p = O_W1 + i * DI + c - DH, fa = DZ1 + i, fb = X + s0 * DI + c - DH, lb = DI;
    else if (c == DH + DI) p = O_B1 + i, fa = DZ1 + i;
    else if (c == DH + DI + 1) p = O_B2 + i, fa = DZ2 + i;
    else if (c == DH + DI + 2) p = O_W3 + i, fa = DY, la = 1, fb = H2 + i;
    else if (c == DH + DI + 3 && i == 0) p = O_B3, fa = DY, la = 1;
    const int groups = blockDim.x / WPC;
    const int64_t per = (n + groups - 1) / groups, t0 = g * per, t1 = t0 + per < n ? t0 + per : n;
    float acc = 0.f;
    constexpr int U = 32; // loads in flight; the additions stay in order
    int64_t t = t0;
    if (fa) {
        for (; t + U <= t1; t += U) {
            float x[U], y[U];
#pragma unroll
            for (int q = 0; q < U; ++q) x[q] = __ldg(fa + (t + q) * la), y[q] = fb ? __ldg(fb + (t + q) * lb) : 1.f;
#pragma unroll
            for (int q = 0; q < U; ++q) acc = fmaf(x[q], y[q], acc); // (times 1: a plain sum)
        }
        for (; t < t1; ++t) acc = fmaf(fa[t * la], fb ? fb[t * lb] : 1.f, acc);
    }
    sum[g][c] = acc;
    __syncthreads();
    if (g == 0 && p >= 0) {
        float v = sum[0][c];
        for (int k = 1; k < groups; ++k) v += sum[k][c];
        if (grad) grad[p] = v;
        if (A.w) adam_step(A, p, v);
    }
}

inline int wgrad_threads(int64_t n) { return n <= 1024 ? WPC : WCH * WPC; }

__global__ void k_to_half(const float *__restrict__ w, __half *__restrict__ w16) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < NPARAM) w16[p] = __float2half_rn(w[p]);
}

struct MlpWs {
    float *w, *g, *m, *v, *H1, *H2, *DZ1, *DZ2, *DY, *sq;
    __half *w16;
};

int mlp_workspace(tb_ctx *ctx, int64_t batch, int64_t nblk_max, MlpWs &o) {
    using namespace tbgf;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t x = off;
        off = align_up(off + bytes, 256);
        return x;
    };
    const size_t ow = take(4 * NPARAM), og = take(4 * NPARAM), om = take(4 * NPARAM), ov = take(4 * NPARAM);
    const size_t o16 = take(2 * NPARAM);
    const size_t oh1 = take(4 * batch * DH), oh2 = take(4 * batch * DH), odz1 = take(4 * batch * DH),
                 odz2 = take(4 * batch * DH), ody = take(4 * batch), osq = take(4 * nblk_max);
    void *base = nullptr;
    int rc = ws_get(ctx, WS_SPMM_STAGE, off, &base);
    if (rc) return rc;
    char *b = (char *)base;
    o.w = (float *)(b + ow), o.g = (float *)(b + og), o.m = (float *)(b + om), o.v = (float *)(b + ov);
    o.w16 = (__half *)(b + o16);
    o.H1 = (float *)(b + oh1), o.H2 = (float *)(b + oh2), o.DZ1 = (float *)(b + odz1), o.DZ2 = (float *)(b + odz2);
    o.DY = (float *)(b + ody), o.sq = (float *)(b + osq);
    return TB_OK;
}

} // namespace

extern "C" {

int mlp_param_count(void) { return NPARAM; }

int mlp_grad(tb_ctx *ctx, const float *params, const float *X, const float *y, int64_t n, float *grad,
             double *loss, void *stream) {
    using namespace tbgf;
    if (!ctx) return TB_ERR_ARG;
    TB_CHECK(ctx, params && X && y && grad && n >= 1 && n <= (1 << 24), TB_ERR_ARG, "mlp_grad: bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    Stager st(ctx, WS_STAGE_IN, s);
    void *dp, *dX, *dy, *dg;
    st.add(params, 4 * NPARAM, true, false, &dp);
    st.add(X, 4 * n * DI, true, false, &dX);
    st.add(y, 4 * n, true, false, &dy);
    st.add(grad, 4 * NPARAM, false, true, &dg);
    int rc = st.commit();
    if (rc) return rc;
    const int64_t nblk = (n + SPC - 1) / SPC;
    MlpWs w;
    rc = mlp_workspace(ctx, n, nblk, w);
    if (rc) return rc;
    StageOrder order(ctx, s);
    if (order.rc) return order.rc;
    k_to_half<<<(NPARAM + 255) / 256, 256, 0, s>>>((const float *)dp, w.w16);
    k_mlp_fwd<<<(int)nblk, FNT, 0, s>>>(w.w16, (const float *)dX, (const float *)dy, 0, n, 1.f / (float)n, nullptr,
                                        w.H1, w.H2, w.DZ1, w.DZ2, w.DY, w.sq);
    k_mlp_wgrad<<<DH, wgrad_threads(n), 0, s>>>((const float *)dX, 0, n, w.H1, w.H2, w.DZ1, w.DZ2, w.DY, (float *)dg,
                                         AdamArgs{});
    TB_CUDA_TRY(ctx, cudaGetLastError());
    if (loss) {
        std::vector<float> sq(nblk);
        TB_CUDA_TRY(ctx, cudaMemcpyAsync(sq.data(), w.sq, 4 * nblk, cudaMemcpyDeviceToHost, s));
        TB_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        double acc = 0;
        for (float v : sq) acc += v;
        *loss = acc / (double)n;
    }
    return st.finish();
}

int mlp_train(tb_ctx *ctx, const float *X, const float *y, int64_t n, int32_t epochs, int32_t batch, float lr,
              float *params, double *loss_hist, void *stream) {
    using namespace tbgf;
    if (!ctx) return TB_ERR_ARG;
    TB_CHECK(ctx, X && y && params && n >= 1 && epochs >= 0 && batch >= 1 && batch <= 65536 && lr > 0.f,
             TB_ERR_ARG, "mlp_train: bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    Stager st(ctx, WS_STAGE_IN, s);
    void *dX, *dy, *dp;
    st.add(X, 4 * n * DI, true, false, &dX);
    st.add(y, 4 * n, true, false, &dy);
    st.add(params, 4 * NPARAM, true, true, &dp);
    int rc = st.commit();
    if (rc) return rc;
    const int64_t bmax = std::min<int64_t>(batch, n);
    const int64_t nblk = mlp_parts(n);
    MlpWs w;
    // rows of squared-error parts, one per epoch, read back together (64 MB of them at most)
    const int64_t rows = loss_hist ? std::max<int64_t>(1, std::min<int64_t>(epochs, (16 << 20) / nblk)) : 1;
    rc = mlp_workspace(ctx, bmax, loss_hist ? nblk * rows : 1, w);
    if (rc) return rc;
    StageOrder order(ctx, s);
    if (order.rc) return order.rc;
    TB_CUDA_TRY(ctx, cudaMemcpyAsync(w.w, dp, 4 * NPARAM, cudaMemcpyDeviceToDevice, s));
    TB_CUDA_TRY(ctx, cudaMemsetAsync(w.m, 0, 4 * NPARAM, s));
    TB_CUDA_TRY(ctx, cudaMemsetAsync(w.v, 0, 4 * NPARAM, s));
    k_to_half<<<(NPARAM + 255) / 256, 256, 0, s>>>(w.w, w.w16);
    int t = 0;
    std::vector<float> sq;
    for (int ep = 0; ep < epochs; ++ep) {
        for (int64_t s0 = 0; s0 < n; s0 += bmax) {
            const int64_t nb = std::min<int64_t>(bmax, n - s0);
            k_mlp_fwd<<<(int)((nb + SPC - 1) / SPC), FNT, 0, s>>>(w.w16, (const float *)dX, (const float *)dy, s0, nb,
                                                                 1.f / (float)nb, nullptr, w.H1, w.H2, w.DZ1, w.DZ2,
                                                                 w.DY, nullptr);
            ++t;
            const AdamArgs A{w.w, w.m, w.v, w.w16, lr, 0.9f, 0.999f, 1e-8f, (float)t};
            k_mlp_wgrad<<<DH, wgrad_threads(nb), 0, s>>>((const float *)dX, s0, nb, w.H1, w.H2, w.DZ1, w.DZ2, w.DY, nullptr, A);
        }
        if (!loss_hist) continue;
        mlp_forward(w.w16, (const float *)dX, (const float *)dy, n, nullptr, w.sq + ep % rows * nblk, s);
        if ((ep + 1) % rows && ep + 1 < epochs) continue;
        const int64_t first = ep / rows * rows, cnt = ep + 1 - first;
        sq.resize(nblk * cnt);
        TB_CUDA_TRY(ctx, cudaMemcpyAsync(sq.data(), w.sq, 4 * nblk * cnt, cudaMemcpyDeviceToHost, s));
        TB_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        for (int64_t r = 0; r < cnt; ++r) {
            double acc = 0;
            for (int64_t q = 0; q < nblk; ++q) acc += sq[r * nblk + q];
            loss_hist[first + r] = acc / (double)n;
        }
    }
    TB_CUDA_TRY(ctx, cudaMemcpyAsync(dp, w.w, 4 * NPARAM, cudaMemcpyDeviceToDevice, s));
    TB_CUDA_TRY(ctx, cudaGetLastError());
    return st.finish();
}

int mlp_predict(tb_ctx *ctx, const float *params, const float *X, int64_t n, float *pred, void *stream) {
    using namespace tbgf;
    if (!ctx) return TB_ERR_ARG;
    TB_CHECK(ctx, params && X && pred && n >= 1, TB_ERR_ARG, "mlp_predict: bad arguments");
    cudaStream_t s = (cudaStream_t)stream;
    Stager st(ctx, WS_STAGE_IN, s);
    void *dp, *dX, *dpred;
    st.add(params, 4 * NPARAM, true, false, &dp);
    st.add(X, 4 * n * DI, true, false, &dX);
    st.add(pred, 4 * n, false, true, &dpred);
    int rc = st.commit();
    if (rc) return rc;
    MlpWs w;
    rc = mlp_workspace(ctx, 1, 1, w);
    if (rc) return rc;
    StageOrder order(ctx, s);
    if (order.rc) return order.rc;
    k_to_half<<<(NPARAM + 255) / 256, 256, 0, s>>>((const float *)dp, w.w16);
    mlp_forward(w.w16, (const float *)dX, nullptr, n, (float *)dpred, nullptr, s);
    TB_CUDA_TRY(ctx, cudaGetLastError());
    return st.finish();
}

} // extern "C"
