// shifted_cocg_solve_local for FP64 and df vectors: one CTA per column, persistent
// over a device work queue, as k_local (local_impl.cuh, which FP32 vectors and
// overlaps without usable spectral bounds run), with
//  - u = (z_s S - H) p kept by recurrence, so an iteration has one product with H on
//    a finished vector and no S p;
//  - the inner solve on S_OO as in the panel solver (engine.cuh): FP32 Chebyshev
//    sweeps, each followed by a product that gives the true residual.  The bounds of
//    S hold for every principal submatrix (interlacing).  Conjugate gradients in df
//    took nine df products and eighteen CTA sums an iteration; a df product costs 12
//    FP32 operations a term, an FP32 one a single FMA;
//  - the shifted recurrences (FP64, over two microseconds of dependent divides) on the
//    last warps, beside the rows of the others;
//  - CTA sums whose first warp adds up the warps' parts and runs the scalar step, two
//    barriers a sum instead of four;
//  - 9x9 blocks transposed (the rows of a block are neighbouring lanes, so a value
//    load touches 4-7 lines instead of 18) and rows of 4x4 blocks in 16-byte loads.
// Seeds that converge long before another shift are kept in range (range_step): on the
// substitution system (median shift between two bands, 130 draws) 64 calls had columns
// that broke down without it, 35 with the kernel before; and the columns need no restart
// with another seed (C5's shifts, tol 1e-5, 255 columns: 1160 iterations on average, FP64
// 1157; with the restarts that made up for lost range before, 1565).
// Measured (df): fcc b = 4 with overlap, 608 columns of up to 225 atoms, 643 -> 192 ms; b =
// 9, 152 columns of up to 561 atoms, 445 -> 207 ms, bound by the longest column.  What
// bounds it: the latency of the block values from L2 (long-scoreboard stalls; b = 9 df
// values exceed L2), then barriers and the scalar steps between the short products.
// Vectors that rows gather (r; with S the sweep vectors) are in shared memory, those
// that only their own row reads (rt, p, u, t) too when they fit, else in a global
// slice per CTA; as a last resort all are global.
#pragma once

#include "engine.cuh"
#include "local_impl.cuh"

namespace tbgf {

template <typename T>
struct LocalArgs2 {
    LocalArgs<T> a;       // a.h_val, a.s_val: blocks transposed as local_transposed() says
    const float *s_val32;
    int32_t terms;
    float inv_theta, om[MAX_TERMS], ga[MAX_TERMS];
    int32_t s_unit;
    int32_t own_global;   // 1: own-row vectors in a.gvec; 2: gathered ones too
    int32_t *fail;
};

// 9x9 blocks in df and FP32 are stored transposed (FP64 uses the caller's values)
template <typename T, int B>
constexpr bool local_transposed() { return B == 9 && !std::is_same<T, double>::value; }

// bytes of the gathered vectors (r; with S T32, X0, X1) and of the own-row ones ((rt, t,)
// p, u) over maxr rows, each vector on a 16-byte boundary
constexpr size_t local2_vec(size_t bytes, int64_t maxr) { return (bytes * maxr + 15) / 16 * 16; }
constexpr size_t local2_gather(bool has_s, size_t csz, int64_t maxr) {
    return local2_vec(csz, maxr) + (has_s ? 3 * local2_vec(8, maxr) : 0);
}
constexpr size_t local2_own(bool has_s, size_t csz, int64_t maxr) { return (has_s ? 4 : 2) * local2_vec(csz, maxr); }

template <typename T, int B>
__device__ __forceinline__ void ld_local_row(const T *__restrict__ blk, int i, T (&a)[B]) {
    if constexpr (local_transposed<T, B>()) {
#pragma unroll
        for (int j = 0; j < B; ++j) a[j] = ldg_val(blk + j * B + i);
    } else {
        T r[B];
        ld_block_rows<T, B, 1>(blk, i, r);
#pragma unroll
        for (int j = 0; j < B; ++j) a[j] = r[j];
    }
}

// y = sum over the in-subspace blocks of row l's block row of A(l, .) x
template <typename T, int B, typename X>
__device__ __forceinline__ cpx<T> local_product(int l, const T *__restrict__ val, const int32_t *nbk, const int16_t *nbl,
                                                const int16_t *cnt, int dmax, const X *x) {
    const int la = l / B, i = l - la * B, nc = cnt[la];
    const int32_t *kb = nbk + la * dmax;
    const int16_t *lb = nbl + la * dmax;
    PSum<T> sr, si;
    sr.zero(), si.zero();
    constexpr int UNR = B == 9 ? (sizeof(T) == 4 ? 2 : 1) : 4;
#pragma unroll UNR
    for (int q = 0; q < nc; ++q) {
        T v[B];
        ld_local_row<T, B>(val + (int64_t)kb[q] * (B * B), i, v);
        const int xb = lb[q] * B;
        if constexpr (std::is_same<X, float>::value && B == 4) { // two FP32 complex values a load
#pragma unroll
            for (int j = 0; j < B; j += 2) {
                const float4 xv = *reinterpret_cast<const float4 *>(x + 2 * (xb + j));
                sr.prod(v[j], xv.x);
                si.prod(v[j], xv.y);
                sr.prod(v[j + 1], xv.z);
                si.prod(v[j + 1], xv.w);
            }
        } else {
#pragma unroll
            for (int j = 0; j < B; ++j) {
                const cpx<X> xv = ld1(x, xb + j);
                sr.prod(v[j], xv.re);
                si.prod(v[j], xv.im);
            }
        }
    }
    return mk(sr.get(), si.get());
}

// The column times 2^k (see range_step): its vectors and the pi of its shifts.  A call,
// so that it takes no registers of the iteration.
template <typename T, bool HAS_S>
__device__ __noinline__ void scale_column(int k, T *R, T *RT, T *P, T *U, int nrows, ShiftL *shs, int nz) {
    for (int l = threadIdx.x; l < nrows; l += blockDim.x) {
        st1(R, l, mul_pow2(k, ld1(R, l)));
        if constexpr (HAS_S) st1(RT, l, mul_pow2(k, ld1(RT, l)));
        st1(P, l, mul_pow2(k, ld1(P, l)));
        st1(U, l, mul_pow2(k, ld1(U, l)));
    }
    for (int m = threadIdx.x; m < nz; m += blockDim.x) {
        shs[m].pi = mul_pow2(k, shs[m].pi);
        shs[m].pi_next = mul_pow2(k, shs[m].pi_next);
    }
}

template <typename T, int B, bool HAS_S>
__global__ void __launch_bounds__(1024) k_local2(const __grid_constant__ LocalArgs2<T> g) {
    const LocalArgs<T> &a = g.a; // (64 registers: 1024 threads of an SM, in one CTA or several)
    extern __shared__ __align__(16) unsigned char smem[];
    const int NTH = blockDim.x, tid = threadIdx.x, nwarp = NTH / 32, warp = tid / 32, lane = tid & 31;
    const int64_t maxr = (int64_t)a.maxa * B;
    // shared: [gathered vectors][own-row vectors][shift states][structure], as far as they fit
    unsigned char *sp = smem, *gp = nullptr;
    if (g.own_global) {
        const size_t per = (g.own_global == 2 ? local2_gather(HAS_S, sizeof(cpx<T>), maxr) : 0) + local2_own(HAS_S, sizeof(cpx<T>), maxr);
        gp = reinterpret_cast<unsigned char *>(a.gvec) + (int64_t)blockIdx.x * per;
    }
    auto take = [&](bool global, size_t bytes) {
        unsigned char *&q = global ? gp : sp;
        unsigned char *r = q;
        q += local2_vec(bytes, maxr);
        return r;
    };
    T *R = reinterpret_cast<T *>(take(g.own_global == 2, sizeof(cpx<T>)));
    float *T32 = nullptr, *X0 = nullptr, *X1 = nullptr;
    if constexpr (HAS_S) {
        T32 = reinterpret_cast<float *>(take(g.own_global == 2, 8));
        X0 = reinterpret_cast<float *>(take(g.own_global == 2, 8));
        X1 = reinterpret_cast<float *>(take(g.own_global == 2, 8));
    }
    T *P = reinterpret_cast<T *>(take(g.own_global != 0, sizeof(cpx<T>)));
    T *U = reinterpret_cast<T *>(take(g.own_global != 0, sizeof(cpx<T>)));
    T *RT = R, *Tv = nullptr;
    if constexpr (HAS_S) {
        RT = reinterpret_cast<T *>(take(g.own_global != 0, sizeof(cpx<T>)));
        Tv = reinterpret_cast<T *>(take(g.own_global != 0, sizeof(cpx<T>)));
    }
    ShiftL *shs = reinterpret_cast<ShiftL *>(sp);
    int32_t *atoms = reinterpret_cast<int32_t *>(shs + a.nz);
    int32_t *nbk = atoms + a.maxa;
    int32_t *kept = nbk + a.maxa * a.dmax;
    int16_t *nbl = reinterpret_cast<int16_t *>(kept + a.max_kept);
    int16_t *cnt = nbl + a.maxa * a.dmax;

    typedef typename Acc<T>::P PP;
    __shared__ PP wpart[3][32];
    __shared__ int s_col, s_jloc, s_nkept, s_nact, s_status, s_stop, s_again;
    __shared__ c64 s_alpha, s_boa, s_beta_prev, s_zs; // s_boa: beta_{n-1} / alpha_{n-1}
    __shared__ double s_rn2;
    __shared__ int s_step;
    __shared__ cpx<T> s_be, s_nal, s_zt; // beta, -alpha, z_s in T
    __shared__ T s_sig;
    __shared__ typename std::conditional<std::is_same<T, double>::value, double, float>::type s_inv;
    __shared__ float s_ratio;
    // scalars that only thread 0 uses
    c64 rho = mk(1.0, 0.0);
    double t2 = 1.0, sig = 1.0;

    c64 *xs = a.scratch + (int64_t)blockIdx.x * 2 * a.max_kept * a.nz;
    c64 *ps = xs + (int64_t)a.max_kept * a.nz;

    // CTA sums; `fin` runs in thread 0 with the K results, behind a barrier and before one
    auto sums = [&](auto &acc, auto fin) {
        constexpr int K = sizeof(acc) / sizeof(acc[0]);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            warp_reduce(acc[k]);
            if (lane == 0) wpart[k][warp] = acc[k].pack();
        }
        __syncthreads();
        if (warp == 0) {
            double v[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                Acc<T> s;
                s.zero();
                if (lane < nwarp) s = Acc<T>::unpack(wpart[k][lane]);
                group_reduce(s, 32);
                v[k] = s.value();
            }
            if (lane == 0) fin(v);
        }
        __syncthreads();
    };

    for (;;) {
        if (tid == 0) s_col = (int)atomicAdd(a.queue, 1ull);
        __syncthreads();
        const int64_t qi = s_col;
        if (qi >= a.n) break;
        const int64_t col = a.order ? a.order[qi] : qi;
        // ---- local structure
        const int64_t a0 = a.sub_ptr[col];
        const int nat = (int)(a.sub_ptr[col + 1] - a0);
        for (int l = tid; l < nat; l += NTH) atoms[l] = a.sub_atoms[a0 + l];
        __syncthreads();
        for (int l = tid; l < nat; l += NTH) {
            const int64_t at = atoms[l];
            int c = 0;
            for (int64_t k = a.h_rp[at]; k < a.h_rp[at + 1] && c < a.dmax; ++k) {
                const int lc = bsearch_atom(atoms, nat, a.h_ci[k]);
                if (lc >= 0) {
                    nbl[l * a.dmax + c] = (int16_t)lc;
                    nbk[l * a.dmax + c] = (int32_t)k;
                    ++c;
                }
            }
            cnt[l] = (int16_t)c;
        }
        const int64_t j = a.rhs[col];
        const int64_t k0 = a.optr[col];
        const int nkept = (int)(a.optr[col + 1] - k0);
        if (tid == 0) {
            const int la = bsearch_atom(atoms, nat, j / B);
            s_jloc = la >= 0 ? la * B + (int)(j % B) : -1;
            s_nkept = nkept;
        }
        for (int k = tid; k < nkept; k += NTH) {
            const int64_t row = a.orows[k0 + k];
            const int la = bsearch_atom(atoms, nat, row / B);
            kept[k] = la >= 0 ? la * B + (int)(row % B) : -1;
        }
        __syncthreads();
        const int nrows = nat * B, jloc = s_jloc;
        // ---- initial state
        auto reset_vectors = [&]() {
            for (int l = tid; l < nrows; l += NTH) {
                st1(RT, l, mk<T>(l == jloc ? (T)1 : (T)0, 0));
                st1(P, l, mk<T>(0, 0));
                st1(U, l, mk<T>(0, 0));
                if constexpr (HAS_S) st1(T32, l, mk(l == jloc ? 1.f : 0.f, 0.f));
            }
        };
        auto reset_scalars = [&]() { // thread 0
            rho = mk(1.0, 0.0);
            s_alpha = mk(0.0, 0.0);
            s_beta_prev = s_boa = mk(0.0, 0.0);
            s_be = mk<T>(0, 0);
            s_rn2 = 1.0;
            s_step = 0;
            t2 = sig = 1.0;
            s_sig = (T)1;
            s_inv = 1;
            s_ratio = 1.f;
        };
        reset_vectors();
        for (int q = tid; q < nkept * a.nz; q += NTH) xs[q] = ps[q] = mk(0.0, 0.0);
        for (int m = tid; m < a.nz; m += NTH) {
            ShiftL s;
            s.pi = s.pi_prev = s.pi_next = mk(1.0, 0.0);
            s.resid = 1.0;
            s.active = 1;
            s.conv_it = -1;
            shs[m] = s;
        }
        if (tid == 0) {
            reset_scalars();
            s_status = jloc < 0 ? TB_COL_BREAKDOWN : TB_COL_MAX_ITER;
            s_stop = (jloc < 0);
            s_zs = a.zs;
            s_zt = cvt<T>(a.zs);
            s_nact = 0;
        }
        __syncthreads();

        int64_t inner_total = 0;
        // R <- S^-1 RT: sweeps on T32 (RT scaled), refinement; thread 0's done(rho) at the end
        auto inner_solve = [&](auto done) {
            if constexpr (HAS_S) {
                int passes = 0;
                for (int mode = 0;; mode = 1) {
                    for (int k = 1; k < g.terms; ++k) {
                        const float om = g.om[k], ga = g.ga[k], it = g.inv_theta;
                        const float *xk = k == 1 ? T32 : (k & 1 ? X1 : X0);
                        float *xn = k & 1 ? X0 : X1;
                        for (int l = tid; l < nrows; l += NTH) {
                            cpx<float> sx = local_product<float, B, float>(l, g.s_val32, nbk, nbl, cnt, a.dmax, xk);
                            const cpx<float> b = ld1(T32, l);
                            cpx<float> x, xm;
                            if (k == 1) {
                                x = it * b, xm = mk(0.f, 0.f), sx = it * sx;
                            } else {
                                x = ld1(xk, l);
                                xm = k == 2 ? it * b : ld1(xn, l);
                            }
                            x.re += om * (x.re - xm.re) + ga * (b.re - sx.re);
                            x.im += om * (x.im - xm.im) + ga * (b.im - sx.im);
                            st1(xn, l, x);
                        }
                        __syncthreads();
                    }
                    inner_total += g.terms - 1;
                    const float *c32 = g.terms & 1 ? X1 : X0;
                    Acc<T> acc[3];
                    acc[0].zero(), acc[1].zero(), acc[2].zero();
                    const T sg = s_sig;
                    const auto inv = s_inv;
                    for (int l = tid; l < nrows; l += NTH) {
                        const cpx<T> sc = local_product<T, B, float>(l, a.s_val, nbk, nbl, cnt, a.dmax, c32);
                        const cpx<float> c = ld1(c32, l);
                        const cpx<T> rt = ld1(RT, l);
                        cpx<T> y, t;
                        if (mode == 0) {
                            y = mk(scaled(sg, c.re), scaled(sg, c.im));
                            t = rt;
                        } else {
                            y = ld1(R, l);
                            y = mk(scaled_add(sg, c.re, y.re), scaled_add(sg, c.im, y.im));
                            t = ld1(Tv, l);
                        }
                        t = mk(fmadd(-sg, sc.re, t.re), fmadd(-sg, sc.im, t.im));
                        st1(R, l, y);
                        st1(Tv, l, t);
                        st1(T32, l, mk(scaled32(t.re, inv), scaled32(t.im, inv)));
                        acc[0].add(t.re * t.re);
                        acc[0].add(t.im * t.im);
                        acc[1].add(y.re * rt.re);
                        acc[1].add(-(y.im * rt.im));
                        acc[2].add(y.re * rt.im);
                        acc[2].add(y.im * rt.re);
                    }
                    ++passes;
                    sums(acc, [&](double *v) {
                        const double eta2 = a.inner_tol * a.inner_tol * s_rn2;
                        if (isfinite(t2) && !(v[0] <= 1e-4 * t2) && !(v[0] <= eta2)) {
                            *g.fail = 1; // the bounds missed part of the spectrum (v[0] may not be finite): the caller takes another path
                            s_stop = 1;
                        }
                        sig = safe_scale(t2);
                        t2 = v[0];
                        const double in = 1.0 / safe_scale(t2);
                        s_sig = (T)sig;
                        s_inv = in;
                        s_again = v[0] > eta2 && isfinite(v[0]) && passes < 8 && !s_stop;
                        if (!s_again) done(mk(v[1], v[2]));
                    });
                    if (!s_again) break;
                }
            }
        };
        // r_0 = S^-1 e_j and rho_0 = r_0^T rt_0 (S != I; rho_0 = 1 when S = I)
        auto start = [&](c64 r) { // thread 0
            rho = r;
            s_inv = 1; // ||rt_0|| = 1
        };
        inner_solve(start);

        int n = 0;
        for (; !s_stop; ++n) {
            // ---- shifted step A on the last warps: rotate pi, residual test, p^m on kept rows
            int my_act = 0;
            for (int m = NTH - 1 - tid; m < a.nz; m += NTH) {
                ShiftL &s = shs[m];
                if (!s.active) continue;
                s.pi_prev = s.pi;
                s.pi = s.pi_next;
                const double pi2 = cabs2(s.pi);
                s.resid = sqrt(s_rn2 / pi2);
                if (s_rn2 <= a.tol * a.tol * pi2) {
                    s.active = 0;
                    s.conv_it = n;
                    continue;
                }
                ++my_act;
                const c64 ipi = cinv(s.pi), ratio = s.pi_prev * ipi;
                const c64 bs = (ratio * ratio) * s_beta_prev;
                for (int k = 0; k < s_nkept; ++k) {
                    const int lr = kept[k];
                    if (lr < 0) continue;
                    const c64 rv = to64(ld1(R, lr));
                    c64 &pk = ps[(int64_t)k * a.nz + m];
                    pk = ipi * rv + bs * pk;
                }
            }
            if (my_act) atomicAdd(&s_nact, my_act);
            // ---- seed step: p, u = z_s rt - H r + beta u, mu = p^T u
            Acc<T> mu[2];
            mu[0].zero(), mu[1].zero();
            const cpx<T> be = s_be, zt = s_zt;
            for (int l = tid; l < nrows; l += NTH) {
                const cpx<T> hr = local_product<T, B, T>(l, a.h_val, nbk, nbl, cnt, a.dmax, R);
                const cpx<T> rv = ld1(R, l), rt = HAS_S ? ld1(RT, l) : rv;
                const cpx<T> pv = cfma(be, ld1(P, l), rv);
                const cpx<T> u = cfma(zt, rt, cfma(be, ld1(U, l), mk(-hr.re, -hr.im)));
                st1(P, l, pv);
                st1(U, l, u);
                mu[0].add(pv.re * u.re);
                mu[0].add(-(pv.im * u.im));
                mu[1].add(pv.re * u.im);
                mu[1].add(pv.im * u.re);
            }
            sums(mu, [&](double *v) {
                const int nact = s_nact;
                s_nact = 0;
                const c64 m = mk(v[0], v[1]);
                if (nact == 0) {
                    s_stop = 1;
                    s_status = TB_COL_CONVERGED;
                } else if (n >= a.max_iter) {
                    s_stop = 1;
                    s_status = TB_COL_MAX_ITER;
                } else if (!cfinite(m) || !cfinite(rho)) {
                    s_stop = 1;
                    s_status = TB_COL_NONFINITE;
                } else if ((m.re == 0.0 && m.im == 0.0) || (rho.re == 0.0 && rho.im == 0.0)) {
                    s_stop = 1;
                    s_status = TB_COL_BREAKDOWN;
                } else {
                    const c64 al = rho * cinv(m);
                    s_alpha = al;
                    s_nal = cvt<T>(mk(-al.re, -al.im));
                    if (!cfinite(al)) {
                        s_stop = 1;
                        s_status = TB_COL_NONFINITE;
                    }
                }
            });
            if (s_stop) break;
            // ---- shifted step B on the last warps: pi_{n+1}, alpha^m, x^m += alpha^m p^m
            const c64 al64 = s_alpha;
            for (int m = NTH - 1 - tid; m < a.nz; m += NTH) {
                ShiftL &s = shs[m];
                if (!s.active) continue;
                const c64 sg = a.z[m] - s_zs;
                const c64 pn = (mk(1.0, 0.0) + al64 * sg) * s.pi + (al64 * s_boa) * (s.pi - s.pi_prev);
                const c64 as = (s.pi * cinv(pn)) * al64;
                if (!cfinite(pn) || (pn.re == 0.0 && pn.im == 0.0) || !cfinite(as)) {
                    s.active = 0;
                    s.resid = nan("");
                    continue;
                }
                s.pi_next = pn;
                for (int k = 0; k < s_nkept; ++k) {
                    c64 &xk = xs[(int64_t)k * a.nz + m];
                    xk = xk + as * ps[(int64_t)k * a.nz + m];
                }
            }
            // ---- residual update (and inner solve when S != I)
            const cpx<T> nal = s_nal;
            auto finish = [&](c64 rn) { // thread 0: beta, rotation
                const c64 be64 = rn * cinv(rho);
                s_beta_prev = be64;
                s_be = cvt<T>(be64);
                s_boa = be64 * cinv(s_alpha);
                rho = rn;
                const int k = s_step = range_step<T>(s_rn2); // the vectors and the pi: below
                if (k) {
                    s_rn2 *= pow2d(2 * k);
                    rho = pow2d(2 * k) * rho;
                }
            };
            if constexpr (HAS_S) {
                Acc<T> rr[1];
                rr[0].zero();
                const auto inv = s_inv; // 1 / ||rt_n||
                for (int l = tid; l < nrows; l += NTH) {
                    const cpx<T> rt = cfma(nal, ld1(U, l), ld1(RT, l));
                    st1(RT, l, rt);
                    st1(T32, l, mk(scaled32(rt.re, inv), scaled32(rt.im, inv)));
                    rr[0].add(rt.re * rt.re);
                    rr[0].add(rt.im * rt.im);
                }
                sums(rr, [&](double *v) {
                    sig = safe_scale(s_rn2);
                    s_rn2 = t2 = v[0];
                    s_sig = (T)sig;
                    s_inv = 1.0 / safe_scale(v[0]);
                });
                inner_solve([&](c64 r) {
                    finish(r);
                    s_inv = 1.0 / safe_scale(s_rn2); // for the next iteration's rt
                });
            } else {
                Acc<T> rr[3];
                rr[0].zero(), rr[1].zero(), rr[2].zero();
                for (int l = tid; l < nrows; l += NTH) {
                    const cpx<T> rt = cfma(nal, ld1(U, l), ld1(RT, l));
                    st1(RT, l, rt);
                    const T x2 = rt.re * rt.re, y2 = rt.im * rt.im;
                    rr[0].add(x2);
                    rr[0].add(-y2);
                    rr[1].add((T)2 * rt.re * rt.im);
                    rr[2].add(x2);
                    rr[2].add(y2);
                }
                sums(rr, [&](double *v) {
                    s_rn2 = v[2];
                    finish(mk(v[0], v[1]));
                });
            }
            if (s_step) {
                scale_column<T, HAS_S>(s_step, R, RT, P, U, nrows, shs, a.nz);
                __syncthreads();
            }
        }
        __syncthreads();
        // ---- outputs
        for (int q = tid; q < s_nkept * a.nz; q += NTH) a.G[(k0 + q / a.nz) * a.nz + q % a.nz] = xs[q];
        for (int m = tid; m < a.nz; m += NTH) a.resid[col * a.nz + m] = shs[m].resid;
        if (tid == 0) {
            a.iters[col] = n;
            a.status[col] = s_status;
            atomicAdd(&a.stat[0], (unsigned long long)n);
            atomicAdd(&a.stat[1], (unsigned long long)inner_total);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ host side
struct LocalLaunch2 {
    tb_ctx *ctx;
    LocalArgs2<double> args; // type-erased
    bool has_s;
    int threads;
    size_t smem;
    int64_t cols;
    int sms;
    cudaStream_t stream;
    int rc = TB_OK;
    int grid = 0; // out: CTAs (probe: at most)
    bool probe = false;
    int static_smem = 0;  // out of a probe: static shared memory; then the most dynamic shared memory of a launch
    int static_bytes = 0;

    template <typename T, int B>
    void go() {
        LocalArgs2<T> a;
        static_assert(sizeof(LocalArgs2<T>) == sizeof(LocalArgs2<double>), "layout");
        std::memcpy(&a, &args, sizeof(a));
        const void *fn = has_s ? (const void *)k_local2<T, B, true> : (const void *)k_local2<T, B, false>;
        cudaError_t e = cudaSuccess;
        if (probe) {
            cudaFuncAttributes at;
            e = cudaFuncGetAttributes(&at, fn);
            static_smem = (int)at.sharedSizeBytes;
            if (e != cudaSuccess) rc = set_error(ctx, TB_ERR_CUDA, "local solver attributes: %s", cudaGetErrorString(e));
            return;
        }
        // the attribute is one per kernel, not per launch: what this device allows
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_smem);
        int per = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem);
        if (e != cudaSuccess || per < 1) {
            rc = set_error(ctx, TB_ERR_CUDA, "local solver occupancy: %s", cudaGetErrorString(e));
            return;
        }
        const int g = (int)std::max<int64_t>(1, std::min<int64_t>(cols, std::min<int64_t>((int64_t)sms * per, grid)));
        if (has_s)
            k_local2<T, B, true><<<g, threads, smem, stream>>>(a);
        else
            k_local2<T, B, false><<<g, threads, smem, stream>>>(a);
        e = cudaGetLastError();
        if (e != cudaSuccess) rc = set_error(ctx, TB_ERR_CUDA, "k_local2 launch: %s", cudaGetErrorString(e));
    }
    template <typename T>
    bool run(int b) {
        switch (b) {
        case 1: go<T, 1>(); return true;
        case 4: go<T, 4>(); return true;
        case 9: go<T, 9>(); return true;
        }
        return false;
    }
};

bool launch_local2_f64(LocalLaunch2 &L, int b);
bool launch_local2_df(LocalLaunch2 &L, int b);

} // namespace tbgf
