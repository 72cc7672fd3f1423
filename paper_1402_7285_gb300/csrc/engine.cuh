// The panel solver as one persistent kernel (FP64 and df panels).
//
// A solve is one cooperative launch: its CTAs stay resident and walk through the
// phases of every outer iteration, with a grid barrier between two phases whose
// last arriver runs the scalar recurrences of that phase (the same code the
// graph's kernels run).  What that is for:
//  - small and middle-sized systems spend their time in launches: a phase of a few
//    thousand rows computes for 1-3 us, a graph node with its last-CTA tail took
//    10-50 us (FP64 divide 436 cycles, dependent FMA 76 on GB300);
//  - a thread owns one row (FP64, and df systems that do not fill the chip) of one
//    slot, so every SM has work (the graph's FP64 kernels put a 3600-row system on 25
//    SMs), and there are no more slots than columns;
//  - the inner solve on S needs no reductions: S is well conditioned (unit diagonal,
//    weak overlaps), so an FP32 sweep is a fixed Chebyshev polynomial on spectral
//    bounds from a short Lanczos run, one product and four FP32 vectors a step,
//    where conjugate gradients take two kernels and ten; each sweep is followed by a
//    product in the panel's precision that gives the true residual, and the loop ends
//    when that is below inner_tol (iterative refinement, as in the graph's df path).
// Per outer iteration:
//   A   p = r + beta p, u = z_s rt - H r + beta u, mu = p^T u  [alpha, retire, refill]
//   B   rt -= alpha u, ||rt||^2 (S = I: rho, beta: next A), FP32 copy of rt
//   X   (terms - 1) Chebyshev steps on S c = t               (barrier only)
//   R   y (+)= sigma c, t = rt - S y, ||t||^2, rho = y^T rt  [again or beta: next A]
// What bounds the phases (131072 rows x 64 slots, df, 3 CTAs per SM; HBM floors at the
// measured 6680 GB/s): A 386 us against 125 (the 12 FP32 operations of a df term: issue
// 62-69 %, the rest register-read stalls; the product alone takes 236); B 89 against 70;
// X 83 against 42 (each row of x comes from L2 once per referencing block, 8 TB/s); R
// 320 (df products again); R in FP32 163 against 93.  The graph took 390 (A with two
// more recurrences), 333, 12 x (87 + 70), 247 + 168 and 74 for rho: 1333 ms a solve of
// 64 columns at eta 0.5, 685 here.  Small systems are bound by the barriers and their
// scalar step, 3-8 us a phase: 256 rows x 2 slots FP64 634 -> 120 us an iteration,
// Anderson 4096 x 32 FP64 81 -> 37.  Keeping columns in range (range_step) takes 0.5 us of A
// and of B there: integer operations on each value of rt and a test per slot.
// A sweep that does not reduce the residual (bounds that miss part of the spectrum)
// ends the kernel with fail = 1; the caller then runs the conjugate-gradient path.
#pragma once

#include "cocg_impl.cuh"

namespace tbgf {

constexpr int MAX_TERMS = 40;
// A df refinement pass takes S c and the residual in FP32 when every residual is below
// this many inner tolerances.  The FP32 residual t - S c errs by up to 1.2e-7 sqrt(hi / lo)
// of the t before the sweep (c is larger along the lowest eigenvectors, where S c cancels;
// emulated on s-p and s+p+d overlaps: 0.4 to 1.5e-7 at hi / lo = 1.6, 0.6 to 5.6e-7 at 24):
// below inner_tol ||rt|| / 20.
inline double engine_light(double lo, double hi) { return 0.05 / (1.2e-7 * std::sqrt(hi / lo)); }
enum EngineFlag : unsigned { F_CONT = 1, F_AGAIN = 2, F_LIGHT = 4, F_LIST = 8, F_DONE = 16, F_ABORT = 32 };
enum EnginePhase { PH_A = 0, PH_B = 1, PH_X = 2, PH_R = 5, PH_R32 = 6, PH_INIT = 7 };

// The word that waiting CTAs poll and the arrival counters lie on lines of their own:
// polls of a shared line hold up the arrivals.
struct GridBarrier {
    alignas(128) unsigned int word;   // (barriers passed << 8) | flags of the last one
    alignas(128) unsigned int arrive; // arrivals of the grid (of its groups)
    alignas(128) unsigned int grp[64][8]; // arrivals within each group, 32 bytes apart
    alignas(128) int32_t err;         // a wait ran out
    int32_t fail;                     // a Chebyshev sweep did not converge
    unsigned long long t_last, ns[8], cnt[8]; // phase times (profiling)
};

// What the rows of a slot need in a phase, in the panel's type: written once by the
// last arriver of the phase before.  (Each thread converting and dividing in FP64
// for itself took 2-6 us a phase: those run at 1.7 lanes per clock.)
template <typename T>
struct SlotScalars {
    cpx<T> beta, zs, alpha;
    T sig;           // scale of the sweep's correction
    typename std::conditional<std::is_same<T, double>::value, double, float>::type
        inv;         // 1 / (scale of the next sweep's residual); FP64 residuals leave FP32's range
    int32_t step;    // B: rt is multiplied by 2^step (alpha and the next beta hold it where they need it)
    float ratio;     // sig * inv
    int32_t restart; // B: rt becomes e_row
    int64_t row;
};

template <typename T>
struct Engine {
    Panel<T> p;
    SlotScalars<T> *sc; // [MAX_W]
    c64 *kr;            // [W][max_col_ent]: r_n on the kept rows
    GridBarrier *bar;
    int32_t W;        // slots = row stride of the panel
    int32_t terms;    // Chebyshev terms of the first sweep of a solve (2..MAX_TERMS)
    int32_t terms2;   // of the others
    int32_t profile;
    int32_t group;    // CTAs of a group of the two-step sums (at most 64 groups)
    float light;      // a pass in FP32 below this many inner tolerances (engine_light; 0: never)
    float inv_theta;
    float om[MAX_TERMS], ga[MAX_TERMS]; // x_{k+1} = x_k + om (x_k - x_{k-1}) + ga (b - S x_k)
    float *X[2];
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// True in every thread of the CTA that arrives last of n.  One thread fences for its
// CTA (the barrier before makes its fence cover the others' writes), and once more
// behind the arrival, so that the last CTA reads what the others wrote.
__device__ __forceinline__ bool group_arrival(unsigned int *counter, int n) {
    __shared__ int is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const bool last = atomicAdd(counter, 1u) == (unsigned)n - 1;
        if (last) *counter = 0u;
        __threadfence();
        is_last = last;
    }
    __syncthreads();
    return is_last != 0;
}

// ------------------------------------------------------------- panel access
// Plain loads (no .nc): the panel vectors change while the kernel runs.
template <typename T>
__device__ __forceinline__ cpx<T> ld1(const T *base, int64_t e) {
    if constexpr (std::is_same<T, df>::value) {
        const float4 v = *(reinterpret_cast<const float4 *>(base) + e);
        return mk(df(v.x, v.y), df(v.z, v.w));
    } else if constexpr (std::is_same<T, double>::value) {
        const double2 v = *(reinterpret_cast<const double2 *>(base) + e);
        return mk(v.x, v.y);
    } else {
        const float2 v = *(reinterpret_cast<const float2 *>(base) + e);
        return mk(v.x, v.y);
    }
}
template <typename T>
__device__ __forceinline__ void st1(T *base, int64_t e, cpx<T> x) {
    if constexpr (std::is_same<T, df>::value)
        *(reinterpret_cast<float4 *>(base) + e) = make_float4(x.re.hi, x.re.lo, x.im.hi, x.im.lo);
    else if constexpr (std::is_same<T, double>::value)
        *(reinterpret_cast<double2 *>(base) + e) = make_double2(x.re, x.im);
    else
        *(reinterpret_cast<float2 *>(base) + e) = make_float2(x.re, x.im);
}
// x + s y and s y - x with fused operations (4 FP64 instructions; operators take 6)
__device__ __forceinline__ double fmadd(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ df fmadd(df a, df b, df c) { return fma(a, b, c); }
template <typename T>
__device__ __forceinline__ cpx<T> cfma(cpx<T> s, cpx<T> y, cpx<T> x) {
    return mk(fmadd(s.re, y.re, fmadd(-s.im, y.im, x.re)), fmadd(s.re, y.im, fmadd(s.im, y.re, x.im)));
}
// s c and y + s c for an FP32 c
__device__ __forceinline__ double scaled(double s, float c) { return s * (double)c; }
__device__ __forceinline__ df scaled(df s, float c) { return mul_f(s, c); }
__device__ __forceinline__ double scaled_add(double s, float c, double y) { return ::fma(s, (double)c, y); }
__device__ __forceinline__ df scaled_add(df s, float c, df y) { return fma_f(s, c, y); }
// v / scale in FP32
__device__ __forceinline__ float scaled32(double v, double inv) { return (float)(v * inv); }
__device__ __forceinline__ float scaled32(df v, float inv) { return v.hi * inv; }

// rows i0 .. i0 + RPT - 1 of a B x B block
template <typename T, int B, int RPT>
__device__ __forceinline__ void ld_block_rows(const T *__restrict__ blk, int i0, T (&a)[RPT * B]) {
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

// Sum of products with values of type T and an operand of type X (T, or FP32 vectors).
template <typename T>
struct PSum {
    T s;
    __device__ __forceinline__ void zero() { s = 0; }
    template <typename X>
    __device__ __forceinline__ void prod(T a, X x) { s = ::fma(a, (T)x, s); }
    template <typename X>
    __device__ __forceinline__ void val(X x) { s = s + (T)x; }
    __device__ __forceinline__ T get() const { return s; }
};
template <>
struct PSum<df> {
    DfSum s;
    __device__ __forceinline__ void zero() { s.zero(); }
    template <typename X>
    __device__ __forceinline__ void prod(df a, X x) { s.add_prod(a, x); }
    template <typename X>
    __device__ __forceinline__ void val(X x) { s.add_val(x); }
    __device__ __forceinline__ df get() const { return s.value(); }
};

// blocks of a block row; k0 < 0: not known yet
struct Range {
    int64_t k0, k1;
};

// y[i][q] = sum_j A(br*B + i0 + i, j) x(j, e0 + q) for CPT neighbouring columns of
// a panel with row stride W; unit: the diagonal block is the identity.
template <typename T, int B, int RPT, typename X, int CPT>
__device__ __forceinline__ void rows_product(const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                             const T *__restrict__ val, int64_t br, int i0, const X *x, int W, int c,
                                             bool unit, cpx<T> (&y)[RPT][CPT], Range rg) {
    const int64_t k0 = rg.k0 >= 0 ? rg.k0 : __ldg(rp + br), k1 = rg.k0 >= 0 ? rg.k1 : __ldg(rp + br + 1);
    PSum<T> sr[RPT][CPT], si[RPT][CPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int q = 0; q < CPT; ++q) sr[i][q].zero(), si[i][q].zero();
    int64_t col_n = k0 < k1 ? (int64_t)__ldg(ci + k0) : 0;
    constexpr int UNR = RPT * CPT == 1 ? (B == 9 ? 1 : 4) : (sizeof(X) == 4 || B == 9 ? 1 : 2);
#pragma unroll UNR
    for (int64_t k = k0; k < k1; ++k) {
        const int64_t col = col_n;
        if (k + 1 < k1) col_n = __ldg(ci + k + 1);
        cpx<X> v[B][CPT];
        const int64_t e = col * B * W + c;
#pragma unroll
        for (int j = 0; j < B; ++j) {
            if constexpr (CPT == 2) { // FP32, two columns: one 16-byte load
                const float4 f = *reinterpret_cast<const float4 *>(x + 2 * (e + (int64_t)j * W));
                v[j][0] = mk<X>(f.x, f.y), v[j][1] = mk<X>(f.z, f.w);
            } else {
                v[j][0] = ld1(x, e + (int64_t)j * W);
            }
        }
        if (unit && col == br) {
#pragma unroll
            for (int j = 0; j < B; ++j)
#pragma unroll
                for (int i = 0; i < RPT; ++i)
                    if (j == i0 + i) // i0 + i is a run-time row when RPT < B
#pragma unroll
                        for (int q = 0; q < CPT; ++q) sr[i][q].val(v[j][q].re), si[i][q].val(v[j][q].im);
        } else {
            T a[RPT * B];
            ld_block_rows<T, B, RPT>(val + k * (int64_t)(B * B), i0, a);
#pragma unroll
            for (int i = 0; i < RPT; ++i)
#pragma unroll
                for (int j = 0; j < B; ++j)
#pragma unroll
                    for (int q = 0; q < CPT; ++q) {
                        sr[i][q].prod(a[i * B + j], v[j][q].re);
                        si[i][q].prod(a[i * B + j], v[j][q].im);
                    }
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int q = 0; q < CPT; ++q) y[i][q] = mk(sr[i][q].get(), si[i][q].get());
}

// ------------------------------------------------------------- thread layout
// Teams of `lanes` threads (one per slot, or one per two neighbouring slots) take
// units of RPT rows of a block row.  Units are dealt in runs of `teams` per CTA, so
// the rows in flight form one window that sweeps the matrix (see spmm.cuh); when one
// pass covers all units they are dealt CTA by CTA instead, so a small system reaches
// every SM.  Which thread adds which rows depends on the number of slots alone, so a
// column's results do not depend on the others; threads of finished slots idle.
struct Layout {
    int lanes, teams, lane, team, c; // c: first slot of this thread, -1: idle
    int64_t u0, step;
    int64_t h0, h1, s0, s1; // block ranges of unit u0 in H and S (threads with one row: a load less in each phase's chain)
};
__device__ __forceinline__ Layout make_layout(int lanes, int cpt, int64_t units) {
    Layout l;
    l.lanes = lanes;
    l.teams = NT / lanes;
    l.team = threadIdx.x / lanes;
    l.lane = threadIdx.x - l.team * lanes;
    const bool on = l.team < l.teams;
    l.c = on ? l.lane * cpt : -1;
    const int64_t all = (int64_t)gridDim.x * l.teams;
    l.step = all;
    l.u0 = units <= all ? (int64_t)l.team * gridDim.x + blockIdx.x : (int64_t)blockIdx.x * l.teams + l.team;
    if (!on) l.u0 = units;
    return l;
}

// Largest power of two <= n, at most 32 (n >= 1).
__device__ __forceinline__ int pow2_le32(int n) { return n >= 32 ? 32 : (1 << (31 - __clz(n))); }

// K sums per slot: threads -> CTA (part[(slot * K + k) * grid + CTA]).
template <typename T, int K, int CPT = 1>
__device__ __forceinline__ void engine_partials(Acc<T> (&acc)[CPT * K], const Layout &l, void *part,
                                                typename Acc<T>::P *sp) {
    typedef typename Acc<T>::P P;
    if (l.team < l.teams) // (an idle slot's sums are zero)
#pragma unroll
        for (int k = 0; k < CPT * K; ++k) sp[(l.team * l.lanes + l.lane) * CPT * K + k] = acc[k].pack();
    __syncthreads();
    const int rows = l.lanes * CPT * K, R = rows >= NT ? 1 : pow2_le32(NT / rows), per = NT / R;
    const int sub = threadIdx.x % R;
    for (int q0 = 0; q0 < rows; q0 += per) {
        const int q = q0 + threadIdx.x / R;
        Acc<T> s;
        s.zero();
        if (q < rows)
            for (int t = sub; t < l.teams; t += R) s.add(Acc<T>::unpack(sp[t * rows + q]));
        group_reduce(s, R);
        if (sub == 0 && q < rows)
            reinterpret_cast<P *>(part)[(int64_t)q * gridDim.x + blockIdx.x] = s.pack();
    }
}

// out(row) = sum of n partials at row * ld + first, for the K rows of each slot (one CTA).  The values of a
// row are added pairwise: a chain of FP64 additions costs 76 cycles a link.
template <typename T, int K, class Out>
__device__ __forceinline__ void sum_rows(int slots, const void *part, int64_t ld, int first, int n, Out out) {
    typedef typename Acc<T>::P P;
    constexpr int U = 8;
    const int rows = slots * K, R = rows >= NT ? 1 : pow2_le32(NT / rows), per = NT / R;
    const int sub = threadIdx.x % R;
    Acc<T> z;
    z.zero();
    const P zp = z.pack();
    for (int q0 = 0; q0 < rows; q0 += per) {
        const int q = q0 + threadIdx.x / R;
        Acc<T> s;
        s.zero();
        if (q < rows) {
            const P *pp = reinterpret_cast<const P *>(part) + q * ld + first;
            for (int b0 = sub; b0 < n; b0 += R * U) {
                Acc<T> v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = Acc<T>::unpack(b0 + u * R < n ? __ldcg(pp + b0 + u * R) : zp);
#pragma unroll
                for (int h = U / 2; h > 0; h >>= 1)
#pragma unroll
                    for (int u = 0; u < h; ++u) v[u].add(v[u + h]);
                s.add(v[0]);
            }
        }
        group_reduce(s, R);
        if (sub == 0 && q < rows) out(q, s);
    }
}

// ------------------------------------------------------------------- kernel
template <typename T, int B, int RPT, bool HAS_S>
struct EngineRun {
    const Engine<T> &e;
    const Panel<T> &p;
    unsigned gen;
    struct Smem {
        typename Acc<T>::P sp[NT * 3 * (RPT > 1 && HAS_S ? 2 : 1)];
        ColState col[MAX_W]; // the last arriver's copy
        double red[MAX_W * 3], rho[MAX_W * 2];
        unsigned flags;
        int any, light, fail;
    };
    Smem &s;
    Layout l;
    int64_t units;
    int W, slot;

    __device__ __forceinline__ EngineRun(const Engine<T> &en, Smem &sm)
        : e(en), p(en.p), gen(0), s(sm), units(en.p.n_brows * (B / RPT)), W(en.W) {}

    // The grid barrier after a phase with K sums per slot (0: none): `last` runs in the
    // CTA that arrives last, with s.red filled, and returns the flags every CTA gets.
    // The sums are taken in two steps, by the last arriver of each group of about
    // sqrt(grid) CTAs and by the last of those: one SM adds 64 rows of 304 FP64
    // partials in 5.5 us (1.7 additions per clock), the groups' SMs in 0.4.  Who adds
    // what depends on the grid alone, so the sums are reproducible.  A wait gives up
    // after 20 s (or as soon as another one did), and the kernel ends.
    template <int K, class F>
    __device__ __forceinline__ unsigned step(int phase, F last) {
        GridBarrier *b = e.bar;
        gen = (gen + 1) & 0xffffffu;
        bool is_last = false;
        if (K == 0 || W * K * (int)gridDim.x <= 2048) { // few enough for one SM
            is_last = group_arrival(&b->arrive, gridDim.x);
            if constexpr (K > 0) {
                if (is_last) {
                    sum_rows<T, K>(W, p.part, gridDim.x, 0, gridDim.x,
                                   [&](int row, const Acc<T> &v) { s.red[row] = v.value(); });
                    __syncthreads();
                }
            }
        } else if constexpr (K > 0) {
            const int G = gridDim.x, gs = e.group, ng = (G + gs - 1) / gs, g = blockIdx.x / gs;
            const int n = min(gs, G - g * gs);
            is_last = group_arrival(b->grp[g], n);
            if (is_last) {
                typedef typename Acc<T>::P P;
                P *gp = reinterpret_cast<P *>(p.part) + (int64_t)MAX_W * 3 * G;
                sum_rows<T, K>(W, p.part, G, g * gs, n,
                               [&](int row, const Acc<T> &v) { gp[(int64_t)row * ng + g] = v.pack(); });
                is_last = group_arrival(&b->arrive, ng);
                if (is_last) {
                    sum_rows<T, K>(W, gp, ng, 0, ng, [&](int row, const Acc<T> &v) { s.red[row] = v.value(); });
                    __syncthreads();
                }
            }
        }
        if (is_last) {
            // the column states come into shared memory for the scalar work, in one trip to L2
            constexpr int CW = sizeof(ColState) / 8;
            static_assert(sizeof(ColState) % 8 == 0, "column state");
            unsigned long long *sc = reinterpret_cast<unsigned long long *>(s.col), *gc = reinterpret_cast<unsigned long long *>(p.col);
            if (K > 0) {
                for (int q = threadIdx.x; q < W * CW; q += NT) sc[q] = __ldcg(gc + q);
                __syncthreads();
            }
            const unsigned f = last();
            __syncthreads();
            if (K > 0) {
                for (int q = threadIdx.x; q < W * CW; q += NT) gc[q] = sc[q];
                __syncthreads();
            }
            if (threadIdx.x == 0) {
                __threadfence();
                if (e.profile) {
                    const unsigned long long t = global_ns();
                    b->ns[phase] += t - b->t_last;
                    b->cnt[phase] += 1;
                    b->t_last = t;
                }
                s.flags = f;
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&b->word), "r"((gen << 8) | f) : "memory");
            }
        } else if (threadIdx.x == 0) {
            unsigned w, spins = 0;
            const unsigned long long t0 = global_ns();
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(&b->word) : "memory");
                if ((w >> 8) == gen) break;
                __nanosleep(20);
                if ((++spins & 1023u) == 0 &&
                    (*(volatile int32_t *)&b->err || global_ns() - t0 > 20000000000ull)) {
                    *(volatile int32_t *)&b->err = 1;
                    w = F_ABORT;
                    break;
                }
            }
            s.flags = w & 0xffu;
        }
        __syncthreads();
        return s.flags;
    }

    // this thread's place, once, and whether its slot is at work, whenever a slot's column finished
    __device__ void place() {
        l = make_layout(W, 1, units);
        slot = l.c;
        if (RPT == 1 && l.u0 < units) {
            const int64_t br = l.u0 / B;
            l.h0 = p.h_rp[br], l.h1 = p.h_rp[br + 1];
            if constexpr (HAS_S) l.s0 = p.s_rp[br], l.s1 = p.s_rp[br + 1];
        }
        mark();
    }
    __device__ void mark() { l.c = slot >= 0 && !p.col[slot].done ? slot : -1; }
    __device__ __forceinline__ Range hrange(const Layout &g, int64_t u) const {
        return RPT == 1 && u == g.u0 ? Range{g.h0, g.h1} : Range{-1, 0};
    }
    __device__ __forceinline__ Range srange(const Layout &g, int64_t u) const {
        return RPT == 1 && u == g.u0 ? Range{g.s0, g.s1} : Range{-1, 0};
    }

    __device__ __forceinline__ void unit_rows(int64_t u, int64_t &br, int &i0) const {
        if constexpr (RPT == B) {
            br = u, i0 = 0;
        } else {
            constexpr int G = B / RPT;
            br = u / G, i0 = (int)(u - br * G) * RPT;
        }
    }

    // f(q) for the W * nz (slot, shift) pairs q, 32 to a warp: an FP64 instruction takes
    // its 19 cycles for one lane as for 32, and a pair has over a hundred
    template <class F>
    __device__ __forceinline__ void pairs(F f) {
        const int P = W * p.nz, nw = (P + 31) / 32, lane = threadIdx.x & 31;
        for (int w = blockIdx.x + (NT / 32 - 1 - (int)threadIdx.x / 32) * gridDim.x; w < nw; w += NT / 32 * gridDim.x)
            if (w * 32 + lane < P) f(w * 32 + lane);
    }

    // The shifted solutions on the kept rows, one (slot, kept row, shift) a thread,
    // shifts fastest, with the coefficients that the pairs left: p^m (and the QMR
    // iterate) from A's, then x^m from B's.  A slot that restarts (its arrays are
    // cleared already) is left out.
    template <bool UPD_A, bool UPD_B>
    __device__ void kept_rows() {
        const int64_t KM = p.max_col_ent, per = KM * p.nz, all = (int64_t)W * per;
        const bool small = all < (int64_t)UINT32_MAX;
        // runs of 32 items to a warp, dealt CTA by CTA
        for (int64_t i = (blockIdx.x + (int64_t)(threadIdx.x / 32) * gridDim.x) * 32 + (threadIdx.x & 31); i < all;
             i += (int64_t)NT * gridDim.x) {
            int c, m;
            int64_t k;
            rows_index(i, per, p.nz, small, c, k, m);
            const ColState &C = p.col[c];
            const int q = c * p.nz + m, n_ent = C.n_ent, restart = C.restart, fa = UPD_A ? p.flagA[q] : 0, fb = UPD_B ? p.flagB[q] : 0;
            if (k >= n_ent) continue;
            if (UPD_A && fa && !restart) {
                if (fa & 2) p.xq[i] = p.xq[i] + p.etaA[q] * (p.xs[i] - p.xq[i]);
                if (fa & 1) p.ps[i] = cfma(p.coefA[2 * q], e.kr[(int64_t)c * KM + k], p.coefA[2 * q + 1] * p.ps[i]);
            }
            if (UPD_B && fb) p.xs[i] = cfma(p.coefB[q], p.ps[i], p.xs[i]);
        }
    }
    // ---------------------------------------------------------------- phase A
    __device__ void phase_A(int n) {
        const T *R = HAS_S ? p.R[0] : p.RT;
        // the shifted recurrences and the kept rows' r_n on the highest threads: their FP64
        // chains and loads run beside the rows of the other warps
        pairs([&](int q) { pair_store_A(p, q, pair_coef_A(p, q, n)); });
        const int KM = p.max_col_ent;
        for (int64_t t = blockIdx.x + (int64_t)(NT - 1 - threadIdx.x) * gridDim.x; t < (int64_t)W * KM; t += (int64_t)NT * gridDim.x) {
            const int c = (int)(t / KM), k = (int)(t - (int64_t)c * KM);
            const ColState &C = p.col[c];
            if (k < C.n_ent) e.kr[t] = to64(ld1(R, p.ent_row[C.ent0 + k] * W + c));
        }
        Acc<T> acc[2];
        acc[0].zero(), acc[1].zero();
        if (l.c >= 0) {
            const cpx<T> be = e.sc[l.c].beta, zs = e.sc[l.c].zs;
            for (int64_t u = l.u0; u < units; u += l.step) {
                int64_t br;
                int i0;
                unit_rows(u, br, i0);
                cpx<T> y[RPT][1];
                rows_product<T, B, RPT, T, 1>(p.h_rp, p.h_ci, p.h_val, br, i0, R, W, l.c, false, y, hrange(l, u));
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int64_t o = (br * B + i0 + i) * W + l.c;
                    cpx<T> pv = ld1(R, o), rt = pv, uv = ld1(p.U, o);
                    if constexpr (HAS_S) rt = ld1(p.RT, o);
                    pv = cfma(be, ld1(p.P[0], o), pv);
                    st1(p.P[0], o, pv);
                    uv = cfma(zs, rt, cfma(be, uv, mk(-y[i][0].re, -y[i][0].im)));
                    st1(p.U, o, uv);
                    acc[0].add(pv.re * uv.re);
                    acc[0].add(-(pv.im * uv.im));
                    acc[1].add(pv.re * uv.im);
                    acc[1].add(pv.im * uv.re);
                }
            }
        }
        engine_partials<T, 2>(acc, l, p.part, s.sp);
    }

    // ---------------------------------------------------------------- phase B
    __device__ void phase_B(int n) {
        pairs([&](int q) {
            c64 as;
            const bool on = pair_coef_B(p, q, as);
            pair_store_B(p, q, on, as);
        });
        constexpr int K = HAS_S ? 1 : 3;
        Acc<T> acc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k].zero();
        if (l.c >= 0) {
            const SlotScalars<T> &C = e.sc[l.c];
            const cpx<T> nal = mk(-C.alpha.re, -C.alpha.im);
            const int step = C.step;
            const bool rst = C.restart != 0;
            const int64_t jrow = C.row;
            const auto inv = C.inv;
            // no product here: one row at a time, whatever RPT is (units of RPT rows)
            for (int64_t u = l.u0; u < units; u += l.step) {
                cpx<T> rt[RPT], uv[RPT];
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int64_t o = (u * RPT + i) * W + l.c;
                    rt[i] = ld1(p.RT, o);
                    uv[i] = ld1(p.U, o);
                }
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int64_t row = u * RPT + i, o = row * W + l.c;
                    if (rst) {
                        rt[i] = mk<T>(row == jrow ? (T)1 : (T)0, 0);
                        clear_restart_row(p, W, n, row, l.c);
                    } else {
                        rt[i] = cfma(nal, uv[i], mul_pow2(step, rt[i]));
                    }
                    st1(p.RT, o, rt[i]);
                    const T rr = rt[i].re * rt[i].re, ii = rt[i].im * rt[i].im;
                    if constexpr (HAS_S) {
                        acc[0].add(rr);
                        acc[0].add(ii);
                        st1(p.T32, o, mk(scaled32(rt[i].re, inv), scaled32(rt[i].im, inv)));
                    } else {
                        acc[0].add(rr);
                        acc[0].add(-ii);
                        acc[1].add((T)2 * rt[i].re * rt[i].im);
                        acc[2].add(rr);
                        acc[2].add(ii);
                    }
                }
            }
        }
        engine_partials<T, K>(acc, l, p.part, s.sp);
    }

    // ------------------------------------------------ Chebyshev step k of a sweep
    // x_1 = b / theta is not stored: step 1 multiplies b, step 2 takes x_1 from b.
    template <int CPT>
    __device__ __forceinline__ void cheb_rows(const Layout &g, int k) {
        if (g.c < 0) return;
        const float om = e.om[k], ga = e.ga[k], it = e.inv_theta;
        const float *xk = k == 1 ? p.T32 : e.X[k & 1];
        float *xn = e.X[(k + 1) & 1]; // holds x_{k-1} from step 3 on
        for (int64_t u = g.u0; u < units; u += g.step) {
            int64_t br;
            int i0;
            unit_rows(u, br, i0);
            cpx<float> sx[RPT][CPT];
            float b[2 * CPT], x[2 * CPT], xm[2 * CPT];
            auto own = [&](int i) {
                const int64_t o = (br * B + i0 + i) * W + g.c;
                auto ld = [&](const float *q, float(&v)[2 * CPT]) {
                    if constexpr (CPT == 2) {
                        const float4 f = *reinterpret_cast<const float4 *>(q + 2 * o);
                        v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
                    } else {
                        const float2 f = *reinterpret_cast<const float2 *>(q + 2 * o);
                        v[0] = f.x, v[1] = f.y;
                    }
                };
                ld(p.T32, b);
                if (k > 1) ld(xk, x);
                if (k > 2) ld(xn, xm);
            };
            if constexpr (RPT == 1) own(0); // in flight during the product
            rows_product<float, B, RPT, float, CPT>(p.s_rp, p.s_ci, p.s_val32, br, i0, xk, W, g.c, p.s_unit, sx, srange(g, u));
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int64_t o = (br * B + i0 + i) * W + g.c;
                if constexpr (RPT > 1) own(i);
#pragma unroll
                for (int q = 0; q < 2 * CPT; ++q) {
                    float sv = q & 1 ? sx[i][q / 2].im : sx[i][q / 2].re;
                    if (k == 1) x[q] = b[q] * it, xm[q] = 0.f, sv *= it;
                    if (k == 2) xm[q] = b[q] * it;
                    x[q] = x[q] + (om * (x[q] - xm[q]) + ga * (b[q] - sv));
                }
                if constexpr (CPT == 2)
                    *reinterpret_cast<float4 *>(xn + 2 * o) = make_float4(x[0], x[1], x[2], x[3]);
                else
                    *reinterpret_cast<float2 *>(xn + 2 * o) = make_float2(x[0], x[1]);
            }
        }
    }
    __device__ void phase_X(int k) {
        if constexpr (RPT > 1) {
            if (W % 2 == 0) { // two slots a thread (a finished slot's sweep is of no use and of no harm)
                const Layout g = make_layout(W / 2, 2, units);
                return cheb_rows<2>(g, k);
            }
        }
        cheb_rows<1>(l, k);
    }

    // ------------------------------------------------------------ refinement pass
    // The pass in FP32 (mode 2 of phase_R) for kernels with the rows of a block in a
    // thread: two slots a thread halve the loads of S and of the index arrays.
    __device__ void phase_R32x2() {
        const Layout g = make_layout(W / 2, 2, units);
        const float *c32 = e.X[e.terms2 & 1];
        Acc<T> acc[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) acc[k].zero();
        if (g.c >= 0) {
            const SlotScalars<T> *sc = e.sc + g.c;
            const T sig[2] = {sc[0].sig, sc[1].sig};
            const float ratio[2] = {sc[0].ratio, sc[1].ratio};
            for (int64_t u = g.u0; u < units; u += g.step) {
                int64_t br;
                int i0;
                unit_rows(u, br, i0);
                cpx<float> sf[RPT][2];
                rows_product<float, B, RPT, float, 2>(p.s_rp, p.s_ci, p.s_val32, br, i0, c32, W, g.c, p.s_unit, sf, Range{-1, 0});
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int64_t o = (br * B + i0 + i) * W + g.c;
                    const float4 c4 = *reinterpret_cast<const float4 *>(c32 + 2 * o), b4 = *reinterpret_cast<const float4 *>(p.T32 + 2 * o);
                    const float c[4] = {c4.x, c4.y, c4.z, c4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
                    float t[4];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const cpx<T> rt = ld1(p.RT, o + q);
                        cpx<T> y = ld1(p.R[0], o + q);
                        y = mk(scaled_add(sig[q], c[2 * q], y.re), scaled_add(sig[q], c[2 * q + 1], y.im));
                        st1(p.R[0], o + q, y);
                        const float tr = b[2 * q] - sf[i][q].re, ti = b[2 * q + 1] - sf[i][q].im;
                        t[2 * q] = tr * ratio[q], t[2 * q + 1] = ti * ratio[q];
                        acc[3 * q].add(tr * tr + ti * ti);
                        acc[3 * q + 1].add(y.re * rt.re);
                        acc[3 * q + 1].add(-(y.im * rt.im));
                        acc[3 * q + 2].add(y.re * rt.im);
                        acc[3 * q + 2].add(y.im * rt.re);
                    }
                    *reinterpret_cast<float4 *>(p.T32 + 2 * o) = make_float4(t[0], t[1], t[2], t[3]);
                }
            }
        }
        engine_partials<T, 3, 2>(acc, g, p.part, s.sp);
    }
    __device__ __forceinline__ int terms_of(int mode) const { return mode == 0 ? e.terms : e.terms2; }
    // mode 0: y = sigma c, t = rt - S y (first pass); 1: y += sigma c, t -= S sigma c;
    // 2: as 1 with S c and the residual in FP32 (the correction is small, see engine_light)
    __device__ void phase_R(int mode) {
        if constexpr (RPT > 1 && HAS_S) {
            if (mode == 2 && W % 2 == 0) return phase_R32x2();
        }
        const float *c32 = e.X[terms_of(mode) & 1];
        Acc<T> acc[3];
        acc[0].zero(), acc[1].zero(), acc[2].zero();
        if (l.c >= 0) {
            const T sig = e.sc[l.c].sig;
            const auto inv = e.sc[l.c].inv;
            const float ratio = e.sc[l.c].ratio;
            for (int64_t u = l.u0; u < units; u += l.step) {
                int64_t br;
                int i0;
                unit_rows(u, br, i0);
                cpx<T> sc[RPT][1];
                cpx<float> sf[RPT][1];
                if (mode == 2)
                    rows_product<float, B, RPT, float, 1>(p.s_rp, p.s_ci, p.s_val32, br, i0, c32, W, l.c, p.s_unit, sf, srange(l, u));
                else
                    rows_product<T, B, RPT, float, 1>(p.s_rp, p.s_ci, p.s_val, br, i0, c32, W, l.c, p.s_unit, sc, srange(l, u));
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    const int64_t o = (br * B + i0 + i) * W + l.c;
                    const cpx<float> c = ld1(c32, o);
                    const cpx<T> rt = ld1(p.RT, o);
                    cpx<T> y;
                    if (mode == 0) {
                        y = mk(scaled(sig, c.re), scaled(sig, c.im));
                    } else {
                        y = ld1(p.R[0], o);
                        y = mk(scaled_add(sig, c.re, y.re), scaled_add(sig, c.im, y.im));
                    }
                    st1(p.R[0], o, y);
                    if (mode == 2) {
                        const cpx<float> b = ld1(p.T32, o);
                        const float tr = b.re - sf[i][0].re, ti = b.im - sf[i][0].im;
                        st1(p.T32, o, mk(tr * ratio, ti * ratio));
                        acc[0].add(tr * tr + ti * ti);
                    } else {
                        cpx<T> t = mode == 0 ? rt : ld1(p.Tv, o);
                        t = mk(t.re - sig * sc[i][0].re, t.im - sig * sc[i][0].im);
                        st1(p.Tv, o, t);
                        st1(p.T32, o, mk(scaled32(t.re, inv), scaled32(t.im, inv)));
                        acc[0].add(t.re * t.re);
                        acc[0].add(t.im * t.im);
                    }
                    acc[1].add(y.re * rt.re);
                    acc[1].add(-(y.im * rt.im));
                    acc[2].add(y.re * rt.im);
                    acc[2].add(y.im * rt.re);
                }
            }
        }
        engine_partials<T, 3>(acc, l, p.part, s.sp);
    }

    // the sweep of slot c works on residuals / sig; the pass behind it scales by the norm it finds there
    __device__ __forceinline__ void set_sweep(int c, double sig, double t2) {
        const double inv = 1.0 / safe_scale(t2);
        e.sc[c].sig = (T)sig;
        e.sc[c].inv = inv;
        e.sc[c].ratio = (float)(sig * inv);
    }
    // what A needs of the recurrences (behind finish_outer)
    __device__ __forceinline__ void set_outer() {
        for (int c = threadIdx.x; c < W; c += NT) {
            e.sc[c].beta = cvt<T>(s.col[c].beta_vec);
            e.sc[c].zs = cvt<T>(s.col[c].zs);
        }
    }

    // end of a refinement pass: another sweep, or the end of the outer iteration
    __device__ unsigned finish_R(int mode, int init) {
        if (threadIdx.x == 0) s.any = 0, s.light = 1, s.fail = 0;
        __syncthreads();
        for (int c = threadIdx.x; c < W; c += NT) {
            ColState &C = s.col[c];
            if (C.done) continue;
            double t2 = s.red[3 * c];
            if (mode == 2) t2 *= C.in_sig * C.in_sig;
            const double eta2 = p.inner_tol * p.inner_tol * C.rn2;
            // (written so that a t2 that is not finite, an FP32 sweep that overflowed, fails too)
            if (isfinite(C.in_t2) && !(t2 <= 1e-4 * C.in_t2) && !(t2 <= eta2)) s.fail = 1;
            C.in_sig = safe_scale(C.in_t2); // the scale the rows used for the next sweep
            C.in_t2 = t2;
            set_sweep(c, C.in_sig, t2);
            C.in_refines += 1;
            if (t2 > eta2 && isfinite(t2) && C.in_refines < p.refine_max) {
                s.any = 1;
                const double lim = e.light * p.inner_tol;
                if (!(t2 <= lim * lim * C.rn2)) s.light = 0;
            }
            s.rho[2 * c] = s.red[3 * c + 1];
            s.rho[2 * c + 1] = s.red[3 * c + 2];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            p.ctl->inner_total += terms_of(mode) - 1;
            p.ctl->refine_total += 1;
            p.ctl->light_total += (mode == 2);
            if (s.fail) e.bar->fail = 1;
        }
        if (s.fail) return F_DONE;
        if (s.any) return F_AGAIN | (s.light ? F_LIGHT : 0u);
        finish_outer(p, W, s.rho, init, s.col);
        set_outer();
        return outer_flags(init);
    }
    __device__ __forceinline__ unsigned outer_flags(int init) {
        __syncthreads();
        if (threadIdx.x == 0)
            s.any = init || (!p.ctl->panel_done && p.ctl->iter_ctr < p.outer_cap);
        __syncthreads();
        return s.any ? F_CONT : 0u;
    }

    // r = S^-1 rt by sweeps and refinement passes; the flags of the last pass
    __device__ unsigned inner_solve(int init) {
        int mode = 0;
        for (;;) {
            for (int k = 1; k < terms_of(mode); ++k) {
                // the kept rows' FP64 updates run beside the first FP32 product
                if (!init && mode == 0 && k == 1) kept_rows<true, true>();
                phase_X(k);
                const unsigned f = step<0>(PH_X, [] { return 0u; });
                if (f & F_ABORT) return f;
            }
            phase_R(mode);
            const int md = mode;
            const unsigned f = step<3>(md == 2 ? PH_R32 : PH_R, [&] { return finish_R(md, init); });
            if (!(f & F_AGAIN)) return f;
            mode = (f & F_LIGHT) ? 2 : 1;
        }
    }

    __device__ void init() {
        const int64_t tid = blockIdx.x * (int64_t)NT + threadIdx.x, stride = (int64_t)gridDim.x * NT;
        const int64_t total = p.n_brows * B * W;
        const cpx<T> zero = mk((T)0, (T)0);
        for (int64_t t = tid; t < total; t += stride) {
            const int c = (int)(t % W);
            const bool one = c < p.n_cols && p.col_row[c] == t / W;
            st1(p.RT, t, mk((T)(one ? 1 : 0), (T)0));
            st1(p.U, t, zero);
            st1(p.P[0], t, zero);
            if constexpr (HAS_S) {
                st1(p.T32, t, mk(one ? 1.f : 0.f, 0.f));
            }
        }
        const int64_t ne = (int64_t)W * p.max_col_ent * p.nz;
        for (int64_t t = tid; t < ne; t += stride) {
            p.xs[t] = mk(0.0, 0.0);
            p.ps[t] = mk(0.0, 0.0);
            if (p.xq) p.xq[t] = mk(0.0, 0.0);
        }
        for (int64_t q = tid; q < (int64_t)W * p.nz; q += stride) p.sh[q] = fresh_shift();
        if (tid < W) {
            ColState C = fresh_column(p, tid);
            C.in_sig = C.in_t2 = 1.0;
            p.col[tid] = C;
            set_sweep((int)tid, 1.0, 1.0);
            e.sc[tid].beta = mk((T)0, (T)0);
            e.sc[tid].zs = cvt<T>(C.zs);
        }
        if (tid == 0) p.ctl->next_col = p.n_cols < W ? p.n_cols : W; // the rest of *ctl is zero
    }

    __device__ void run() {
        init();
        unsigned f = step<0>(PH_INIT, [] { return 0u; });
        place();
        int n = 0;
        bool pend = false; // S = I: the x^m update of the last B is still to do
        if constexpr (HAS_S)
            f = inner_solve(1);
        else
            f = (f & F_ABORT) ? f : (unsigned)F_CONT;
        while (f & F_CONT) {
            if (!HAS_S && pend) kept_rows<false, true>();
            pend = false;
            phase_A(n);
            f = step<2>(PH_A, [&] {
                const bool fin = finish_alpha(p, W, s.red, s.col);
                for (int c = threadIdx.x; c < W; c += NT) {
                    const ColState &C = s.col[c];
                    e.sc[c].alpha = cvt<T>(C.step ? pow2d(C.step) * C.alpha : C.alpha);
                    e.sc[c].step = C.step;
                    e.sc[c].restart = C.restart;
                    e.sc[c].row = C.row;
                    if constexpr (HAS_S) e.sc[c].inv = 1.0 / (C.restart ? 1.0 : safe_scale(C.rn2));
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    s.any = p.ctl->panel_done;
                    if (s.any) p.ctl->iter_ctr += 1;
                }
                __syncthreads();
                return (fin ? F_LIST : 0u) | (s.any ? F_DONE : 0u);
            });
            if (f & (F_DONE | F_ABORT)) break;
            if (f & F_LIST) mark();
            if (!HAS_S) kept_rows<true, false>();
            phase_B(n);
            pend = true;
            f = step<HAS_S ? 1 : 3>(PH_B, [&] {
                if constexpr (HAS_S) {
                    for (int c = threadIdx.x; c < W; c += NT) {
                        ColState &C = s.col[c];
                        if (C.done) continue;
                        C.in_sig = C.restart ? 1.0 : safe_scale(C.rn2); // the scale the rows used
                        C.rn2 = s.red[c];
                        C.in_t2 = C.rn2;
                        C.in_refines = 0;
                        set_sweep(c, C.in_sig, C.in_t2);
                    }
                    return 0u;
                } else {
                    for (int c = threadIdx.x; c < W; c += NT) {
                        s.rho[2 * c] = s.red[3 * c];
                        s.rho[2 * c + 1] = s.red[3 * c + 1];
                        if (!s.col[c].done) s.col[c].rn2 = s.red[3 * c + 2];
                    }
                    __syncthreads();
                    finish_outer(p, W, s.rho, 0, s.col);
                    set_outer();
                    return outer_flags(0);
                }
            });
            if (f & F_ABORT) break;
            if constexpr (HAS_S) f = inner_solve(0);
            ++n;
        }
        if (f & F_ABORT) return;
        if (!HAS_S && pend) { // the loop's cap was reached behind a B
            kept_rows<false, true>();
            f = step<0>(PH_INIT, [] { return 0u; });
            if (f & F_ABORT) return;
        }
        if (!p.G) return;
        // results of the columns still in their slots (the others were written when they retired)
        const int64_t stride = (int64_t)gridDim.x * NT, tid = blockIdx.x * (int64_t)NT + threadIdx.x;
        const int64_t per_slot = (int64_t)p.max_col_ent * p.nz;
        for (int64_t t = tid; t < W * per_slot; t += stride) {
            const ColState &C = p.col[t / per_slot];
            const int64_t r = t % per_slot;
            if (C.dst < 0 || r >= (int64_t)C.n_ent * p.nz) continue;
            p.G[C.ent0 * p.nz + r] = p.qmr ? p.xq[t] : p.xs[t];
        }
        for (int64_t q = tid; q < (int64_t)W * p.nz; q += stride) {
            const int64_t dst = p.col[q / p.nz].dst;
            if (dst >= 0) p.resid[dst * p.nz + q % p.nz] = p.sh[q].resid;
        }
        if (tid < W) {
            const ColState &C = p.col[tid];
            if (C.dst >= 0) {
                p.iters[C.dst] = C.iters;
                p.status[C.dst] = C.done ? C.status : TB_COL_MAX_ITER;
            }
        }
        if (tid == 0 && p.stats) {
            p.stats[0] = p.ctl->iter_ctr;
            p.stats[1] = p.ctl->inner_total;
            p.stats[2] = p.ctl->refine_total;
            p.stats[3] = p.ctl->light_total;
        }
    }
};

// CTAs per SM the kernel is compiled for: three when a thread holds the rows of a
// block, two when it holds one row of a system that may be small.  At three a thread has
// 80 registers: k_engine<df, 4, 4, S> spills 1008 bytes of stores and 1152 of loads, <df, 9, 3,
// S> 928 and 1176 (-Xptxas -v).  The same kernels without S, which have the same A, spill 12 to
// 20 bytes, so that is R's df product and the FP32 passes.  Two CTAs (128 registers, none
// spilled) were slower as a whole: A 382 us against 397, X 96 against 82, R in FP32 279 against 227.
template <int RPT>
constexpr int engine_ctas() { return RPT > 1 ? 3 : 2; }

template <typename T, int B, int RPT, bool HAS_S>
__global__ void __launch_bounds__(NT, engine_ctas<RPT>()) k_engine(const __grid_constant__ Engine<T> e) {
    __shared__ typename EngineRun<T, B, RPT, HAS_S>::Smem s;
    EngineRun<T, B, RPT, HAS_S>(e, s).run();
}

// ------------------------------------------------------------------ host side
// Chebyshev coefficients of a sweep for a spectrum within [lo, hi] (x_{k+1} = x_k +
// om_k (x_k - x_{k-1}) + ga_k (b - S x_k), x_1 = b / theta; Saad, Iterative Methods,
// Sec. 12.3; the first n of them are those of a sweep of n terms).  The sweeps of an
// inner solve share inner_tol evenly, each at best 3e-7 (FP32 rounding); false where they
// would take more than inner_max products in a sweep (df) or in all (FP64), or the bounds
// are not those of a definite matrix.
// light > 0 (df panels, engine_light): where the first sweep can end below light inner
// tolerances, FP32 rounding included, it is given the terms for a quarter of that and the
// others what is left: the passes behind it then run in FP32.  C2 (hi / lo 1.6): 8 and 6
// terms, 12 products, as 7 and 7 take, which left the first residual at 5e-7, above light.
template <class E>
bool chebyshev_terms(double lo, double hi, double inner_tol, int inner_max, bool lowp, E &en, double light = 0.0,
                     int32_t *terms2 = nullptr) {
    // (FP32 holds the values of S and the coefficients, which go with 1 / hi)
    if (!(lo > 1e-30) || !(hi >= lo) || !(hi < 1e30) || hi > 30 * lo) return false;
    const double theta = 0.5 * (hi + lo), delta = std::max(0.5 * (hi - lo), 1e-3 * theta), s1 = theta / delta;
    const double rate = s1 - std::sqrt(s1 * s1 - 1.0);
    auto terms_for = [&](double target) {
        int n = 2;
        while (n < MAX_TERMS && 2 * std::pow(rate, n) > target) ++n;
        return n;
    };
    const int passes = std::max(1, (int)std::ceil(std::log(inner_tol) / std::log(3e-7)));
    const double target = std::max(0.5 * std::pow(inner_tol, 1.0 / passes), 1e-7);
    int terms = terms_for(target), second = terms;
    if (2 * std::pow(rate, terms) > target || (terms - 1) * (lowp ? 1 : passes) > inner_max) return false;
    const double rounding = 1.2e-7 * std::sqrt(hi / lo);
    if (light > 0.0 && passes == 2) {
        const int first = terms_for(0.25 * light * inner_tol);
        const double left = 2 * std::pow(rate, first) + rounding;
        if (left <= light * inner_tol && first - 1 <= inner_max) {
            terms = first;
            second = terms_for(inner_tol / left);
        }
    }
    en.terms = terms;
    if (terms2) *terms2 = second;
    en.inv_theta = (float)(1.0 / theta);
    double rho = 1.0 / s1;
    for (int k = 1; k < std::max(terms, second); ++k) {
        const double next = 1.0 / (2.0 * s1 - rho);
        en.om[k] = (float)(next * rho);
        en.ga[k] = (float)(2.0 * next / delta);
        rho = next;
    }
    return true;
}

// Bounds of the spectrum of S (lanczos.cu); *lo > *hi when there are none.
int spectral_bounds(tb_ctx *ctx, const int64_t *rp, const int32_t *ci, const double *val, int64_t n_brows, int b,
                    int sms, cudaStream_t s, double *lo, double *hi);

struct EngineLaunch {
    tb_ctx *ctx;
    Engine<double> e; // type-erased (T-dependent members are pointers)
    bool has_s;
    int per_sm;       // CTAs per SM asked for (0: as many as the kernel is compiled for)
    int sms;
    cudaStream_t stream;
    int rc = TB_OK;

    template <typename T, int B, int RPT, bool HAS_S>
    void go() {
        Engine<T> en;
        static_assert(sizeof(Engine<T>) == sizeof(Engine<double>), "layout");
        std::memcpy(&en, &e, sizeof(en));
        const void *fn = (const void *)k_engine<T, B, RPT, HAS_S>;
        int occ = 0;
        cudaError_t er = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, NT, 0);
        if (er != cudaSuccess || occ < 1) {
            rc = set_error(ctx, TB_ERR_CUDA, "panel solver occupancy: %s", cudaGetErrorString(er));
            return;
        }
        const int64_t units = e.p.n_brows * (B / RPT), thr = (units * e.W + NT - 1) / NT;
        const int64_t cap = (int64_t)sms * std::min(occ, per_sm > 0 ? per_sm : occ);
        const int g = (int)std::max<int64_t>(1, std::min(cap, std::max(thr, std::min<int64_t>(sms, units))));
        en.group = 1;
        while (en.group * en.group < g || (g + en.group - 1) / en.group > 64) ++en.group;
        void *args[] = {&en};
        er = cudaLaunchCooperativeKernel(fn, dim3(g), dim3(NT), args, 0, stream);
        if (er != cudaSuccess) rc = set_error(ctx, TB_ERR_CUDA, "panel solver launch: %s", cudaGetErrorString(er));
    }
    // rows of a thread: FP64 one (its pipe sets the time).  df a block row (b = 4) or three rows (b = 9), which
    // reads each neighbour once, unless that leaves less than four CTAs of 64 threads' work per SM; then one.
    template <typename T, int B, bool HAS_S>
    void rows() {
        constexpr int BIG = std::is_same<T, df>::value ? (B == 9 ? 3 : B) : 1;
        if constexpr (BIG > 1) {
            if (e.p.n_brows * (B / BIG) * e.W >= (int64_t)sms * 256) return go<T, B, BIG, HAS_S>();
        }
        go<T, B, 1, HAS_S>();
    }
    template <typename T>
    bool run(int b) {
        switch (b) {
        case 1: has_s ? rows<T, 1, true>() : rows<T, 1, false>(); return true;
        case 4: has_s ? rows<T, 4, true>() : rows<T, 4, false>(); return true;
        case 9: has_s ? rows<T, 9, true>() : rows<T, 9, false>(); return true;
        }
        return false;
    }
};

bool launch_engine_f64(EngineLaunch &L, int b);
bool launch_engine_df(EngineLaunch &L, int b);

} // namespace tbgf
