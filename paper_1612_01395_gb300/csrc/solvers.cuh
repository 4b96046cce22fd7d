// Persistent cooperative solver kernels: one launch runs a whole solve.
//
// A thread owns the rows lo + threadIdx.x + m * row_step below hi in every
// phase. On a grid lo is the block's first row and row_step the threads of the
// grid, so all blocks sweep through the rows together and a row's neighbours a
// plane away were read moments before by another block and are still in L2
// (contiguous ranges per block read them again from DRAM: 256^3 CSR rows, 413
// bytes a row and iteration against 360, 1212 against 1073 us); a block or
// cluster that solves alone owns a contiguous range. A phase is one sweep over
// the rows that fuses an SpMV, the AXPY recurrences that consume it and the
// partial dot products of a reduction; phases are separated by exchange /
// grid_sync. An exchange also forms the scalars (alpha, beta, omega, rho), the
// same in every block, so they never leave the GPU and the host is not involved
// between iterations.
//
// Pipelined BiCGStab (Algorithm 9) takes 2 grid-wide synchronisations per
// iteration: on one GPU the SpMV of each phase needs its input vector complete
// across the grid, and that same synchronisation completes the reduction whose
// scalar the phase consumes -- the two reductions of Algorithm 9 ride on the
// two synchronisations its SpMVs need anyway. Standard BiCGStab (Algorithm 7)
// needs 3 (variant 3: neighbour values of p and q are formed on the fly inside
// the SpMV) or 5 (variant 5: p and q are written first, fewer FP64 operations).
#pragma once

#include "dots.cuh"
#include "operators.cuh"

namespace pbcg {

template <typename T>
struct VectorsT {
    T *r, *r0, *p, *s, *z, *q, *y, *w, *t, *v;
};
using Vectors = VectorsT<double>;

template <typename T>
struct SolveArgsT {
    int n;
    const T *b;
    T *x;
    VectorsT<T> V;
    Control *ctl;
    double *partials;
    double *hist;       // nullable
    double rtol;
    int limit;          // iterations allowed (maxit or fixed_iters)
    int fixed;          // 1: ignore rtol
    int replace_period;
    int max_repl;       // < 0: unlimited
    int variant;        // Algorithm 7 only: 3 or 5
    // preconditioned solves (Algorithms 10 and 11): M^{-1} u = minv .* u and the
    // hat vectors r^, s^, z^, q^, w^ (null when unpreconditioned)
    const T *minv;
    T *rh, *sh, *zh, *qh, *wh;
};
using SolveArgs = SolveArgsT<double>;

// Threads per block of a grid solver kernel; both kinds fill an SM with 1024
// threads at 64 registers. Every block repeats an exchange's arrival, polling
// and slot sums, so large blocks are cheaper: at 1216 blocks of 128 threads an
// exchange cost about 15 us, at 304 of 512 about 5. Per iteration of Algorithm
// 9 (stencil): 110k unknowns 28.7 us with 304 blocks of 128 threads, 22.1 with
// 152 of 256; 2.1M 178 and 138 us; 16.8M 1177 and 940 us (with the wide sums).
template <bool Wide>
struct SolverBlock {
    static constexpr int kThreads = Wide ? 512 : 256;
};

// lo of a grid kernel's thread. Consecutive runs of 32 rows go to the same warp
// of consecutive blocks, so that a sweep with fewer rows (or groups of rows)
// than threads, or a last round that is not full, still uses every SM. Against
// blockDim.x rows in a row per block, us per iteration of Algorithm 9: 48^3
// 22.2 -> 21.4, 96^3 74.7 -> 72.4, 256^3 CSR 1088 -> 1047, 200k random rows
// 91.1 -> 82.1; FP32 stencil iterations of 64^3 26.0 -> 25.0, 110^3 68.0 ->
// 58.7. The FP32 CSR sweeps of 7-point rows lost 2 to 3 % (193x160x131 184 ->
// 190) and keep whole blocks of rows.
__device__ __forceinline__ int grid_lo() {
    return (int)(((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u + (threadIdx.x & 31u)) - (int)threadIdx.x;
}

struct Outcome {
    int iters, status, half, nrr;
    double nr0, nr;   // nr: squared norm of the last recursive residual (or of q after a half step)
};

// The steps are unsigned: the row after the last may lie above 2^31.
#define PBCG_STEPS(i, end)                                            \
    for (int i = lo + (int)threadIdx.x; (unsigned)i < (unsigned)(end); \
         i = (int)((unsigned)i + (unsigned)row_step(g)))
#define PBCG_ROWS(i) PBCG_STEPS(i, hi)

// A sweep of Algorithms 7 and 10 without a product with A, two of the thread's
// rows a step: load(i) returns a row's values, use(i, values) may store. Bound
// by DRAM, and the compiler moves no load across a store, so one row a step
// left too few loads in flight. An iteration of Algorithm 7 takes 825 us
// against 931 at 256^3, 120 against 130 at 128^3, 241 against 247 on CSR at
// 2048^2; of Algorithm 10 at 500,001 rows 191 against 201. Three and four rows
// a step, guarded one by one, were slower (869 and 890 us at 256^3).
template <class Sync, class Load, class Use>
__device__ __forceinline__ void sweep_pairs(const Sync &g, int lo, int hi, Load load, Use use) {
    const unsigned step = (unsigned)row_step(g), end = (unsigned)hi;
    for (unsigned i = (unsigned)lo + threadIdx.x; i < end; i += 2 * step) {
        const unsigned j = i + step;
        const bool two = j < end;
        decltype(load(0)) v = load((int)i), w = {};
        if (two) w = load((int)j);
        use((int)i, v);
        if (two) use((int)j, w);
    }
}
struct Row2 {
    double a, b;
};
struct Row3 {
    double a, b, c;
};
struct Row4 {
    double a, b, c, d;
};
struct Row5 {
    double a, b, c, d, e;
};
struct Row6 {
    double a, b, c, d, e, f;
};

// Tests on scalars that need no FP64 instruction (64 cycles of a sub-partition's
// FP64 pipe, about 140 to its result): finite and zero from the bits, and the
// order of non-negative numbers as the order of their bits.
__device__ __forceinline__ bool is_finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool is_zero(double v) { return (__double_as_longlong(v) << 1) == 0; }
template <int K>
__device__ __forceinline__ bool all_finite(const double (&v)[K]) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < K; ++i) ok = ok && is_finite(v[i]);
    return ok;
}

// sqrt(sq) <= tol for a finite sq >= 0. The root (about ten FP64 instructions)
// is taken only where it decides: sqrt(sq) <= tol implies sq <= 2 tol^2 unless
// tol^2 underflows. bound: 2 tol^2, or infinity where tol^2 is below the normal
// range.
__device__ __forceinline__ bool norm_below(double sq, double tol, double bound) {
    return __double_as_longlong(sq) <= __double_as_longlong(bound) && sqrt(sq) <= tol;
}
__device__ __forceinline__ double norm_bound(double tol) {
    const double t2 = __dmul_rn(tol, tol);
    return t2 >= 2.2250738585072014e-308 ? 2.0 * t2 : __longlong_as_double(0x7ff0000000000000ll);
}

// The scalar steps of an iteration. Each runs on one warp of a block (the last
// block to arrive, on large grids), with all lanes alike, inside an exchange:
// an FP64 instruction occupies its sub-partition's FP64 pipe for 64 cycles and
// takes about 140 to complete, so tests and divisions repeated by every warp
// of every resident block queued on the pipes between two sweeps.

// r_0: rho = (r0, r_0), the stopping tolerance
__device__ __forceinline__ void start_scalars(Scalars &S, double rr, double rtol) {
    S.rho = rr;
    S.nr = rr;
    S.nr0 = sqrt(rr);
    S.tol = __dmul_rn(rtol, S.nr0);
    S.bound = norm_bound(S.tol);
    S.alpha = S.beta = S.omega = 0.0;
    S.status = PBCG_OK;
    S.action = is_zero(S.nr0) ? kStop : kGo;
}
__device__ __forceinline__ void stop_scalars(Scalars &S, int status) {
    S.action = kStop;
    S.status = status;
}
// alpha = rho / d
__device__ __forceinline__ void alpha_scalars(Scalars &S, double d) {
    S.action = kGo;
    if (!is_finite(d)) return stop_scalars(S, PBCG_NONFINITE);
    if (is_zero(d)) return stop_scalars(S, PBCG_BREAKDOWN);
    S.alpha = __ddiv_rn(S.rho, d);
}
// omega = (q,y) / (y,y), or the half step x + alpha p when ||q|| meets the
// tolerance. Lanes 1 and 2 divide for the next beta in the same instructions:
// gain = (alpha / rho) (1 / omega), so that beta = gain rho' waits for no
// division when rho' arrives (64^2 on one cluster 9.1 -> 8.5 us an iteration,
// with the shorter sum of the cluster's slots).
__device__ __forceinline__ void omega_scalars(Scalars &S, double qy, double yy, double qq, bool fixed) {
    S.action = kGo;
    const bool small_q = !fixed && norm_below(qq, S.tol, S.bound);
    if (small_q || is_zero(yy)) {
        if (!small_q && !is_zero(qq)) return stop_scalars(S, PBCG_BREAKDOWN);
        S.nr = qq;
        S.action = kHalf;
        return;
    }
    const int lane = threadIdx.x & 31;
    const double f = __ddiv_rn(lane == 0 ? qy : lane == 1 ? yy : S.alpha, lane == 0 ? yy : lane == 1 ? qy : S.rho);
    S.omega = __shfl_sync(kFull, f, 0);
    if (is_zero(S.omega)) return stop_scalars(S, PBCG_BREAKDOWN);
    S.gain = beta_gain(__shfl_sync(kFull, f, 2), __shfl_sync(kFull, f, 1));
}
// Test of r_{i+1}; beta = (alpha / omega) (rho' / rho), by the gain where that
// stayed in range, else by its two quotients on even and odd lanes.
__device__ __forceinline__ void beta_scalars(Scalars &S, double rho_n, double rr, bool finite, bool fixed) {
    S.action = kGo;
    S.nr = rr;
    if (!finite) return stop_scalars(S, PBCG_NONFINITE);
    if (!fixed && norm_below(rr, S.tol, S.bound)) return stop_scalars(S, PBCG_OK);
    if (is_zero(rho_n)) return stop_scalars(S, PBCG_BREAKDOWN);
    if (!is_zero(S.gain)) {
        S.beta = __dmul_rn(S.gain, rho_n);
    } else {
        const bool odd = threadIdx.x & 1;
        const double f = __ddiv_rn(odd ? rho_n : S.alpha, odd ? S.rho : S.omega);
        S.beta = __dmul_rn(__shfl_sync(kFull, f, 0), __shfl_sync(kFull, f, 1));
    }
}
// Algorithm 9: the test and beta, then the denominator of eq. (3),
// r0w + beta (r0s - omega r0z), and alpha_{i+1} = rho' / denominator
__device__ __forceinline__ void beta_alpha_scalars(Scalars &S, double rho_n, double r0w, double rr, bool fixed) {
    beta_scalars(S, rho_n, rr, is_finite(rho_n) && is_finite(r0w) && is_finite(rr), fixed);
    if (S.action != kGo) return;
    const double d = fma(S.beta, S.slope, r0w);
    if (is_zero(d)) return stop_scalars(S, PBCG_BREAKDOWN);
    S.alpha = __ddiv_rn(rho_n, d);
    S.rho = rho_n;
}

// Final true residual ||b - A x|| and the result record (block 0). The
// history holds squared norms during the loop; they become norms here.
template <class Op, int B, class Sync>
__device__ __forceinline__ void finish(const Op &A, const SolveArgs &a, Sync &g, Exchange<B> &X, int lo,
                                       int hi, const Outcome &o, int spmvs) {
    double d[1] = {0.0};
    PBCG_ROWS(i) {
        const double res = a.b[i] - A.row(i, VecLoad{a.x});
        d[0] = fma(res, res, d[0]);
    }
    if (!exchange(g, d, X, [](Scalars &S, const double (&t)[1]) { S.aux = t[0]; })) return;
    if (blockIdx.x == 0) {
        if (a.hist)
            for (int i = 1 + (int)threadIdx.x; i <= o.iters; i += (int)blockDim.x) a.hist[i] = sqrt(a.hist[i]);
        if (threadIdx.x == 0) {
            Control *c = a.ctl;
            const double nt = sqrt(X.s.aux);
            const double nr = o.iters > 0 ? sqrt(o.nr) : o.nr0;
            c->iters = o.iters;
            c->status = o.status;
            c->half_step = o.half;
            c->n_repl = o.nrr;
            c->grid_syncs = g.count;
            c->spmvs = spmvs + 1;
            c->nr0 = o.nr0;
            c->rel_rec = o.nr0 > 0.0 ? nr / o.nr0 : 0.0;
            c->rel_true = o.nr0 > 0.0 ? nt / o.nr0 : nt;
        }
    }
}

// Per-thread accumulation of a dot product over the rows of a sweep. FP64
// vectors: an FMA into a double. FP32 vectors (the inner solves of the
// mixed-precision refinement, CSR and stencil form): compensated FP32
// accumulation, algorithm Dot2 of Ogita, Rump & Oishi ("Accurate sum and dot
// product", SIAM J. Sci. Comput. 26, 2005): each product is split exactly into
// its rounded value and rounding error (TwoProduct by FMA), the running sum is
// updated by the error-free TwoSum and all errors are summed apart; the result
// is as accurate as if accumulated in twice the working precision and is
// converted to double once per thread and sweep, and the threads' values are
// summed in FP64. On this GPU an FP32 operation costs 1/64 of an FP64 one, so
// the inner solves keep FP64-grade dot products (the ones that set alpha,
// beta and omega) without any FP64 instruction per row. Explicit _rn
// intrinsics keep the compiler from fusing the steps of the error-free
// transformations.
template <typename T>
struct DotAcc;
template <>
struct DotAcc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = fma(a, b, s); }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct DotAcc<float> {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float a, float b) {
        const float p = __fmul_rn(a, b);
        const float pe = __fmaf_rn(a, b, -p);   // a b - p, exactly
        const float t = __fadd_rn(s, p);
        const float z = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));   // s + p - t, exactly
        s = t;
        c = __fadd_rn(c, __fadd_rn(e, pe));
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};
// The dot products P of a sweep accumulated one by one in T.
template <class P, typename T>
struct PlainDots {
    DotAcc<T> acc[P::np];
    __device__ __forceinline__ PlainDots(WideSlot *, bool) {}
    __device__ __forceinline__ void add(const T (&v)[P::nv]) {
#pragma unroll
        for (int k = 0; k < P::np; ++k) acc[k].add(v[P::a(k)], v[P::b(k)]);
    }
    __device__ __forceinline__ void values(double (&d)[P::np]) const {
#pragma unroll
        for (int k = 0; k < P::np; ++k) d[k] = acc[k].value();
    }
};
// Accumulator of a sweep: FP64 sweeps of a Wide kernel sum on the integer pipes.
template <bool Wide, class P, typename T, int B>
struct DotsFor {
    using type = PlainDots<P, T>;
};
template <class P, int B>
struct SharedWideDots : WideDots<P> {
    bool any;   // this thread has a row
    __device__ __forceinline__ SharedWideDots(WideSlot *s, bool any_row)
        : WideDots<P>(s + threadIdx.x, B, __ballot_sync(kFull, any_row)), any(any_row) {}
    __device__ __forceinline__ void values(double (&d)[P::np]) const { WideDots<P>::values(any, d); }
};
template <class P, int B>
struct DotsFor<true, P, double, B> {
    using type = SharedWideDots<P, B>;
};
constexpr int kWideSlots = 5;   // dot products of the largest reduction

// Adjacent elements p[i..i+cnt) of a vector (cnt <= G; the rest read as 0) and
// their store. wide: the FP32 sweeps' one 64-bit (G = 2) or 128-bit (G = 4)
// access, where all G elements are present and i is a multiple of G.
template <int G, typename T>
__device__ __forceinline__ void load_group(const T *p, int i, int cnt, bool wide, T (&out)[G]) {
    if constexpr (G == 2) {
        if (wide) {
            const float2 q = *reinterpret_cast<const float2 *>(p + i);
            out[0] = q.x;
            out[1] = q.y;
            return;
        }
    }
    if constexpr (G == 4) {
        if (wide) {
            const float4 q = *reinterpret_cast<const float4 *>(p + i);
            out[0] = q.x;
            out[1] = q.y;
            out[2] = q.z;
            out[3] = q.w;
            return;
        }
    }
#pragma unroll
    for (int u = 0; u < G; ++u) out[u] = u < cnt ? p[i + u] : T(0);
}
// load_group for a fused sweep: through L2 only (ld.global.cg) for operators
// whose sweeps leave L1 to their SpMV's row streams.
template <class Op, int G, typename T>
__device__ __forceinline__ void load_sweep(const T *p, int i, int cnt, bool wide, T (&out)[G]) {
    if constexpr (SweepLoadsL2<Op>::value) {
#pragma unroll
        for (int u = 0; u < G; ++u) out[u] = u < cnt ? __ldcg(p + i + u) : T(0);
    } else {
        load_group(p, i, cnt, wide, out);
    }
}
template <int G, typename T>
__device__ __forceinline__ void store_group(T *p, int i, int cnt, bool wide, const T (&in)[G]) {
    if constexpr (G == 2) {
        if (wide) {
            *reinterpret_cast<float2 *>(p + i) = make_float2(in[0], in[1]);
            return;
        }
    }
    if constexpr (G == 4) {
        if (wide) {
            *reinterpret_cast<float4 *>(p + i) = make_float4(in[0], in[1], in[2], in[3]);
            return;
        }
    }
#pragma unroll
    for (int u = 0; u < G; ++u)
        if (u < cnt) p[i + u] = in[u];
}

// Adjacent rows that a thread takes at a step of the two main sweeps, all
// loaded before any is stored (the stores of one row may alias the loads of
// the next as far as the compiler knows). FP64 sweeps are bound by the FP64
// pipe and take one row; FP32 sweeps take two (CSR) or four of an x-line
// (stencil, StencilOpT::Group) with 64- and 128-bit accesses. Groups are only
// used on a grid, whose rows start at 0.
template <class Op, typename T>
struct RowGroup {
    static constexpr int kRows = sizeof(T) == 8 ? 1 : HasGroups<Op>::value ? 4 : 2;
};
// Groups of the sweep: a group's number takes the place of a row's in PBCG_ROWS.
template <class Op, int G>
__device__ __forceinline__ int group_end(const Op &A, int hi) {
    if constexpr (HasGroups<Op>::value && G == 4) return A.groups();
    else return groups_of(hi, G);
}
// Rows i0 .. i0 + cnt - 1 of group gi, y = A u there and mid = u there (where asked for).
template <bool kMid, class Op, int G, typename T>
__device__ __forceinline__ void group_product(const Op &A, int gi, int hi, const T *u, int &i0, int &cnt, bool &wide,
                                              T (&mid)[G], T (&y)[G]) {
    if constexpr (HasGroups<Op>::value && G == 4) {
        const auto q = A.group(gi);
        i0 = q.r;
        cnt = q.cnt;
        wide = A.aligned != 0;
        A.product4(q, u, mid, y);
    } else {
        i0 = G * gi;
        cnt = G == 1 ? 1 : (hi - i0 < G ? hi - i0 : G);
        wide = G > 1 && cnt == G;
#pragma unroll
        for (int m = 0; m < G; ++m) y[m] = m < cnt ? A.row(i0 + m, VecLoadT<T>{u}) : T(0);
        if constexpr (kMid) load_sweep<Op>(u, i0, cnt, wide, mid);
    }
}

// ===========================================================================
// Algorithm 9 (pipelined BiCGStab) with the residual replacement of
// Section 4.2 (r := b - A x, w := A r before the second reduction of iteration
// i-1; s := A p, z := A s after p_i; for i mod k == 0).
// ===========================================================================
// T is the vector and sweep arithmetic type: double for the FP64 solver,
// float for the inner solves of the mixed-precision refinement. The dot
// products of a thread's rows are summed by DotsFor (FP64 FMAs, compensated
// FP32, or the integers of a Wide kernel) and those of the threads in double;
// alpha, beta, omega, rho are doubles, and a sweep uses them rounded to T.
template <class Op, typename T, int B, class Sync = GridSync, bool Wide = false>
__device__ __forceinline__ bool pipelined_loop(const Op &A, const SolveArgsT<T> &a, Sync &g, Exchange<B> &X,
                                               int lo, int hi, Outcome &o, int &spmvs, WideSlot *wide) {
    const VectorsT<T> &V = a.V;
    T *x = a.x;
    const bool fixed = a.fixed != 0;
    constexpr int kGroup = RowGroup<Op, T>::kRows;

    // r_0 := b - A x_0; shadow r0 := r_0; p, s, z, v := 0 (they are multiplied by beta_{-1} = 0)
    double d0[1];
    {
        DotAcc<T> acc;
        PBCG_ROWS(i) {
            const T ri = a.b[i] - A.row(i, VecLoadT<T>{x});
            V.r[i] = ri;
            V.r0[i] = ri;
            V.p[i] = T(0);
            V.s[i] = T(0);
            V.z[i] = T(0);
            V.v[i] = T(0);
            acc.add(ri, ri);
        }
        d0[0] = acc.value();
    }
    ++spmvs;
    if (!exchange(g, d0, X, [&](Scalars &S, const double (&t)[1]) { start_scalars(S, t[0], a.rtol); })) return false;
    o.nr0 = X.s.nr0;
    o.nr = o.nr0;
    if (threadIdx.x == 0 && a.hist && is_leader(g)) a.hist[0] = o.nr0;
    if (X.s.action == kStop) { o.status = X.s.status; return true; }

    // w_0 := A r_0; alpha_0 := (r0, r0) / (r0, w0)
    {
        DotAcc<T> acc;
        PBCG_ROWS(i) {
            const T wi = A.row(i, VecLoadT<T>{V.r});
            V.w[i] = wi;
            acc.add(V.r0[i], wi);
        }
        d0[0] = acc.value();
    }
    ++spmvs;
    if (!exchange(g, d0, X, [](Scalars &S, const double (&t)[1]) { alpha_scalars(S, t[0]); })) return false;
    if (X.s.action == kStop) { o.status = X.s.status; return true; }

    bool replaced_rw = false;   // r_i, w_i were replaced at the end of iteration i-1
    int it = 0;
    while (it < a.limit) {
        // ---- phase A: t_i = A w_i; p_i, s_i, z_i, q_i, y_i; first reduction
        typename DotsFor<Wide, PairsPipeA, T, B>::type a1(wide, lo + (int)threadIdx.x < hi);   // (q,y) (y,y) (q,q) (r0,s) (r0,z)
        const T al = (T)X.s.alpha, be = (T)X.s.beta, om = (T)X.s.omega;
        if (!replaced_rw) {
            const int end = group_end<Op, kGroup>(A, hi);
            PBCG_STEPS(gi, end) {
                int i0, cnt;
                bool vec;
                T ti[kGroup], ri[kGroup], wi[kGroup], si[kGroup], zi[kGroup], pi[kGroup], vi[kGroup], r0i[kGroup];
                group_product<true>(A, gi, hi, V.w, i0, cnt, vec, wi, ti);
                load_sweep<Op>(V.r, i0, cnt, vec, ri);
                load_sweep<Op>(V.s, i0, cnt, vec, si);
                load_sweep<Op>(V.z, i0, cnt, vec, zi);
                load_sweep<Op>(V.p, i0, cnt, vec, pi);
                load_sweep<Op>(V.v, i0, cnt, vec, vi);
                load_sweep<Op>(V.r0, i0, cnt, vec, r0i);
                T pn[kGroup], sn[kGroup], zn[kGroup], qn[kGroup], yn[kGroup];
#pragma unroll
                for (int u = 0; u < kGroup; ++u) {
                    pn[u] = fmaT(be, fmaT(-om, si[u], pi[u]), ri[u]);   // p_i
                    sn[u] = fmaT(be, fmaT(-om, zi[u], si[u]), wi[u]);   // s_i, eq. (1)
                    zn[u] = fmaT(be, fmaT(-om, vi[u], zi[u]), ti[u]);   // z_i, eq. (6)
                    qn[u] = fmaT(-al, sn[u], ri[u]);                    // q_i
                    yn[u] = fmaT(-al, zn[u], wi[u]);                    // y_i, eq. (4)
                    if (kGroup != 2 || u < cnt) a1.add({qn[u], yn[u], r0i[u], sn[u], zn[u]});
                }
                store_group(V.t, i0, cnt, vec, ti);
                store_group(V.p, i0, cnt, vec, pn);
                store_group(V.s, i0, cnt, vec, sn);
                store_group(V.z, i0, cnt, vec, zn);
                store_group(V.q, i0, cnt, vec, qn);
                store_group(V.y, i0, cnt, vec, yn);
            }
            ++spmvs;
        } else {
            // replacement, second part: t_i = A w_i (w_i replaced), p_i; then s_i := A p_i; z_i := A s_i
            PBCG_ROWS(i) {
                V.t[i] = A.row(i, VecLoadT<T>{V.w});
                V.p[i] = fmaT(be, fmaT(-om, V.s[i], V.p[i]), V.r[i]);
            }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) { V.s[i] = A.row(i, VecLoadT<T>{V.p}); }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const T zn = A.row(i, VecLoadT<T>{V.s});
                const T sn = V.s[i], ri = V.r[i], wi = V.w[i];
                const T qi = fmaT(-al, sn, ri);
                const T yi = fmaT(-al, zn, wi);
                V.z[i] = zn;
                V.q[i] = qi;
                V.y[i] = yi;
                const T r0i = V.r0[i];
                a1.add({qi, yi, r0i, sn, zn});
            }
            spmvs += 3;
        }
        double d1[5];
        a1.values(d1);
        if (!exchange(g, d1, X, [&](Scalars &S, const double (&t)[5]) {
                if (!all_finite(t)) return stop_scalars(S, PBCG_NONFINITE);
                omega_scalars(S, t[0], t[1], t[2], fixed);
                if (S.action == kGo) S.slope = fma(-S.omega, t[4], t[3]);
            }))
            return false;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        if (X.s.action == kHalf) {
            PBCG_ROWS(i) { x[i] = fmaT(al, V.p[i], x[i]); }   // half step x_i + alpha_i p_i
            if (!grid_sync(g, X)) return false;
            ++it;
            o.nr = X.s.nr;
            o.half = 1;
            o.status = PBCG_OK;
            if (threadIdx.x == 0 && a.hist && is_leader(g)) a.hist[it] = X.s.nr;
            break;
        }

        // ---- phase B: v_i = A z_i; x_{i+1}, r_{i+1}, w_{i+1}; second reduction
        const bool replace_now = a.replace_period > 0 && (it + 1) % a.replace_period == 0 &&
                                 (a.max_repl < 0 || o.nrr < a.max_repl);
        typename DotsFor<Wide, PairsPipeB, T, B>::type a2(wide, lo + (int)threadIdx.x < hi);   // (r0,r) (r0,w) (r,r)
        const T om2 = (T)X.s.omega;
        if (!replace_now) {
            const int end = group_end<Op, kGroup>(A, hi);
            PBCG_STEPS(gi, end) {
                int i0, cnt;
                bool vec;
                T vi[kGroup], mid[kGroup], qi[kGroup], yi[kGroup], xi[kGroup], pi[kGroup], ti[kGroup], r0i[kGroup];
                group_product<false>(A, gi, hi, V.z, i0, cnt, vec, mid, vi);
                load_sweep<Op>(V.q, i0, cnt, vec, qi);
                load_sweep<Op>(V.y, i0, cnt, vec, yi);
                load_sweep<Op>(x, i0, cnt, vec, xi);
                load_sweep<Op>(V.p, i0, cnt, vec, pi);
                load_sweep<Op>(V.t, i0, cnt, vec, ti);
                load_sweep<Op>(V.r0, i0, cnt, vec, r0i);
                T xn[kGroup], rn[kGroup], wn[kGroup];
#pragma unroll
                for (int u = 0; u < kGroup; ++u) {
                    xn[u] = fmaT(om2, qi[u], fmaT(al, pi[u], xi[u]));
                    rn[u] = fmaT(-om2, yi[u], qi[u]);                     // eq. (7)
                    wn[u] = fmaT(-om2, fmaT(-al, vi[u], ti[u]), yi[u]);   // eq. (8)
                    if (kGroup != 2 || u < cnt) a2.add({r0i[u], rn[u], wn[u]});
                }
                store_group(x, i0, cnt, vec, xn);
                store_group(V.v, i0, cnt, vec, vi);
                store_group(V.r, i0, cnt, vec, rn);
                store_group(V.w, i0, cnt, vec, wn);
            }
            ++spmvs;
        } else {
            // replacement, first part: x_{i+1}; r_{i+1} := b - A x_{i+1}; w_{i+1} := A r_{i+1}
            PBCG_ROWS(i) { x[i] = fmaT(om2, V.q[i], fmaT(al, V.p[i], x[i])); }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) { V.r[i] = a.b[i] - A.row(i, VecLoadT<T>{x}); }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const T wn = A.row(i, VecLoadT<T>{V.r});
                const T ri = V.r[i], r0i = V.r0[i];
                V.w[i] = wn;
                a2.add({r0i, ri, wn});
            }
            spmvs += 2;
            o.nrr++;
        }
        double d2[3];
        a2.values(d2);
        replaced_rw = replace_now;
        if (!exchange(g, d2, X, [&](Scalars &S, const double (&t)[3]) { beta_alpha_scalars(S, t[0], t[1], t[2], fixed); }))
            return false;
        ++it;
        o.nr = X.s.nr;
        if (threadIdx.x == 0 && a.hist && is_leader(g)) a.hist[it] = X.s.nr;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
    }
    o.iters = it;
    if (it == a.limit && o.status == PBCG_NOT_CONVERGED && fixed) o.status = PBCG_OK;
    return true;
}

// ===========================================================================
// Algorithm 11 (preconditioned pipelined BiCGStab) with a diagonal M^{-1},
// applied elementwise inside the sweeps, so an iteration still takes two
// grid-wide exchanges. The hat vectors of Algorithm 11 are M^{-1} times their
// plain counterparts (r^ = M^{-1} r, s^ = M^{-1} s, q^ = M^{-1} q, z^, w^);
// the algorithm carries r^, s^, q^ as recurrences because applying a general
// M^{-1} costs a solve. With a diagonal M^{-1} it costs one product, so this
// loop forms r^, s^, q^ where they are used (m_i r_i, m_i s_i, m_i q_i) and
// stores only the hat vectors an SpMV reads: z^ (v = A z^) and w^ (t = A w^),
// plus p^ (V.p). That removes the r^, s^, q^ recurrences and their 48 bytes
// per unknown and iteration of traffic; in exact arithmetic the iterates are
// Algorithm 11's. Residual replacement (Section 4.2): r := b - A x and
// w := A r^ before the second reduction of iteration i-1; s := A p^ and
// z := A s^ after p^_i; r^ and s^ are then stored as SpMV inputs (rh, sh).
// ===========================================================================
template <class Op, int B, bool Wide>
__device__ __forceinline__ bool pipelined_prec_loop(const Op &A, const SolveArgs &a, GridSync &g, Exchange<B> &X,
                                                    int lo, int hi, Outcome &o, int &spmvs, WideSlot *wide) {
    const Vectors &V = a.V;
    double *x = a.x;
    const double *mi = a.minv;
    double *rh = a.rh, *sh = a.sh, *zh = a.zh, *wh = a.wh;
    const bool fixed = a.fixed != 0;

    // r_0 := b - A x_0; r0 := r_0; r^_0 := M^{-1} r_0 (an SpMV input); p^, s, z, v := 0
    double d0[1] = {0.0};
    PBCG_ROWS(i) {
        const double ri = a.b[i] - A.row(i, VecLoad{x});
        V.r[i] = ri;
        V.r0[i] = ri;
        rh[i] = mi[i] * ri;
        V.p[i] = 0.0;
        V.s[i] = 0.0;
        V.z[i] = 0.0;
        V.v[i] = 0.0;
        d0[0] = fma(ri, ri, d0[0]);
    }
    ++spmvs;
    if (!exchange(g, d0, X, [&](Scalars &S, const double (&t)[1]) { start_scalars(S, t[0], a.rtol); })) return false;
    o.nr0 = X.s.nr0;
    o.nr = o.nr0;
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[0] = o.nr0;
    if (X.s.action == kStop) { o.status = X.s.status; return true; }

    // w_0 := A r^_0; w^_0 := M^{-1} w_0; alpha_0 := (r0, r0) / (r0, w0)
    d0[0] = 0.0;
    PBCG_ROWS(i) {
        const double wi = A.row(i, VecLoad{rh});
        V.w[i] = wi;
        wh[i] = mi[i] * wi;
        d0[0] = fma(V.r0[i], wi, d0[0]);
    }
    ++spmvs;
    if (!exchange(g, d0, X, [](Scalars &S, const double (&t)[1]) { alpha_scalars(S, t[0]); })) return false;
    if (X.s.action == kStop) { o.status = X.s.status; return true; }

    bool replaced = false;
    int it = 0;
    while (it < a.limit) {
        const double alpha = X.s.alpha, beta = X.s.beta, om1 = X.s.omega;
        // ---- phase A: t = A w^; p^, s, z, z^, q, y; first reduction
        typename DotsFor<Wide, PairsPipeA, double, B>::type a1(wide, lo + (int)threadIdx.x < hi);   // (q,y) (y,y) (q,q) (r0,s) (r0,z)
        if (!replaced) {
            PBCG_ROWS(i) {
                const double ti = A.row(i, VecLoad{wh});
                const double m = mi[i], ri = V.r[i], si = V.s[i], zi = V.z[i], wi = V.w[i];
                const double ph = fma(beta, fma(-om1, m * si, V.p[i]), m * ri);   // p^_i = r^_i + beta (p^ - omega s^)
                const double sn = fma(beta, fma(-om1, zi, si), wi);               // s_i
                const double zn = fma(beta, fma(-om1, V.v[i], zi), ti);           // z_i
                const double qi = fma(-alpha, sn, ri);                              // q_i
                const double yi = fma(-alpha, zn, wi);                              // y_i
                V.t[i] = ti;
                V.p[i] = ph;
                V.s[i] = sn;
                V.z[i] = zn;
                zh[i] = m * zn;                                                     // z^_i
                V.q[i] = qi;
                V.y[i] = yi;
                const double r0i = V.r0[i];
                a1.add({qi, yi, r0i, sn, zn});
            }
            ++spmvs;
        } else {
            // replacement, second part: t = A w^ (w^ replaced), p^; then s := A p^, s^ := M^{-1} s, z := A s^
            PBCG_ROWS(i) {
                const double m = mi[i];
                V.t[i] = A.row(i, VecLoad{wh});
                V.p[i] = fma(beta, fma(-om1, m * V.s[i], V.p[i]), m * V.r[i]);   // r^ = M^{-1} r replaced
            }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const double sn = A.row(i, VecLoad{V.p});
                V.s[i] = sn;
                sh[i] = mi[i] * sn;
            }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const double zn = A.row(i, VecLoad{sh});
                const double sn = V.s[i];
                const double qi = fma(-alpha, sn, V.r[i]);
                const double yi = fma(-alpha, zn, V.w[i]);
                V.z[i] = zn;
                zh[i] = mi[i] * zn;
                V.q[i] = qi;
                V.y[i] = yi;
                const double r0i = V.r0[i];
                a1.add({qi, yi, r0i, sn, zn});
            }
            spmvs += 3;
        }
        double d1[5];
        a1.values(d1);
        if (!exchange(g, d1, X, [&](Scalars &S, const double (&t)[5]) {
                if (!all_finite(t)) return stop_scalars(S, PBCG_NONFINITE);
                omega_scalars(S, t[0], t[1], t[2], fixed);
                if (S.action == kGo) S.slope = fma(-S.omega, t[4], t[3]);
            }))
            return false;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        if (X.s.action == kHalf) {
            PBCG_ROWS(i) { x[i] = fma(alpha, V.p[i], x[i]); }   // half step x_i + alpha_i p^_i
            if (!grid_sync(g, X)) return false;
            ++it;
            o.nr = X.s.nr;
            o.half = 1;
            o.status = PBCG_OK;
            if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[it] = X.s.nr;
            break;
        }

        // ---- phase B: v = A z^; x, r, w, w^; second reduction
        const double omega = X.s.omega;
        const bool replace_now = a.replace_period > 0 && (it + 1) % a.replace_period == 0 &&
                                 (a.max_repl < 0 || o.nrr < a.max_repl);
        typename DotsFor<Wide, PairsPipeB, double, B>::type a2(wide, lo + (int)threadIdx.x < hi);   // (r0,r) (r0,w) (r,r)
        if (!replace_now) {
            PBCG_ROWS(i) {
                const double vi = A.row(i, VecLoad{zh});
                const double m = mi[i], qi = V.q[i], yi = V.y[i];
                x[i] = fma(omega, m * qi, fma(alpha, V.p[i], x[i]));   // x + alpha p^ + omega q^
                const double rn = fma(-omega, yi, qi);
                const double wn = fma(-omega, fma(-alpha, vi, V.t[i]), yi);
                V.v[i] = vi;
                V.r[i] = rn;
                V.w[i] = wn;
                wh[i] = m * wn;                                         // w^_{i+1}
                const double r0i = V.r0[i];
                a2.add({r0i, rn, wn});
            }
            ++spmvs;
        } else {
            PBCG_ROWS(i) { x[i] = fma(omega, mi[i] * V.q[i], fma(alpha, V.p[i], x[i])); }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const double rn = a.b[i] - A.row(i, VecLoad{x});
                V.r[i] = rn;
                rh[i] = mi[i] * rn;
            }
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const double wn = A.row(i, VecLoad{rh});
                const double rn = V.r[i], r0i = V.r0[i];
                V.w[i] = wn;
                wh[i] = mi[i] * wn;
                a2.add({r0i, rn, wn});
            }
            spmvs += 2;
            o.nrr++;
        }
        replaced = replace_now;
        double d2[3];
        a2.values(d2);
        if (!exchange(g, d2, X, [&](Scalars &S, const double (&t)[3]) { beta_alpha_scalars(S, t[0], t[1], t[2], fixed); }))
            return false;
        ++it;
        o.nr = X.s.nr;
        if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[it] = X.s.nr;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
    }
    o.iters = it;
    if (it == a.limit && o.status == PBCG_NOT_CONVERGED && fixed) o.status = PBCG_OK;
    return true;
}

template <class Op, bool Prec, bool Wide>
__global__ void __launch_bounds__(SolverBlock<Wide>::kThreads, 1024 / SolverBlock<Wide>::kThreads)
    pbicgstab_kernel(const Op A, const SolveArgs a) {
    constexpr int B = SolverBlock<Wide>::kThreads;
    __shared__ Exchange<B> X;
    __shared__ WideSlot wide[Wide ? kWideSlots * B : 1];
    if (threadIdx.x == 0) X.ok = 1;   // read only after the first exchange's barrier
    GridSync g{a.ctl, a.partials, 0u, 0, (int)(gridDim.x * blockDim.x)};   // partials: the exchange slots
    const int lo = grid_lo(), hi = a.n;
    Outcome o{0, PBCG_NOT_CONVERGED, 0, 0, 0.0, 0.0};
    int spmvs = 0;
    bool ok;
    if constexpr (Prec)
        ok = pipelined_prec_loop<Op, B, Wide>(A, a, g, X, lo, hi, o, spmvs, wide);
    else
        ok = pipelined_loop<Op, double, B, GridSync, Wide>(A, a, g, X, lo, hi, o, spmvs, wide);
    if (!ok) return;
    finish(A, a, g, X, lo, hi, o, spmvs);
}

// ===========================================================================
// Algorithm 7 (standard BiCGStab). p and s use two buffers each in variant 3:
// the phase that forms p_i for its SpMV reads p_{i-1}, s_{i-1} of neighbours
// while writing p_i, s_i, so the old and new values must not share storage.
// ===========================================================================
template <class Op, int B, class Sync = GridSync, bool Wide = false>
__device__ __forceinline__ bool standard_loop(const Op &A, const SolveArgs &a, Sync &g, Exchange<B> &X,
                                              int lo, int hi, Outcome &o, int &spmvs, WideSlot *wide) {
    const Vectors &V = a.V;
    double *x = a.x;
    const bool fixed = a.fixed != 0;
    const bool v3 = !Wide && a.variant == 3;   // the wide kernel holds variant 5 alone
    // buffers: variant 3 ping-pongs p between V.p / V.z and s between V.s / V.w
    double *pA = V.p, *pB = V.z, *sA = V.s, *sB = V.w;

    // r_0 := b - A x_0; shadow r0 := r_0; p_0 := r_0 (as r + 0 (0 - 0 s))
    double d0[1] = {0.0};
    PBCG_ROWS(i) {
        const double ri = a.b[i] - A.row(i, VecLoad{x});
        V.r[i] = ri;
        V.r0[i] = ri;
        pA[i] = 0.0;
        sA[i] = 0.0;
        d0[0] = fma(ri, ri, d0[0]);
    }
    ++spmvs;
    if (!exchange(g, d0, X, [&](Scalars &S, const double (&t)[1]) { start_scalars(S, t[0], a.rtol); })) return false;
    o.nr0 = X.s.nr0;
    o.nr = o.nr0;
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[0] = o.nr0;
    if (X.s.action == kStop) { o.status = X.s.status; return true; }

    int it = 0;
    while (it < a.limit) {
        const double beta = X.s.beta, om1 = X.s.omega;
        // ---- s_i = A p_i, alpha_i = (r0, r_i) / (r0, s_i)
        typename DotsFor<Wide, PairsOne, double, B>::type a1(wide, lo + (int)threadIdx.x < hi);   // (r0,s)
        if (v3) {
            const PLoad pl{V.r, pA, sA, beta, om1};
            PBCG_ROWS(i) {
                const double si = A.row(i, pl);
                pB[i] = pl(i);
                sB[i] = si;
                a1.add({V.r0[i], si});
            }
        } else {
            sweep_pairs(g, lo, hi, [&](int i) { return Row3{sA[i], pA[i], V.r[i]}; },
                        [&](int i, const Row3 &v) { pA[i] = fma(beta, fma(-om1, v.a, v.b), v.c); });
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const double si = A.row(i, VecLoad{pA});
                sA[i] = si;
                a1.add({V.r0[i], si});
            }
        }
        ++spmvs;
        double *pc = v3 ? pB : pA, *sc = v3 ? sB : sA;   // p_i, s_i
        double d1[1];
        a1.values(d1);
        if (!exchange(g, d1, X, [](Scalars &S, const double (&t)[1]) { alpha_scalars(S, t[0]); })) return false;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        const double alpha = X.s.alpha;

        // ---- q_i = r_i - alpha s_i; y_i = A q_i; omega_i
        typename DotsFor<Wide, PairsOmega, double, B>::type a2(wide, lo + (int)threadIdx.x < hi);   // (q,y) (y,y) (q,q)
        if (v3) {
            const QLoad ql{V.r, sc, alpha};
            PBCG_ROWS(i) {
                const double yi = A.row(i, ql);
                const double qi = ql(i);
                V.q[i] = qi;
                V.y[i] = yi;
                a2.add({qi, yi});
            }
        } else {
            sweep_pairs(g, lo, hi, [&](int i) { return Row2{sc[i], V.r[i]}; },
                        [&](int i, const Row2 &v) { V.q[i] = fma(-alpha, v.a, v.b); });
            if (!grid_sync(g, X)) return false;
            PBCG_ROWS(i) {
                const double yi = A.row(i, VecLoad{V.q});
                const double qi = V.q[i];
                V.y[i] = yi;
                a2.add({qi, yi});
            }
        }
        ++spmvs;
        double d2[3];
        a2.values(d2);
        if (!exchange(g, d2, X, [&](Scalars &S, const double (&t)[3]) {
                if (!all_finite(t)) return stop_scalars(S, PBCG_NONFINITE);
                omega_scalars(S, t[0], t[1], t[2], fixed);
            }))
            return false;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        if (X.s.action == kHalf) {
            PBCG_ROWS(i) { x[i] = fma(alpha, pc[i], x[i]); }
            if (!grid_sync(g, X)) return false;
            ++it;
            o.nr = X.s.nr;
            o.half = 1;
            o.status = PBCG_OK;
            if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[it] = X.s.nr;
            break;
        }
        const double omega = X.s.omega;

        // ---- x_{i+1}, r_{i+1}; beta_i
        typename DotsFor<Wide, PairsRho, double, B>::type a3(wide, lo + (int)threadIdx.x < hi);   // (r0,r) (r,r)
        sweep_pairs(g, lo, hi, [&](int i) { return Row5{V.q[i], pc[i], x[i], V.y[i], V.r0[i]}; },
                    [&](int i, const Row5 &v) {
                        x[i] = fma(omega, v.a, fma(alpha, v.b, v.c));
                        const double rn = fma(-omega, v.d, v.a);
                        V.r[i] = rn;
                        a3.add({v.e, rn});
                      });
        double d3[2];
        a3.values(d3);
        if (!exchange(g, d3, X, [&](Scalars &S, const double (&t)[2]) {
                beta_scalars(S, t[0], t[1], all_finite(t), fixed);
                S.rho = t[0];
            }))
            return false;
        ++it;
        o.nr = X.s.nr;
        if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[it] = X.s.nr;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        if (v3) {
            double *tp = pA; pA = pB; pB = tp;
            double *ts = sA; sA = sB; sB = ts;
        }
    }
    o.iters = it;
    if (it == a.limit && o.status == PBCG_NOT_CONVERGED && fixed) o.status = PBCG_OK;
    return true;
}

// ===========================================================================
// Algorithm 10 (preconditioned BiCGStab) with a diagonal M^{-1}: the
// five-exchange form of the standard loop with p^ = M^{-1} p and
// q^ = M^{-1} q written next to p and q. Buffers: V.z holds p^, a.qh holds q^.
// ===========================================================================
template <class Op, int B, bool Wide>
__device__ __forceinline__ bool standard_prec_loop(const Op &A, const SolveArgs &a, GridSync &g, Exchange<B> &X,
                                                   int lo, int hi, Outcome &o, int &spmvs, WideSlot *wide) {
    const Vectors &V = a.V;
    double *x = a.x;
    const double *mi = a.minv;
    double *ph = V.z, *qh = a.qh;
    const bool fixed = a.fixed != 0;

    double d0[1] = {0.0};
    PBCG_ROWS(i) {
        const double ri = a.b[i] - A.row(i, VecLoad{x});
        V.r[i] = ri;
        V.r0[i] = ri;
        V.p[i] = 0.0;
        V.s[i] = 0.0;
        d0[0] = fma(ri, ri, d0[0]);
    }
    ++spmvs;
    if (!exchange(g, d0, X, [&](Scalars &S, const double (&t)[1]) { start_scalars(S, t[0], a.rtol); })) return false;
    o.nr0 = X.s.nr0;
    o.nr = o.nr0;
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[0] = o.nr0;
    if (X.s.action == kStop) { o.status = X.s.status; return true; }

    int it = 0;
    while (it < a.limit) {
        const double beta = X.s.beta, om1 = X.s.omega;
        // p_i := r_i + beta (p_{i-1} - omega s_{i-1}); p^_i := M^{-1} p_i; s_i := A p^_i
        sweep_pairs(g, lo, hi, [&](int i) { return Row4{V.s[i], V.p[i], V.r[i], mi[i]}; },
                    [&](int i, const Row4 &v) {
                        const double pn = fma(beta, fma(-om1, v.a, v.b), v.c);
                        V.p[i] = pn;
                        ph[i] = v.d * pn;
                    });
        if (!grid_sync(g, X)) return false;
        typename DotsFor<Wide, PairsOne, double, B>::type a1(wide, lo + (int)threadIdx.x < hi);   // (r0,s)
        PBCG_ROWS(i) {
            const double si = A.row(i, VecLoad{ph});
            V.s[i] = si;
            a1.add({V.r0[i], si});
        }
        ++spmvs;
        double d1[1];
        a1.values(d1);
        if (!exchange(g, d1, X, [](Scalars &S, const double (&t)[1]) { alpha_scalars(S, t[0]); })) return false;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        const double alpha = X.s.alpha;
        // q_i := r_i - alpha s_i; q^_i := M^{-1} q_i; y_i := A q^_i
        sweep_pairs(g, lo, hi, [&](int i) { return Row3{V.s[i], V.r[i], mi[i]}; },
                    [&](int i, const Row3 &v) {
                        const double qi = fma(-alpha, v.a, v.b);
                        V.q[i] = qi;
                        qh[i] = v.c * qi;
                    });
        if (!grid_sync(g, X)) return false;
        typename DotsFor<Wide, PairsOmega, double, B>::type a2(wide, lo + (int)threadIdx.x < hi);   // (q,y) (y,y) (q,q)
        PBCG_ROWS(i) {
            const double yi = A.row(i, VecLoad{qh});
            const double qi = V.q[i];
            V.y[i] = yi;
            a2.add({qi, yi});
        }
        ++spmvs;
        double d2[3];
        a2.values(d2);
        if (!exchange(g, d2, X, [&](Scalars &S, const double (&t)[3]) {
                if (!all_finite(t)) return stop_scalars(S, PBCG_NONFINITE);
                omega_scalars(S, t[0], t[1], t[2], fixed);
            }))
            return false;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
        if (X.s.action == kHalf) {
            PBCG_ROWS(i) { x[i] = fma(alpha, ph[i], x[i]); }
            if (!grid_sync(g, X)) return false;
            ++it;
            o.nr = X.s.nr;
            o.half = 1;
            o.status = PBCG_OK;
            if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[it] = X.s.nr;
            break;
        }
        const double omega = X.s.omega;
        // x_{i+1} := x_i + alpha p^_i + omega q^_i; r_{i+1} := q_i - omega y_i
        typename DotsFor<Wide, PairsRho, double, B>::type a3(wide, lo + (int)threadIdx.x < hi);   // (r0,r) (r,r)
        sweep_pairs(g, lo, hi, [&](int i) { return Row6{qh[i], ph[i], x[i], V.y[i], V.q[i], V.r0[i]}; },
                    [&](int i, const Row6 &v) {
                        x[i] = fma(omega, v.a, fma(alpha, v.b, v.c));
                        const double rn = fma(-omega, v.d, v.e);
                        V.r[i] = rn;
                        a3.add({v.f, rn});
                      });
        double d3[2];
        a3.values(d3);
        if (!exchange(g, d3, X, [&](Scalars &S, const double (&t)[2]) {
                beta_scalars(S, t[0], t[1], all_finite(t), fixed);
                S.rho = t[0];
            }))
            return false;
        ++it;
        o.nr = X.s.nr;
        if (blockIdx.x == 0 && threadIdx.x == 0 && a.hist) a.hist[it] = X.s.nr;
        if (X.s.action == kStop) { o.status = X.s.status; break; }
    }
    o.iters = it;
    if (it == a.limit && o.status == PBCG_NOT_CONVERGED && fixed) o.status = PBCG_OK;
    return true;
}

template <class Op, bool Prec, bool Wide>
__global__ void __launch_bounds__(SolverBlock<Wide>::kThreads, 1024 / SolverBlock<Wide>::kThreads)
    bicgstab_kernel(const Op A, const SolveArgs a) {
    constexpr int B = SolverBlock<Wide>::kThreads;
    __shared__ Exchange<B> X;
    __shared__ WideSlot wide[Wide ? kWideSlots * B : 1];
    if (threadIdx.x == 0) X.ok = 1;   // read only after the first exchange's barrier
    GridSync g{a.ctl, a.partials, 0u, 0, (int)(gridDim.x * blockDim.x)};   // partials: the exchange slots
    const int lo = grid_lo(), hi = a.n;
    Outcome o{0, PBCG_NOT_CONVERGED, 0, 0, 0.0, 0.0};
    int spmvs = 0;
    bool ok;
    if constexpr (Prec)
        ok = standard_prec_loop<Op, B, Wide>(A, a, g, X, lo, hi, o, spmvs, wide);
    else
        ok = standard_loop<Op, B, GridSync, Wide>(A, a, g, X, lo, hi, o, spmvs, wide);
    if (!ok) return;
    finish(A, a, g, X, lo, hi, o, spmvs);
}

// ===========================================================================
// Mixed precision: FP64 iterative refinement around an FP32 pipelined solve.
// Each refinement step computes the true residual r = b - A x with the FP64
// matrix and FP64 vectors, rounds it to float, solves A d = r with Algorithm 9
// on float vectors and the low-precision copy of A (FP32 or BF16 values; dot
// products summed per thread in compensated FP32 and across threads in FP64),
// and adds d to x in FP64. The inner solve runs without residual replacement:
// the FP64 residual of every refinement step plays that role.
//
// Refinement contracts only while the low-precision operator is close enough
// to A (roughly cond(A) times the value rounding below 1). So the loop also
// stops when `stall_steps` steps in a row fail to bring the FP64 residual
// below the best one so far, and returns the best iterate with
// PBCG_NOT_CONVERGED. A converging refinement can have an occasional step
// without progress: an inner solve capped at inner_maxit may end on one of
// BiCGStab's residual peaks. The best iterate is kept without an extra sweep: the
// sweep that adds d to x first saves x in `xbest` when x is the best so far,
// i.e. exactly when the loop is about to move away from it.
// ===========================================================================
// Default of stall_steps. Measured on the 192^3 convection-diffusion system
// (40 FP32 refinements to 1e-10: both forms, inner tolerance and cap 0.1/50
// and 0.03/150, five grids, two roundings of b): runs of up to 4 steps
// without a new best occur in converging refinements, so 6.
constexpr int kMixedStallSteps = 6;

struct MixedArgs {
    int n;
    const double *b;
    double *x;
    double *xbest;       // FP64 copy of the best iterate, written when the loop leaves it
    float *d;            // correction of the current step (inner solution)
    float *rhs;          // residual of the current step, rounded to float
    VectorsT<float> V;   // inner work vectors
    Control *ctl;
    double *partials;
    double *hist;        // nullable: true residual norm before each step, length max_outer + 1
    double *inner_hist;  // nullable: recursive residual norms of the first step's inner solve
    double rtol;
    int max_outer;
    double inner_rtol;
    int inner_maxit;
    int inner_fixed;     // > 0: every inner solve runs exactly this many iterations
    int dealt;           // CSR: rows in runs of 32 to all blocks in turn (grid_lo)
    int stall_steps;     // steps in a row without a new best residual that stop the loop
};

// Most threads per block of the mixed kernel (64 registers at 1024 threads per
// SM). The 4-row groups spill there, and are faster than with 80 or 127
// registers at fewer threads: 192^3, 167 us an inner iteration against 185 and
// 217 (174 in blocks of 512).
constexpr int kMixedTPB = 256;
template <class Op64, class Op32>
__global__ void __launch_bounds__(kMixedTPB, 4)
    mixed_kernel(const Op64 A, const Op32 A32, const MixedArgs m) {
    __shared__ Exchange<kMixedTPB> X;
    if (threadIdx.x == 0) X.ok = 1;   // read only after the first exchange's barrier
    GridSync g{m.ctl, m.partials, 0u, 0, (int)(gridDim.x * blockDim.x)};
    const int lo = HasGroups<Op32>::value || m.dealt ? grid_lo() : (int)(blockIdx.x * blockDim.x), hi = m.n;
    int outer = 0, inner_total = 0, status = PBCG_NOT_CONVERGED, spmvs = 0, stalls = 0;
    double nr0 = 0.0, tol = 0.0, bound = 0.0, last = 0.0;
    double best = 0.0;        // smallest squared FP64 residual so far (valid when have_best)
    bool have_best = false;
    bool at_best = false;     // x is the best iterate so far
    for (;;) {
        if (outer > 0) {
            const bool save = at_best;   // the same in every block
            PBCG_ROWS(i) {
                const double xi = m.x[i];
                if (save) m.xbest[i] = xi;
                m.x[i] = xi + (double)m.d[i];
            }
            if (!grid_sync(g, X)) return;
        }
        double d[1] = {0.0};
        PBCG_ROWS(i) {
            const double r = m.b[i] - A.row(i, VecLoad{m.x});
            m.rhs[i] = (float)r;
            m.d[i] = 0.0f;
            d[0] = fma(r, r, d[0]);
        }
        ++spmvs;
        if (!exchange(g, d, X, [](Scalars &S, const double (&t)[1]) { S.aux = t[0]; })) return;
        d[0] = X.s.aux;
        last = d[0];
        if (outer == 0) {
            nr0 = sqrt(d[0]);
            tol = __dmul_rn(m.rtol, nr0);
            bound = norm_bound(tol);
        }
        if (blockIdx.x == 0 && threadIdx.x == 0 && m.hist) m.hist[outer] = d[0];
        if (!isfinite(d[0])) { at_best = false; status = PBCG_NONFINITE; break; }
        if (nr0 == 0.0 || norm_below(d[0], tol, bound)) { at_best = true; status = PBCG_OK; break; }
        if (!have_best || d[0] < best) {
            best = d[0];
            have_best = true;
            at_best = true;
            stalls = 0;
        } else {
            at_best = false;
            if (++stalls >= m.stall_steps) break;   // refinement does not contract
        }
        if (outer >= m.max_outer) break;
        SolveArgsT<float> ia;
        ia.n = m.n;
        ia.b = m.rhs;
        ia.x = m.d;
        ia.V = m.V;
        ia.ctl = m.ctl;
        ia.partials = m.partials;
        ia.hist = outer == 0 ? m.inner_hist : nullptr;
        ia.rtol = m.inner_rtol;
        ia.limit = m.inner_fixed > 0 ? m.inner_fixed : m.inner_maxit;
        ia.fixed = m.inner_fixed > 0 ? 1 : 0;
        ia.replace_period = 0;
        ia.max_repl = -1;
        ia.variant = 0;
        Outcome io{0, PBCG_NOT_CONVERGED, 0, 0, 0.0, 0.0};
        if (!pipelined_loop<Op32, float, kMixedTPB>(A32, ia, g, X, lo, hi, io, spmvs, nullptr))
            return;
        // the inner history holds squared norms after entry 0 (thread 0 of block 0 wrote them)
        if (blockIdx.x == 0 && threadIdx.x == 0 && ia.hist)
            for (int i = 1; i <= io.iters; ++i) ia.hist[i] = sqrt(ia.hist[i]);
        inner_total += io.iters;
        ++outer;
        if (io.status == PBCG_NONFINITE) { status = PBCG_NONFINITE; break; }
    }
    // A solve that stops unconverged returns the best iterate: x := xbest when x is not it.
    const bool restore = status != PBCG_OK && have_best && !at_best;
    if (restore) {
        PBCG_ROWS(i) { m.x[i] = m.xbest[i]; }
        last = best;
    }
    if (blockIdx.x == 0) {
        if (m.hist)
            for (int i = (int)threadIdx.x; i <= outer; i += (int)blockDim.x) m.hist[i] = sqrt(m.hist[i]);
        if (threadIdx.x == 0) {
            Control *c = m.ctl;
            c->iters = outer;
            c->inner_iters = inner_total;
            c->status = status;
            c->grid_syncs = g.count;
            c->spmvs = spmvs;
            c->nr0 = nr0;
            c->rel_true = nr0 > 0.0 ? sqrt(last) / nr0 : sqrt(last);
            c->rel_rec = c->rel_true;
            c->half_step = restore ? 1 : 0;   // mixed solves: 1 if x was reset to the best iterate
        }
    }
}

// ===========================================================================
// Single small systems on one thread-block cluster. A cooperative grid pays a
// round trip through L2 and an arrival counter per exchange (several us at a
// few thousand unknowns); the CTAs of one cluster instead cross the hardware
// cluster barrier and exchange their block sums through distributed shared
// memory (ClusterSync). The solver loops are the same code as on the grid.
// Rows are split into `size` contiguous ranges, one per CTA; CTA rank 0
// writes the result record. Every CTA takes the same branches (identical
// scalars), so all of them execute the same sequence of cluster barriers.
// ===========================================================================
template <class Op, bool Pipelined>
__global__ void __launch_bounds__(kTPB, 1) cluster_solve_kernel(const Op A, const SolveArgs a) {
    __shared__ Exchange<kTPB> X;
    __shared__ double slots[2][kMaxCluster][kSlotDoubles];   // cluster reductions: every CTA's block sums
    const unsigned size = cluster_ctas(), rank = cluster_rank();
    if (threadIdx.x == 0) X.ok = 1;
    cluster_barrier();   // every CTA started before its shared memory is written by the others
    ClusterSync g{slots, rank, size, 0u, 0};
    const int lo = (int)((long long)rank * a.n / size);
    const int hi = (int)((long long)(rank + 1) * a.n / size);
    Outcome o{0, PBCG_NOT_CONVERGED, 0, 0, 0.0, 0.0};
    int spmvs = 0;
    if constexpr (Pipelined)
        pipelined_loop<Op, double, kTPB, ClusterSync>(A, a, g, X, lo, hi, o, spmvs, nullptr);
    else
        standard_loop<Op, kTPB, ClusterSync>(A, a, g, X, lo, hi, o, spmvs, nullptr);
    finish(A, a, g, X, lo, hi, o, spmvs);
    cluster_barrier();   // no CTA leaves while another may still address its shared memory
}

// ===========================================================================
// The same with everything on the chip: CTA `rank` owns rows [rank m, rank m +
// m) and keeps their vectors and their matrix entries in its shared memory. An
// entry holds its value and the shared-memory address, in the window of the
// CTA that owns its column, of that column's slot in the first vector; the
// slot in another vector is a constant away. So a product with A reads
// neighbours' values through distributed shared memory, and an iteration
// touches neither L1 nor L2, whose round trips (row pointers, then entries,
// then vector elements) took a quarter of it: 64^2 11.6 -> 9.1 us an iteration
// of Algorithm 9, 17x15x13 14.1 -> 9.5 of Algorithm 7; what is left is the
// FP64 latency of the sums and scalars. The loops are the same code: their
// vectors are addressed as before, by generic pointers offset to the CTA's
// first row.
// ===========================================================================
constexpr int kOnChipTPB = 256;
constexpr int kOnChipVecs = 11;            // r r0 p s z q y w t v x
constexpr size_t kOnChipMaxBytes = 200 * 1024;
__host__ __device__ inline size_t onchip_bytes(int m, int cap) {
    return (size_t)m * (kOnChipVecs * sizeof(double) + sizeof(int2)) + (size_t)cap * (sizeof(double) + sizeof(uint32_t));
}

struct OnChipOp {
    int n, lo, m;
    FastDiv dm;                // by m: the owner of a column
    uint32_t pool;             // shared address of the first vector
    const int2 *range;         // entries of each own row
    const double *val;
    const uint32_t *addr;      // null: the entries did not fit, taken from col and val in global memory
    const int *col;

    __device__ __forceinline__ uint32_t address(int c) const {
        const uint32_t owner = dm.div((uint32_t)c);
        uint32_t a;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(pool), "r"(owner));
        return a + (uint32_t)(c - (int)owner * m) * 8u;
    }
    // Distance of vector p (as the loops address it) from the first one.
    __device__ __forceinline__ uint32_t apart(const double *p) const {
        return (uint32_t)__cvta_generic_to_shared(p + lo) - pool;
    }
    __device__ __forceinline__ static double peek(uint32_t a) {
        double v;
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
        return v;
    }
    __device__ __forceinline__ double value(const VecLoad &u, uint32_t a) const { return peek(a + apart(u.x)); }
    __device__ __forceinline__ double value(const PLoad &u, uint32_t a) const {
        return fma(u.beta, fma(-u.omega, peek(a + apart(u.s)), peek(a + apart(u.p))), peek(a + apart(u.r)));
    }
    __device__ __forceinline__ double value(const QLoad &u, uint32_t a) const {
        return fma(-u.alpha, peek(a + apart(u.s)), peek(a + apart(u.r)));
    }

    template <class L>
    __device__ __forceinline__ double row(int i, const L &u) const {
        constexpr int kC = 8;
        const int2 q = range[i - lo];
        double acc = 0.0;
        for (int k0 = q.x; k0 < q.y; k0 += kC) {
            double v[kC], x[kC];
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                v[j] = x[j] = 0.0;
                if (k0 + j < q.y) {
                    v[j] = val[k0 + j];
                    x[j] = value(u, addr ? addr[k0 + j] : address(PBCG_SAFE(col[k0 + j], n)));
                }
            }
#pragma unroll
            for (int j = 0; j < kC; ++j) {
                if (k0 + j >= q.y) break;
                acc = fma(v[j], x[j], acc);
            }
        }
        return acc;
    }
};

// The CTA's entries into shared memory.
template <int kChunk>
__device__ __forceinline__ void onchip_entries(const CsrOpT<double, kChunk> &A, OnChipOp &op, int hi, int cap, int2 *range,
                                               double *val, uint32_t *addr) {
    const int base = hi > op.lo ? A.rowptr[op.lo] : 0, count = hi > op.lo ? A.rowptr[hi] - base : 0;
    const bool fits = count <= cap;
    for (int i = op.lo + (int)threadIdx.x; i < hi; i += (int)blockDim.x) {
        const int b = A.rowptr[i], e = A.rowptr[i + 1];
        range[i - op.lo] = fits ? make_int2(b - base, e - base) : make_int2(b, e);
    }
    if (fits)
        for (int k = (int)threadIdx.x; k < count; k += (int)blockDim.x) {
            val[k] = A.val[base + k];
            addr[k] = op.address(PBCG_SAFE(A.col[base + k], op.n));
        }
    op.val = fits ? val : A.val;
    op.addr = fits ? addr : nullptr;
    op.col = A.col;
}
__device__ __forceinline__ void onchip_entries(const StencilOp &A, OnChipOp &op, int hi, int, int2 *range, double *val,
                                               uint32_t *addr) {
    const int per = A.nz == 1 ? 5 : 7;   // the host gives per * m entries
    for (int r = op.lo + (int)threadIdx.x; r < hi; r += (int)blockDim.x) {
        const int t = (int)A.dx.div((uint32_t)r), i = r - t * A.nx, k = (int)A.dy.div((uint32_t)t), j = t - k * A.ny;
        int at = per * (r - op.lo);
        const int first = at;
        auto put = [&](bool in, int d, int off) {
            if (!in) return;
            val[at] = A.coef(d, i, j, k);
            addr[at] = op.address(r + off);
            ++at;
        };
        put(k > 0, PBCG_B, -A.nxy);
        put(j > 0, PBCG_S, -A.nx);
        put(i > 0, PBCG_W, -1);
        put(true, PBCG_C, 0);
        put(i < A.nx - 1, PBCG_E, 1);
        put(j < A.ny - 1, PBCG_N, A.nx);
        put(k < A.nz - 1, PBCG_T, A.nxy);
        range[r - op.lo] = make_int2(first, at);
    }
    op.val = val;
    op.addr = addr;
    op.col = nullptr;
}

template <class Op, bool Pipelined>
__global__ void __launch_bounds__(kOnChipTPB, 1) onchip_solve_kernel(const Op A, const SolveArgs a, int m, FastDiv dm,
                                                                     int cap) {
    extern __shared__ __align__(16) double onchip[];
    __shared__ Exchange<kOnChipTPB> X;
    __shared__ double slots[2][kMaxCluster][kSlotDoubles];   // cluster reductions: every CTA's block sums
    const unsigned size = cluster_ctas(), rank = cluster_rank();
    if (threadIdx.x == 0) X.ok = 1;
    ClusterSync g{slots, rank, size, 0u, 0};
    const int lo = (int)rank * m < a.n ? (int)rank * m : a.n;
    const int hi = lo + m < a.n ? lo + m : a.n;
    // vectors (by rows of the system), then the entries' values, the rows' ranges, the entries' addresses
    double *val = onchip + (size_t)kOnChipVecs * m;
    int2 *range = reinterpret_cast<int2 *>(val + cap);
    uint32_t *addr = reinterpret_cast<uint32_t *>(range + m);
    OnChipOp op{a.n, lo, m, dm, (uint32_t)__cvta_generic_to_shared(onchip), range, nullptr, nullptr, nullptr};
    onchip_entries(A, op, hi, cap, range, val, addr);
    SolveArgs s = a;
    double **vecs[kOnChipVecs] = {&s.V.r, &s.V.r0, &s.V.p, &s.V.s, &s.V.z, &s.V.q, &s.V.y, &s.V.w, &s.V.t, &s.V.v, &s.x};
#pragma unroll
    for (int k = 0; k < kOnChipVecs; ++k) *vecs[k] = onchip + (size_t)k * m - lo;
    PBCG_ROWS(i) { s.x[i] = a.x[i]; }
    cluster_barrier();   // every CTA started, and its x is in place
    Outcome o{0, PBCG_NOT_CONVERGED, 0, 0, 0.0, 0.0};
    int spmvs = 0;
    if constexpr (Pipelined)
        pipelined_loop<OnChipOp, double, kOnChipTPB, ClusterSync>(op, s, g, X, lo, hi, o, spmvs, nullptr);
    else
        standard_loop<OnChipOp, kOnChipTPB, ClusterSync>(op, s, g, X, lo, hi, o, spmvs, nullptr);
    finish(op, s, g, X, lo, hi, o, spmvs);
    PBCG_ROWS(i) { a.x[i] = s.x[i]; }
    cluster_barrier();   // no CTA leaves while another may still address its shared memory
}

// M^{-1} = 1 / diag(A) (Jacobi). A zero or non-finite diagonal entry sets *bad.
__global__ void jacobi_csr_kernel(int n, const int *rowptr, const int *col, const double *val, double *minv, int *bad) {
    PBCG_ELEMENTS(i, n) {
        double d = 0.0;
        for (int k = rowptr[i]; k < rowptr[i + 1]; ++k)
            if (col[k] == i) d = val[k];
        const double m = 1.0 / d;
        if (d == 0.0 || !isfinite(m)) atomicOr(bad, 1);
        minv[i] = m;
    }
}
__global__ void jacobi_stencil_kernel(const StencilOp A, double *minv, int *bad) {
    PBCG_ELEMENTS(r, A.n) {
        const int t = (int)A.dx.div((uint32_t)r);
        const int i = r - t * A.nx;
        const int k = (int)A.dy.div((uint32_t)t);
        const int j = t - k * A.ny;
        const double d = A.coef(PBCG_C, i, j, k);
        const double m = 1.0 / d;
        if (d == 0.0 || !isfinite(m)) atomicOr(bad, 1);
        minv[r] = m;
    }
}

// ===========================================================================
// Batched solves: many independent systems in one launch. The launch is made
// of thread-block clusters of `size` CTAs (size 1: plain blocks). The first
// CTA of a cluster takes the next system from an atomic counter; a system with
// at least `cluster_min_rows` rows is solved by the whole cluster (rows split
// into `size` contiguous ranges, reductions through distributed shared memory
// and the hardware cluster barrier, ClusterSync); otherwise the first CTA
// takes `size` - 1 further systems and every CTA solves one alone (block-level
// reductions and barriers, BlockSync). Clusters never wait on each other, so
// no co-residency beyond the cluster is needed and the launch can be captured
// in a CUDA graph. System s owns the global rows [row_offset[s],
// row_offset[s+1]) of the concatenated CSR arrays (row pointers index the
// shared col/val arrays; column indices are local to the system) and of b, x
// and the work vectors. Systems are taken in index order; ordering them
// largest first balances the load.
// ===========================================================================
struct BatchArgs {
    int nsys;
    int nnz;
    long long total_rows;
    const long long *row_offset;   // [nsys + 1]
    const int *rowptr;             // [total rows + 1], global offsets into col/val
    const int *col;                // local column indices
    const double *val;
    const double *b;
    double *x;
    Vectors V;                     // global work vectors (total rows each)
    unsigned *next;                // work counter, zero before the launch
    pbcg_batch_result *out;        // [nsys]
    double rtol;
    int maxit;
    int replace_period;
    long long cluster_min_rows;    // systems this large are solved by a whole cluster
    int fixed;                     // > 0: every system runs exactly this many iterations
    double *hist;                  // nullable: ||r_i|| of system s at hist[s * hist_stride + i]
    long long hist_stride;
};

// Solve system `sys` on rows [lo, hi) of it (the whole system for BlockSync,
// this CTA's share for ClusterSync); the first CTA writes the result.
template <class Sync>
__device__ __forceinline__ void batched_system(const BatchArgs &B, int sys, Sync &g, unsigned part, unsigned parts,
                                               Exchange<kTPB> &X) {
    const long long r0 = B.row_offset[sys], r1 = B.row_offset[sys + 1];
    // structure check of this system: its rows inside the batch, entries inside
    // the shared arrays, columns local to the system (each CTA checks its rows)
    int bad = (r0 < 0 || r1 < r0 || r1 > B.total_rows || r1 - r0 >= (1ll << 31)) ? 1 : 0;
    const int n = bad ? 0 : (int)(r1 - r0);
    const int lo = (int)((long long)part * n / parts), hi = (int)((long long)(part + 1) * n / parts);
    const CsrOpGatherL2 A{{n, B.rowptr + (bad ? 0 : r0), B.col, B.val, B.nnz}};
    PBCG_ROWS(i) {
        const int e0 = A.rowptr[i], e1 = A.rowptr[i + 1];
        if (e0 < 0 || e1 < e0 || e1 > B.nnz) { bad = 1; continue; }
        for (int k = e0; k < e1 && !bad; ++k)
            if (B.col[k] < 0 || B.col[k] >= n) bad = 1;
    }
    double fb[1] = {(double)bad};
    exchange(g, fb, X, [](Scalars &S, const double (&t)[1]) { S.aux = t[0]; });
    pbcg_batch_result res{0, PBCG_ERR_ARG, 0, 0, 0.0, 0.0};
    if (X.s.aux == 0.0) {
        SolveArgs a;
        a.n = n;
        a.b = B.b + r0;
        a.x = B.x + r0;
        a.V = Vectors{B.V.r + r0, B.V.r0 + r0, B.V.p + r0, B.V.s + r0, B.V.z + r0,
                      B.V.q + r0, B.V.y + r0, B.V.w + r0, B.V.t + r0, B.V.v + r0};
        a.ctl = nullptr;
        a.partials = nullptr;
        a.hist = B.hist ? B.hist + (size_t)sys * (size_t)B.hist_stride : nullptr;
        a.rtol = B.rtol;
        a.limit = B.fixed > 0 ? B.fixed : B.maxit;
        a.fixed = B.fixed > 0 ? 1 : 0;
        a.replace_period = B.replace_period;
        a.max_repl = -1;
        a.variant = 0;
        a.minv = nullptr;
        a.rh = a.sh = a.zh = a.qh = a.wh = nullptr;
        Outcome o{0, PBCG_NOT_CONVERGED, 0, 0, 0.0, 0.0};
        int spmvs = 0;
        pipelined_loop<CsrOpGatherL2, double, kTPB, Sync>(A, a, g, X, lo, hi, o, spmvs, nullptr);
        // the history holds squared norms after entry 0 (written by this thread)
        if (a.hist && part == 0 && threadIdx.x == 0)
            for (int i = 1; i <= o.iters; ++i) a.hist[i] = sqrt(a.hist[i]);
        // true residual of the returned x
        double d[1] = {0.0};
        PBCG_ROWS(i) {
            const double rr = a.b[i] - A.row(i, VecLoad{a.x});
            d[0] = fma(rr, rr, d[0]);
        }
        exchange(g, d, X, [](Scalars &S, const double (&t)[1]) { S.aux = t[0]; });
        res.iters = o.iters;
        res.status = o.status;
        res.half_step = o.half;
        res.n_replacements = o.nrr;
        const double nr = o.iters > 0 ? sqrt(o.nr) : o.nr0;
        res.rel_res_recursive = o.nr0 > 0.0 ? nr / o.nr0 : 0.0;
        res.rel_res_true = o.nr0 > 0.0 ? sqrt(X.s.aux) / o.nr0 : sqrt(X.s.aux);
    }
    if (part == 0 && threadIdx.x == 0) B.out[sys] = res;
}

__global__ void __launch_bounds__(kTPB, 6) batched_kernel(const BatchArgs B) {
    __shared__ Exchange<kTPB> X;
    __shared__ double slots[2][kMaxCluster][kSlotDoubles];   // cluster reductions: every CTA's block sums
    __shared__ int item[2];   // system of this CTA (-1: none), whole-cluster flag (-1: no work left)
    const unsigned size = cluster_ctas(), rank = cluster_rank();
    if (size > 1) cluster_barrier();   // every CTA started before its shared memory is addressed
    for (;;) {
        if (rank == 0 && threadIdx.x == 0) {
            const int s = (int)atomicAdd(B.next, 1u);
            int whole = 0;
            if (s >= B.nsys) {
                whole = -1;
            } else if (size > 1) {
                const long long rows = B.row_offset[s + 1] - B.row_offset[s];
                whole = rows >= B.cluster_min_rows ? 1 : 0;
            }
            int extra = 0;
            if (whole == 0 && size > 1) extra = (int)atomicAdd(B.next, size - 1);
            for (unsigned r = 0; r < size; ++r) {
                int mine = s;
                if (whole == -1) mine = -1;
                else if (whole == 0 && r > 0) mine = extra + (int)r - 1 < B.nsys ? extra + (int)r - 1 : -1;
                if (size > 1) {
                    st_cluster_s32(cluster_map(&item[0], r), mine);
                    st_cluster_s32(cluster_map(&item[1], r), whole);
                } else {
                    item[0] = mine;
                    item[1] = whole;
                }
            }
        }
        if (size > 1) cluster_barrier();
        else __syncthreads();
        const int sys = item[0], whole = item[1];
        if (whole < 0) return;   // the same for every CTA of the cluster
        if (whole == 1) {
            ClusterSync g{slots, rank, size, 0u, 0};
            batched_system(B, sys, g, rank, size, X);
        } else if (sys >= 0) {
            BlockSync g{0};
            batched_system(B, sys, g, 0u, 1u, X);
        }
        // every CTA is done with this item (and with the slots) before the next claim
        if (size > 1) cluster_barrier();
        else __syncthreads();
    }
}

// Diagnostic of the bounded grid-wide wait: every block but the last enters a
// grid synchronisation that the last block never joins, so the wait cannot
// complete and must end at its limit. The first block to give up records
// PBCG_ERR_TIMEOUT in the abort flag; the others see the flag (or their own
// limit) and return. Block 0 then reports the flag.
__global__ void sync_timeout_probe_kernel(Control *ctl, double *slots, uint64_t limit_ns) {
    __shared__ Exchange<kTPB> X;
    if (blockIdx.x == gridDim.x - 1) return;
    if (threadIdx.x == 0) X.ok = 1;
    GridSync g{ctl, slots, 0u, 0, kTPB, limit_ns};
    const bool ok = grid_sync(g, X);
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->status = ok ? (int)PBCG_OK : ld_relaxed_s32(&ctl->abort);
}

// out[k] = (float)in[k], k < len (FP32 copies of stencil coefficient tables).
__global__ void to_float_kernel(const double *in, float *out, long long len) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < len; k += (long long)gridDim.x * blockDim.x)
        out[k] = (float)in[k];
}

// y = A x, one row per thread, grid-stride.
template <class Op>
__global__ void __launch_bounds__(kTPB) spmv_kernel(const Op A, const double *x, double *y) {
    const VecLoad u{x};
    PBCG_ELEMENTS(i, A.n) y[i] = A.row(i, u);
}

// CSR structure check: rowptr[0] == 0, non-decreasing, rowptr[n] == nnz, 0 <= col < n.
__global__ void csr_check_kernel(int n, int nnz, const int *rowptr, const int *col, int *bad) {
    PBCG_ELEMENTS(i, (unsigned)n + 1u) {
        const int a = rowptr[i];
        if (i == 0 && a != 0) atomicOr(bad, 1);
        if (i == n && a != nnz) atomicOr(bad, 2);
        if (i < n && rowptr[i + 1] < a) atomicOr(bad, 4);
        if (a < 0 || a > nnz) atomicOr(bad, 8);
    }
    PBCG_ELEMENTS(k, nnz) {
        const int c = col[k];
        if (c < 0 || c >= n) atomicOr(bad, 16);
    }
}

#undef PBCG_ROWS
#undef PBCG_STEPS

}  // namespace pbcg
