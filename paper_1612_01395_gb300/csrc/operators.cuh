// The sparse operators A of A x = b: CSR and 5/7-point stencil.
//
// Each operator computes one row of a product, (A u)_row = sum_j a_{row,j} u_j,
// where u_j is produced by a loader functor. The plain loader reads a vector;
// other loaders form a vector on the fly (e.g. p = r + beta (p - omega s) for
// neighbours), which lets a solver phase fuse an AXPY into its SpMV.
//
// Summation order of a row: its stored entries in order (CSR); B, S, W, C, E,
// N, T (stencil) -- ascending column index, so a stencil and its sorted CSR
// assembly give bitwise identical rows. Products are accumulated with FMA.
#pragma once

#include <cuda_bf16.h>

#include "device_common.cuh"

namespace pbcg {

// fma for the arithmetic type of a sweep (FP64 path, or FP32 inner solves).
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }

// A stored matrix value as the arithmetic type T of a sweep.
template <typename T>
__device__ __forceinline__ T value_as(double v) { return (T)v; }
template <typename T>
__device__ __forceinline__ T value_as(float v) { return (T)v; }
template <typename T>
__device__ __forceinline__ T value_as(__nv_bfloat16 v) { return (T)__bfloat162float(v); }

// u_j = x[j]
template <typename T>
struct VecLoadT {
    const T *x;
    __device__ __forceinline__ T operator()(int j) const { return x[j]; }
};
using VecLoad = VecLoadT<double>;

// u_j = r_j + beta (p_j - omega s_j): the p-recurrence of Algorithm 7
struct PLoad {
    const double *r, *p, *s;
    double beta, omega;
    __device__ __forceinline__ double operator()(int j) const { return fma(beta, fma(-omega, s[j], p[j]), r[j]); }
};

// u_j = r_j - alpha s_j: q of Algorithm 7
struct QLoad {
    const double *r, *s;
    double alpha;
    __device__ __forceinline__ double operator()(int j) const { return fma(-alpha, s[j], r[j]); }
};

// CSR with values stored as V (double; float or bfloat16 for low-precision
// inner solves). A row is accumulated in the loader's type, in storage order.
// kChunk > 1 takes a row's entries kChunk at a time: all column indices and
// values of a chunk in flight together, then all gathers, then the FMAs in
// storage order (the same sum as the one-by-one loop). The entries missing
// from a row's last chunk are predicated off. kChunk = 1 is the plain loop.
// Which one pays was measured per matrix class (time per iteration, both
// methods, FP64):
// * 7-point rows (256^3): 7 at a time 5.5 % (Algorithm 9) and 6 % (Algorithm
//   7) faster than one at a time; 8 at a time spilled registers and gained
//   half as much, 4 at a time lost. Taking only whole chunks and the rest one
//   at a time lost 10 %: warps holding a boundary row ran both paths.
// * Random rows of 9-33 entries (2^20 rows): 7 at a time 4-5 % faster.
// * 5-point rows: 5 at a time 3-6 % (Algorithm 9) and 1-5 % (Algorithm 7)
//   faster than one at a time, from 160^2 (13.0 against 13.4 us an iteration)
//   to 2048^2 (254.6 against 269.7 us); 3 at a time slower than one, and 7
//   slower still: a predicated-off FP64 FMA occupies the FP64 pipe like a
//   live one, and 2 of every 7 were dead.
// The grid solves therefore use 7 at a time for matrices averaging more than
// 6 entries per row and 5 otherwise. FP32 and BF16 values (the inner solves)
// take 8 at a time (4 and 6 measured slower); the batched solver keeps the
// plain loop (its rows gained nothing from chunks), with its gathers through
// L2 only (CsrOpGatherL2).
template <typename V, int kChunk = 8>
struct CsrOpT {
    int n;
    const int *__restrict__ rowptr;
    const int *__restrict__ col;
    const V *__restrict__ val;
    int nnz;   // entries readable at col and val (the bounds of a checked build)

    template <class L>
    __device__ __forceinline__ auto row(int r, const L &u) const -> decltype(u(0)) {
        using T = decltype(u(0));
        const int b = __ldg(rowptr + PBCG_SAFE(r, n)), e = __ldg(rowptr + PBCG_SAFE(r, n) + 1);
        T acc = T(0);
        if constexpr (kChunk <= 1) {
            for (int k = b; k < e; ++k) {
                const int kk = PBCG_SAFE(k, nnz);
                acc = fmaT(value_as<T>(__ldg(val + kk)), u(PBCG_SAFE(__ldg(col + kk), n)), acc);
            }
        } else {
            // Counted from the row's first entry, as b + kChunk may pass 2^31. 7 at
            // a time compares with the length (SpMV at 256^3 311 against 332 us),
            // the others with what is left (FP32 iterations at 64^3 26.4 against
            // 27.6 us, 5-entry rows at 2048^2 254 against 261).
            const int len = e - b;
            for (int k0 = 0, left = len; left > 0; k0 += kChunk, left -= kChunk) {
                const auto has = [&](int j) { return kChunk == 7 ? k0 + j < len : j < left; };
                int c[kChunk] = {};
                V v[kChunk] = {};
                T xv[kChunk] = {};
#pragma unroll
                for (int j = 0; j < kChunk; ++j)
                    if (has(j)) {
                        const int kk = PBCG_SAFE(b + k0 + j, nnz);
                        c[j] = __ldg(col + kk);
                        v[j] = __ldg(val + kk);
                    }
#pragma unroll
                for (int j = 0; j < kChunk; ++j)
                    if (has(j)) xv[j] = u(PBCG_SAFE(c[j], n));
#pragma unroll
                for (int j = 0; j < kChunk; ++j)
                    if (has(j)) acc = fmaT(value_as<T>(v[j]), xv[j], acc);
            }
        }
        return acc;
    }
};
using CsrOpScalar = CsrOpT<double, 1>;    // one entry at a time
using CsrOpChunked = CsrOpT<double, 7>;   // 7 entries at a time
using CsrOpShort = CsrOpT<double, 5>;     // 5 entries at a time

// A loader whose vector reads bypass L1 (ld.global.cg: cached in L2 only).
template <class L>
struct L2Gather {
    L u;
    __device__ __forceinline__ auto operator()(int j) const -> decltype(u(0)) { return u(j); }
};
template <typename T>
struct L2Gather<VecLoadT<T>> {
    VecLoadT<T> u;
    __device__ __forceinline__ T operator()(int j) const { return __ldcg(u.x + j); }
};

// The batched solver's CSR operator (random systems, 9-33 entries a row with
// uniformly random columns). Each lane streams its own row's column indices
// and values, and a sector of them serves 4 to 8 consecutive entries if it
// stays in L1 that long. So everything else bypasses L1 (ld.global.cg, cached
// in L2 only): the SpMV's gathers, and the fused sweeps' vector loads, which
// are used once (SweepLoadsL2). On the 512-system batch, the gathers alone
// took 52.4 against 55.1 ms, the gathers and sweep loads 50.6 against 52.8
// ms; an evict_last priority on the row streams' loads changed nothing
// (52.4 ms). The results are bit for bit the same.
struct CsrOpGatherL2 : CsrOpScalar {
    template <class L>
    __device__ __forceinline__ auto row(int r, const L &u) const -> decltype(u(0)) {
        return CsrOpScalar::row(r, L2Gather<L>{u});
    }
};
// Rows averaging more than this many entries take the chunked operator.
constexpr long long kChunkedMinAvgRow = 6;

// One coefficient: t1[i*a1 + j*b1 + k*c1] (or `value` when t1 is null) plus
// t2[i*a2 + j*b2 + k*c2] when t2 is set (n2 = 1, else 0). Indices fit 31 bits
// (checked at create). C is the type of the tables: double, or float for the
// low-precision inner solves (tables rounded to FP32 by the library).
template <typename C>
struct StCoefT {
    const C *t1, *t2;
    int a1, b1, c1, a2, b2, c2;
    int n2;
    C value;
    int len1, len2;   // elements readable at t1 and t2 (the bounds of a checked build)
};
using StCoef = StCoefT<double>;

__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

template <typename C, bool kAhead = true>
struct StencilOpT {
    int n, nx, ny, nz;
    int nxy;
    FastDiv dx, dy;
    StCoefT<C> c[7];   // C, W, E, S, N, B, T

    // First table (or value) of coefficient d at node (i, j, k).
    __device__ __forceinline__ C first(int d, int i, int j, int k) const {
        const StCoefT<C> &q = c[d];
        return q.t1 ? __ldg(q.t1 + PBCG_SAFE(i * q.a1 + j * q.b1 + k * q.c1, q.len1)) : q.value;
    }
    // v plus the second table of coefficient d. The second table is rare (a
    // coefficient varying along two separate directions), and its addition is
    // written as a loop of n2 (0 or 1) trips so that the compiler jumps over it
    // rather than predicating it: a DADD whose lanes are all predicated off
    // still occupies the FP64 pipe for a whole warp instruction (64 cycles per
    // sub-partition on this GPU), which as an if-converted branch cost 6 dead
    // DADDs per row of a 7-point stencil with one summed coefficient.
    __device__ __forceinline__ C second(int d, int i, int j, int k, C v) const {
        const StCoefT<C> &q = c[d];
#pragma unroll 1
        for (int m = 0; m < q.n2; ++m) v = add_rn(v, __ldg(q.t2 + PBCG_SAFE(i * q.a2 + j * q.b2 + k * q.c2, q.len2)));
        return v;
    }
    __device__ __forceinline__ C coef(int d, int i, int j, int k) const { return second(d, i, j, k, first(d, i, j, k)); }

    // kAhead: all neighbour values and first tables are loaded before the sum,
    // whose chain (about 140 cycles a step, and a loop per second table that
    // loads are not moved across) would otherwise wait for one load after
    // another. Algorithm 9 per iteration: 32^3 18.9 -> 16.6 us, 48^3 29.4 ->
    // 27.0, 128^3 179 -> 174. The mixed-precision kernel, with 64 registers for
    // its FP32 sweeps, spills more with it and loads one neighbour at a time, as
    // does the SpMV of systems that stay in L2.
    template <class L>
    __device__ __forceinline__ auto row(int r, const L &u) const -> decltype(u(0)) {
        using T = decltype(u(0));
        const int t = (int)dx.div((uint32_t)r);
        const int i = r - t * nx;
        const int k = (int)dy.div((uint32_t)t);
        const int j = t - k * ny;
        const bool in[7] = {true, i > 0, i < nx - 1, j > 0, j < ny - 1, k > 0, k < nz - 1};
        const int off[7] = {0, -1, 1, -nx, nx, -nxy, nxy};
        constexpr int order[7] = {PBCG_B, PBCG_S, PBCG_W, PBCG_C, PBCG_E, PBCG_N, PBCG_T};
        T acc = T(0);
        if constexpr (kAhead) {
            T uv[7];
            C cf[7];
#pragma unroll
            for (int d = 0; d < 7; ++d) uv[d] = in[d] ? u(PBCG_SAFE(r + off[d], n)) : T(0);
#pragma unroll
            for (int d = 0; d < 7; ++d) cf[d] = first(d, i, j, k);
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                const int d = order[m];
                if (in[d]) acc = fmaT((T)second(d, i, j, k, cf[d]), uv[d], acc);
            }
        } else {
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                const int d = order[m];
                if (in[d]) acc = fmaT((T)coef(d, i, j, k), u(PBCG_SAFE(r + off[d], n)), acc);
            }
        }
        return acc;
    }

    // ---- FP32 sweeps: groups of up to 4 adjacent rows of one x-line, so that
    // a group shares the decomposition of its row number, the boundary tests
    // and the coefficient loads that do not vary along x, and takes its vectors
    // in 128-bit accesses where nx % 4 == 0 (then every group starts on a
    // multiple of 4 rows, and so do its neighbours at nx and nx*ny).
    int gx;        // groups per x-line, groups_of(nx, 4)
    FastDiv dg;    // by gx
    int aligned;   // nx % 4 == 0

    struct Group {
        int r, cnt;     // first row, rows (4; fewer at the end of an x-line)
        int i, j, k;    // node of the first row
    };
    __device__ __forceinline__ int groups() const { return gx * ny * nz; }
    __device__ __forceinline__ Group group(int gi) const {
        Group q;
        const int t = (int)dg.div((uint32_t)gi);
        q.i = 4 * (gi - t * gx);
        q.k = (int)dy.div((uint32_t)t);
        q.j = t - q.k * ny;
        q.r = t * nx + q.i;
        q.cnt = nx - q.i < 4 ? nx - q.i : 4;
        return q;
    }
    // u at rows at .. at + cnt - 1, zero beyond
    __device__ __forceinline__ void load4(const float *u, int at, int cnt, float (&v)[4]) const {
        if (aligned) {
            const float4 f = *reinterpret_cast<const float4 *>(u + PBCG_SAFE(at, n - 3));
            v[0] = f.x;
            v[1] = f.y;
            v[2] = f.z;
            v[3] = f.w;
        } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) v[m] = m < cnt ? u[PBCG_SAFE(at + m, n)] : 0.0f;
        }
    }
    // acc[m] += coefficient d at node (i + m, j, k) * v[m] for m in [from, to);
    // each sum of two tables formed per node as in coef()
    __device__ __forceinline__ void add4(int d, const Group &q, const float (&v)[4], float (&acc)[4], int from = 0,
                                         int to = 4) const {
        const StCoefT<C> &f = c[d];
        float w[4];
        if (f.t1) {
            const int at = q.i * f.a1 + q.j * f.b1 + q.k * f.c1;
            w[0] = __ldg(f.t1 + PBCG_SAFE(at, f.len1));
            if (f.a1 == 0) {
                w[1] = w[2] = w[3] = w[0];
            } else {
#pragma unroll
                for (int m = 1; m < 4; ++m) w[m] = m < q.cnt ? __ldg(f.t1 + PBCG_SAFE(at + m * f.a1, f.len1)) : 0.0f;
            }
        } else {
            w[0] = w[1] = w[2] = w[3] = f.value;
        }
        if (f.n2) {
            const int at = q.i * f.a2 + q.j * f.b2 + q.k * f.c2;
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (m < q.cnt) w[m] = add_rn(w[m], __ldg(f.t2 + PBCG_SAFE(at + m * f.a2, f.len2)));
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float t = fmaT(w[m], v[m], acc[m]);
            acc[m] = m >= from && m < to ? t : acc[m];
        }
    }
    // y = A u on the rows of a group, mid = u there; each row summed as row()
    // sums it. The entries of neighbours outside the grid are left out, whatever
    // the tables hold there (0 times a NaN or an infinity would be NaN). Rows
    // past cnt read 0.
    __device__ __forceinline__ void product4(const Group &q, const float *u, float (&mid)[4], float (&y)[4]) const {
        float vb[4] = {}, vs[4] = {}, vn[4] = {}, vt[4] = {}, ve[4], vw[4];
        if (q.k > 0) load4(u, q.r - nxy, q.cnt, vb);
        if (q.j > 0) load4(u, q.r - nx, q.cnt, vs);
        load4(u, q.r, q.cnt, mid);
        if (q.j < ny - 1) load4(u, q.r + nx, q.cnt, vn);
        if (q.k < nz - 1) load4(u, q.r + nxy, q.cnt, vt);
        const float left = q.i > 0 ? u[PBCG_SAFE(q.r - 1, n)] : 0.0f;
        const float right = q.i < nx - 4 ? u[PBCG_SAFE(q.r + 4, n)] : 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            vw[m] = m > 0 ? mid[m - 1] : left;
            ve[m] = m < 3 ? mid[m + 1] : right;
            y[m] = 0.0f;
        }
        if (q.k > 0) add4(PBCG_B, q, vb, y);
        if (q.j > 0) add4(PBCG_S, q, vs, y);
        add4(PBCG_W, q, vw, y, q.i > 0 ? 0 : 1);
        add4(PBCG_C, q, mid, y);
        add4(PBCG_E, q, ve, y, 0, nx - 1 - q.i);
        if (q.j < ny - 1) add4(PBCG_N, q, vn, y);
        if (q.k < nz - 1) add4(PBCG_T, q, vt, y);
#pragma unroll
        for (int m = 1; m < 4; ++m)
            if (m >= q.cnt) y[m] = 0.0f;
    }
};
using StencilOp = StencilOpT<double>;
using StencilOpLean = StencilOpT<double, false>;   // FP64 residual of the mixed-precision kernel, SpMV in L2

// Operators whose fused sweeps load their vectors through L2 only.
template <class Op>
struct SweepLoadsL2 {
    static constexpr bool value = false;
};
template <>
struct SweepLoadsL2<CsrOpGatherL2> {
    static constexpr bool value = true;
};

// Operators with groups of FP32 rows.
template <class Op>
struct HasGroups {
    static constexpr bool value = false;
};
template <>
struct HasGroups<StencilOpT<float, false>> {
    static constexpr bool value = true;
};

}  // namespace pbcg
