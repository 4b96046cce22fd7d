// Device-side building blocks shared by the solver kernels: constants, the
// workspace control block, fast integer division, fixed-order reductions and
// the bounded grid-wide synchronisation.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "dots.cuh"
#include "pbicgstab.h"

namespace pbcg {

constexpr int kTPB = 128;          // threads per block of the batched kernel, the cluster kernel and the SpMV
constexpr int kMaxGrid = 2040;     // upper bound on thread blocks (kPartialBytes holds their slots)
constexpr int kMaxDots = 8;        // dot products carried by one reduction
constexpr uint64_t kSyncTimeoutNs = 4000000000ull;   // 4 s per grid-wide wait

// Bounds-checked build (-DPBCG_CHECK): PBCG_SAFE(i, n) yields i when 0 <= i < n,
// else records the source line in g_check_fault (the first such access only)
// and yields 0, so the access stays in bounds and the solve carries on; the
// host reads the record with pbicgstab_check_faults. It guards the indices
// that the operators form from data or geometry (gathered columns, stencil
// neighbours, row pointers). The default build compiles it to plain i.
#ifdef PBCG_CHECK
__device__ int g_check_fault;
__device__ __forceinline__ long long checked_index(long long i, long long n, int line) {
    if (i >= 0 && i < n) return i;
    atomicCAS(&g_check_fault, 0, line);
    return 0;
}
#define PBCG_SAFE(i, n) ((int)::pbcg::checked_index((long long)(i), (long long)(n), __LINE__))
#else
#define PBCG_SAFE(i, n) (i)
#endif

// Control block at the start of the workspace; zeroed before every solve.
struct Control {
    unsigned int arrivals;   // grid-sync arrivals, monotonic within one launch
    int abort;               // nonzero: pbcg_status that stopped the launch
    unsigned int ready;      // large grids: 1 + the last exchange whose totals are published
    int pad0[13];
    // result, written by block 0 at the end of a solve
    int iters, status, half_step, n_repl, grid_syncs, spmvs, inner_iters, pad1;
    double nr0, rel_rec, rel_true, pad2;
};
static_assert(sizeof(Control) <= 256, "control block must fit 256 bytes");
constexpr size_t kControlBytes = 256;
// 3 rotating buffers of one 8-double slot per block, then 3 rotating records of
// 16 doubles; a multiple of 256 bytes, so the vectors after it stay 256-byte aligned
constexpr size_t kPartialBytes = 393472;
static_assert((3ull * kMaxGrid * 8 + 3 * 16) * sizeof(double) <= kPartialBytes && kPartialBytes % 256 == 0,
              "slots and records fit");

// n / d for 0 <= n < 2^31 and 1 <= d < 2^31 by one multiply-high: the
// round-up method of Granlund & Montgomery, "Division by invariant integers
// using multiplication" (PLDI 1994): l = ceil(log2 d),
// m = floor(2^32 (2^l - d) / d) + 1, q = (mulhi(m, n) + n) >> l.
struct FastDiv {
    uint32_t d, m, l;
    __host__ void init(uint32_t dd) {
        d = dd;
        l = 0;
        while ((1ull << l) < dd) ++l;
        m = (uint32_t)(((((1ull << l) - dd)) << 32) / dd + 1);
    }
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return (__umulhi(m, n) + n) >> l; }
};

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Add 1: every store of the block ordered before this thread's by a barrier is
// ordered before the addition (release); the second form also returns the old
// value and orders later loads after it (acquire).
__device__ __forceinline__ void red_release_inc(unsigned *p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ unsigned atom_acq_rel_inc(unsigned *p) {
    unsigned v;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_relaxed_s32(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

constexpr unsigned kFull = 0xffffffffu;

// Sum of each of K values over the 32 lanes of a warp, returned to every lane.
// FP64 adds are the scarce resource on this GPU (one warp-wide DADD occupies a
// sub-partition's FP64 pipe for ~64 cycles), so the first log2(P) levels use
// recursive halving (P = K rounded up to a power of two): at each level a lane
// keeps half of its values and adds its partner's copy of them, costing P/2
// additions instead of P; the remaining levels are a butterfly on one value.
// K = 5 takes 9 additions instead of 25. After the halving, value index k
// lives in the lanes whose bits 4, 3, 2 (most significant first) spell k.
// Deterministic: in the butterfly both partners add the same two numbers (in
// either order, hence to the same bits), so all lanes holding index k agree.
template <int K>
__device__ __forceinline__ void warp_allsum(double (&v)[K]) {
    constexpr int P = K <= 1 ? 1 : K <= 2 ? 2 : K <= 4 ? 4 : 8;
    constexpr int M = P == 1 ? 0 : P == 2 ? 1 : P == 4 ? 2 : 3;
    static_assert(K <= 8, "at most 8 values");
    const int lane = threadIdx.x & 31;
    double w[P];
#pragma unroll
    for (int k = 0; k < P; ++k) w[k] = k < K ? v[k] : 0.0;
#pragma unroll
    for (int lvl = 0; lvl < M; ++lvl) {
        const int o = 16 >> lvl;
        const int half = P >> (lvl + 1);
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const double send = upper ? w[k] : w[k + half];
            const double keep = upper ? w[k + half] : w[k];
            w[k] = keep + __shfl_xor_sync(kFull, send, o);
        }
    }
#pragma unroll
    for (int o = 16 >> M; o > 0; o >>= 1) w[0] += __shfl_xor_sync(kFull, w[0], o);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        int src = 0;
#pragma unroll
        for (int b = 0; b < M; ++b)
            if (k & (1 << (M - 1 - b))) src |= 16 >> b;
        v[k] = __shfl_sync(kFull, w[0], src);
    }
}

// What the threads of a block share in an exchange. Every field after `part`
// is the same in all blocks of a solve once an exchange has completed.
struct alignas(16) Scalars {
    double alpha, beta, omega, rho;   // of the iteration
    double gain, slope;   // alpha / (rho omega) and (r0,s) - omega (r0,z): the next beta and alpha from them
    double nr;          // squared norm tested last
    double nr0, tol, bound;   // ||r_0||, the tolerance, the squared norms it can accept
    double aux;         // total of an exchange outside the iteration
    int action, status;   // what the loop does next (kGo, kHalf, kStop); pbcg_status of a stop
};
constexpr int kScalarWords = sizeof(Scalars) / 8;
static_assert(kScalarWords <= 16, "the scalars fit one published record");
enum { kGo = 0, kHalf = 1, kStop = 2 };

template <int T>   // most threads of the block
struct Exchange {
    double part[T / 32][kMaxDots];   // the warps' sums
    Scalars s;
    int ok;     // cleared when a wait is abandoned, never set again: a slow thread cannot read a later value
    int last;
};

// Sum of the first `rows` (at most 16) rows of K values, returned to every lane of the warp:
// warp_allsum on half-warps, the upper one holding the upper half of the values,
// which saves the first level of additions.
template <int K>
__device__ __forceinline__ void sum_rows(const double (*a)[kMaxDots], int rows, double (&v)[K]) {
    constexpr int P = K <= 1 ? 1 : K <= 2 ? 2 : K <= 4 ? 4 : 8;
    constexpr int H = P > 1 ? P / 2 : 1;                      // values of a lane
    constexpr int M = H == 1 ? 0 : H == 2 ? 1 : 2;            // halvings left
    const int lane = threadIdx.x & 31, row = lane & 15, first = P > 1 && lane >= 16 ? H : 0;
    double w[H];
#pragma unroll
    for (int k = 0; k < H; ++k) w[k] = row < rows && first + k < K ? a[row][first + k] : 0.0;
#pragma unroll
    for (int lvl = 0; lvl < M; ++lvl) {
        const int o = 8 >> lvl, half = H >> (lvl + 1);
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const double send = upper ? w[k] : w[k + half];
            const double keep = upper ? w[k + half] : w[k];
            w[k] = keep + __shfl_xor_sync(kFull, send, o);
        }
    }
#pragma unroll
    for (int o = 8 >> M; o > 0; o >>= 1) w[0] += __shfl_xor_sync(kFull, w[0], o);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        int src = k / H * 16;
#pragma unroll
        for (int b = 0; b < M; ++b)
            if (k % H & (1 << (M - 1 - b))) src |= 8 >> b;
        v[k] = __shfl_sync(kFull, w[0], src);
    }
}

// Fixed-order block sums, returned to every lane of warp 0: the warps reduce
// independently, then warp 0 adds their sums.
template <int K, int T>
__device__ __forceinline__ void block_sum(double (&v)[K], Exchange<T> &X) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    warp_allsum<K>(v);
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) X.part[wid][k] = v[k];
    }
    __syncthreads();
    if (wid == 0) {
        const int warps = (int)(blockDim.x >> 5);
        if constexpr (T / 32 <= 4) {   // lane k adds value k of the warps in warp order
            double t = 0.0;
            if (lane < K) {
                t = X.part[0][lane];
#pragma unroll
                for (int w = 1; w < T / 32; ++w)
                    if (w < warps) t += X.part[w][lane];
            }
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] = __shfl_sync(kFull, t, k);
        } else {                       // a tree is shorter than 7 or 15 additions in a row
            sum_rows<K>(X.part, warps, v);
        }
    }
}

// Grid-wide exchange of a cooperative launch. Each block owns one 64-byte
// slot (8 doubles) in each of 3 rotating buffers; exchange number e uses
// buffer e % 3. Thread 0 of a block stores its K block sums in its slot and adds
// 1 to the arrival counter with release at gpu scope (every store of the phase,
// made visible to thread 0 by __syncthreads, is ordered before the arrival;
// the waits are acquire loads). Then, by grid size:
//  * small grids: thread 0 spins on the counter until all blocks of exchange
//    e arrived, every block adds all slots in the same fixed order, and its
//    warp 0 forms the scalars;
//  * large grids (at least kLastReduceGrid blocks): the block whose arrival
//    completes the count adds all slots (same fixed order), forms the scalars,
//    publishes them and raises `ready`; the others spin on `ready` and read
//    them. Every block adding every slot costs each SM (blocks per SM x
//    blocks x K) FP64 additions per exchange against one extra flag hop.
// One poller per block on one word: polling all slots from every thread
// congests the L2 and was measured slower. The rotation keeps a slot or a
// total from being rewritten while a slow block may still read it (exchange
// e+3 is written only after all blocks arrived at e+2, i.e. after all finished
// reading exchange e). Results are bitwise identical in every block and do
// not depend on arrival order. Every wait is bounded (limit_ns,
// kSyncTimeoutNs by default) and watches the abort flag.
constexpr int kSlotDoubles = kMaxDots;
constexpr int kLastReduceGrid = 512;

struct GridSync {
    Control *ctl;
    double *slots;      // [3][gridDim.x][kSlotDoubles], then [3][16]: the scalars of an exchange
    unsigned epoch;     // exchanges done by this block
    int count;          // exchanges performed (for diagnostics)
    int step;           // distance between a thread's rows
    uint64_t limit_ns = kSyncTimeoutNs;   // bound on each wait
};
__device__ __forceinline__ int row_step(const GridSync &g) { return g.step; }

__device__ __forceinline__ double *slot_ptr(const GridSync &g, unsigned buf, int block) {
    return g.slots + ((size_t)buf * gridDim.x + block) * kSlotDoubles;
}
__device__ __forceinline__ double *totals_ptr(const GridSync &g, unsigned buf) {
    return g.slots + (size_t)3 * gridDim.x * kSlotDoubles + (size_t)buf * 16;
}
__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The block that records per-solve results (the residual history) under each
// synchronisation policy: block 0 of a grid; the block itself when a block
// solves alone; CTA rank 0 of a cluster (is_leader overloads below).
__device__ __forceinline__ bool is_leader(const GridSync &) { return blockIdx.x == 0; }

// Thread 0: spin until *word has reached target, bounded; false on abort or timeout.
// (A solve of more than 2^32 / blocks exchanges wraps the counter of arrivals.)
__device__ __forceinline__ bool wait_until(GridSync &g, const unsigned *word, unsigned target) {
    const uint64_t t0 = globaltimer_ns();
    for (unsigned spin = 1; !reached(ld_acquire_u32(word), target); ++spin) {
        if (spin % 8 != 0) continue;   // the flag and the clock now and then: each poll is a round trip to L2
        if (ld_relaxed_s32(&g.ctl->abort) != 0) return false;
        if (globaltimer_ns() - t0 > g.limit_ns) {
            atomicCAS(&g.ctl->abort, 0, (int)PBCG_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

// Barrier without data.
template <int T>
__device__ __forceinline__ bool grid_sync(GridSync &g, Exchange<T> &X) {
    __syncthreads();   // every thread's stores of this phase precede thread 0's arrival
    if (threadIdx.x == 0) {
        red_release_inc(&g.ctl->arrivals);
        if (!wait_until(g, &g.ctl->arrivals, (g.epoch + 1u) * gridDim.x)) X.ok = 0;
    }
    __syncthreads();
    g.epoch++;
    g.count++;
    return X.ok != 0;
}

// Fixed-order sum over all slots of buffer buf, returned to every lane of warp
// 0. Warps without a slot add nothing: their additions would queue on the FP64
// pipes with the others'.
template <int K, int T>
__device__ __forceinline__ void sum_slots(const GridSync &g, unsigned buf, double (&v)[K], Exchange<T> &X) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int grid = (int)gridDim.x, warps = (int)(blockDim.x >> 5);
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.0;
    if (wid * 32 < grid) {
        for (int b = threadIdx.x; b < grid; b += (int)blockDim.x) {
            const double *src = slot_ptr(g, buf, b);
#pragma unroll
            for (int k = 0; k < K; ++k) v[k] += __ldcg(src + k);
        }
        warp_allsum<K>(v);
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) X.part[wid][k] = v[k];
        }
    }
    __syncthreads();
    if (wid == 0) sum_rows<K>(X.part, (grid + 31) / 32 < warps ? (grid + 31) / 32 : warps, v);
}

// Barrier that adds the K values v of all threads of the grid in a fixed order
// and lets `f` turn the totals into the loop's scalars: f(scalars, totals) runs
// on one warp (all lanes alike) of every block, or of the last block to arrive,
// and every thread of every block finds the same result in X.s afterwards.
template <int K, int T, class F>
__device__ __forceinline__ bool exchange(GridSync &g, double (&v)[K], Exchange<T> &X, F f) {
    static_assert(K <= kSlotDoubles, "the values fit a slot");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    block_sum(v, X);
    const unsigned buf = g.epoch % 3u;
    const unsigned target = (g.epoch + 1u) * gridDim.x;
    const bool by_last = gridDim.x >= (unsigned)kLastReduceGrid;
    if (threadIdx.x == 0) {
        double *out = slot_ptr(g, buf, blockIdx.x);
#pragma unroll
        for (int k = 0; k < K; ++k) out[k] = v[k];
        if (by_last) {
            X.last = atom_acq_rel_inc(&g.ctl->arrivals) == target - 1u;
        } else {
            red_release_inc(&g.ctl->arrivals);
            if (!wait_until(g, &g.ctl->arrivals, target)) X.ok = 0;
        }
    }
    __syncthreads();
    if (!by_last) {
        sum_slots(g, buf, v, X);
        if (wid == 0) f(X.s, v);
    } else if (X.last) {   // every slot is visible: all blocks arrived with release
        sum_slots(g, buf, v, X);
        if (wid == 0) {
            f(X.s, v);
            __syncwarp();
            double *tot = totals_ptr(g, buf);
            if (lane < kScalarWords) tot[lane] = reinterpret_cast<const double *>(&X.s)[lane];
            __syncwarp();
            if (lane == 0) {
                st_release_u32(&g.ctl->ready, g.epoch + 1u);
            }
        }
    } else if (wid == 0) {
        if (lane == 0) {
            if (!wait_until(g, &g.ctl->ready, g.epoch + 1u)) X.ok = 0;
        }
        __syncwarp();
        const double *tot = totals_ptr(g, buf);
        if (lane < kScalarWords) reinterpret_cast<double *>(&X.s)[lane] = __ldcg(tot + lane);
    }
    g.epoch++;
    g.count++;
    __syncthreads();
    return X.ok != 0;
}

// Synchronisation policy of a solve owned by one thread block (batched
// solves): the "grid" is the block, a barrier is __syncthreads and a reduction
// is the block sum. Same interface as GridSync, so the solver loops are shared.
struct BlockSync {
    int count;
};

__device__ __forceinline__ bool is_leader(const BlockSync &) { return true; }
__device__ __forceinline__ int row_step(const BlockSync &) { return kTPB; }

template <int T>
__device__ __forceinline__ bool grid_sync(BlockSync &g, Exchange<T> &) {
    __syncthreads();
    g.count++;
    return true;
}

template <int K, int T, class F>
__device__ __forceinline__ bool exchange(BlockSync &g, double (&v)[K], Exchange<T> &X, F f) {
    block_sum(v, X);   // its barrier also orders the block's stores of the phase
    if (threadIdx.x < 32) f(X.s, v);
    g.count++;
    __syncthreads();
    return true;
}

// ---------------------------------------------------------------------------
// Thread-block clusters (batched solves of large systems). The CTAs of a
// cluster are co-scheduled by the hardware, so a wait on the hardware cluster
// barrier always completes once every CTA reaches it; each CTA can address
// the shared memory of the others (distributed shared memory).
// ---------------------------------------------------------------------------
constexpr int kMaxCluster = 16;

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_ctas() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Every thread of every CTA of the cluster arrives and waits. Release on
// arrival and acquire on the wait (cluster scope) order each CTA's earlier
// stores -- global and shared -- before the other CTAs' later loads.
// (The non-.aligned forms: no requirement that a warp arrives converged.)
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Address of *p (a __shared__ object of this CTA) in the shared memory of CTA `rank`.
__device__ __forceinline__ uint32_t cluster_map(const void *p, unsigned rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(a), "r"(rank));
    return out;
}
__device__ __forceinline__ void st_cluster_f64(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_s32(uint32_t addr, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Synchronisation policy of a solve shared by the `size` CTAs of a cluster:
// a barrier is the cluster barrier; a reduction pushes each CTA's K block sums
// into slot [rank] of EVERY CTA's slot array (distributed shared memory,
// posted stores), crosses the barrier, and then warp 0 of each CTA adds the
// `size` slots of its own shared memory and forms the scalars -- the same
// additions in the same order everywhere, so all CTAs hold identical scalars, with no remote
// loads on the critical path. Slot arrays alternate between two buffers:
// buffer e % 2 is rewritten by exchange e + 2, which a CTA starts only after
// the barrier of exchange e + 1, which every thread of every CTA reaches only
// after it has read exchange e. Same interface as GridSync and BlockSync.
struct ClusterSync {
    double (*slots)[kMaxCluster][kSlotDoubles];   // this CTA's shared [2][kMaxCluster][kSlotDoubles]
    unsigned rank, size;
    unsigned epoch;     // reductions done
    int count;
};

__device__ __forceinline__ bool is_leader(const ClusterSync &g) { return g.rank == 0; }
__device__ __forceinline__ int row_step(const ClusterSync &) { return (int)blockDim.x; }

template <int T>
__device__ __forceinline__ bool grid_sync(ClusterSync &g, Exchange<T> &) {
    cluster_barrier();
    g.count++;
    return true;
}

template <int K, int T, class F>
__device__ __forceinline__ bool exchange(ClusterSync &g, double (&v)[K], Exchange<T> &X, F f) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    block_sum(v, X);
    const unsigned buf = g.epoch & 1u;
    if (wid == 0 && lane < (int)g.size) {
#pragma unroll
        for (int k = 0; k < K; ++k) st_cluster_f64(cluster_map(&g.slots[buf][g.rank][k], (unsigned)lane), v[k]);
    }
    cluster_barrier();
    if (wid == 0) {
        sum_rows<K>(g.slots[buf], (int)g.size, v);
        f(X.s, v);
    }
    g.epoch++;
    g.count++;
    __syncthreads();
    return true;
}

}  // namespace pbcg
