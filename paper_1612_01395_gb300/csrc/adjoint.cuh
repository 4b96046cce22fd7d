// Building blocks of the adjoint (reverse-mode) solve: the transpose of a CSR
// matrix and the gradient with respect to its stored values.
//
// For x = A^{-1} b and a loss L(x), the adjoint lambda = A^{-T} dL/dx gives
// dL/db = lambda and dL/da_ij = -lambda_i x_j for every stored entry (i, j).
// The transpose is built deterministically: entries are scattered with atomic
// cursors and each row of A^T is then sorted by column, so the row order (and
// hence every SpMV with A^T) does not depend on scheduling.
#pragma once

#include "device_common.cuh"

namespace pbcg {

// counts[c + 1] += 1 for every stored column c (counts zeroed by the caller)
__global__ void transpose_count_kernel(int nnz, const int *col, int *counts) {
    PBCG_ELEMENTS(k, nnz)
        atomicAdd(&counts[col[k] + 1], 1);
}

// Inclusive prefix sum over the threads of a block of 1024.
__device__ __forceinline__ int block_scan(int v, int *warps) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) warps[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int w = warps[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += u;
        }
        warps[lane] = w;
    }
    __syncthreads();
    return wid > 0 ? v + warps[wid - 1] : v;
}

// In-place inclusive prefix sum of a[0..m) in tiles of 4096 elements, which turns
// counts into row pointers. Three passes: the sum of each tile, the tile sums
// scanned by one block, and each tile scanned from its offset. One
// block walking 1024 uncoalesced chunks took 787 us for 1M counts; these take
// about 10.
constexpr int kScanTile = 4096, kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(int m, const int *a, int *sums) {
    __shared__ int warps[32];
    const long long base = (long long)blockIdx.x * kScanTile;
    int v = 0;
#pragma unroll
    for (int k = 0; k < kScanTile / kScanThreads; ++k) {
        const long long i = base + k * kScanThreads + threadIdx.x;
        if (i < m) v += a[i];
    }
    v = block_scan(v, warps);
    if (threadIdx.x == kScanThreads - 1) sums[blockIdx.x] = v;
}
__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(int tiles, int *sums) {
    __shared__ int warps[32];
    int run = 0;
    for (int t0 = 0; t0 < tiles; t0 += kScanThreads) {
        const int t = t0 + (int)threadIdx.x;
        const int own = t < tiles ? sums[t] : 0;
        const int v = block_scan(own, warps);
        if (t < tiles) sums[t] = run + v - own;   // exclusive
        __syncthreads();
        run += warps[31];
        __syncthreads();
    }
}
__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(int m, int *a, const int *sums) {
    __shared__ int warps[32];
    constexpr int kEach = kScanTile / kScanThreads;
    const long long base = (long long)blockIdx.x * kScanTile + (long long)threadIdx.x * kEach;
    int v[kEach], s = 0;
#pragma unroll
    for (int k = 0; k < kEach; ++k) {
        v[k] = base + k < m ? a[base + k] : 0;
        s += v[k];
        v[k] = s;
    }
    const int off = block_scan(s, warps) - s + sums[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kEach; ++k)
        if (base + k < m) a[base + k] = off + v[k];
}

// Scatter entry (i, c, v) of A to row c of A^T at the next free slot.
__global__ void transpose_scatter_kernel(int n, const int *rowptr, const int *col, const double *val,
                                         const int *trow, int *cursor, int *tcol, double *tval) {
    PBCG_ELEMENTS(i, n) {
        for (int k = rowptr[i]; k < rowptr[i + 1]; ++k) {
            const int c = PBCG_SAFE(col[k], n);
            const int pos = trow[c] + atomicAdd(&cursor[c], 1);
            tcol[pos] = i;
            tval[pos] = val[k];
        }
    }
}

// Sort every row of A^T by column (insertion sort; rows are short).
__global__ void sort_rows_kernel(int n, const int *rowptr, int *col, double *val) {
    PBCG_ELEMENTS(i, n) {
        const int b = rowptr[i], e = rowptr[i + 1];
        for (int k = b + 1; k < e; ++k) {
            const int c = col[k];
            const double v = val[k];
            int j = k - 1;
            while (j >= b && col[j] > c) {
                col[j + 1] = col[j];
                val[j + 1] = val[j];
                --j;
            }
            col[j + 1] = c;
            val[j + 1] = v;
        }
    }
}

// g[k] = -lambda[i] * x[col[k]] for every stored entry k of row i.
__global__ void value_grad_kernel(int n, const int *rowptr, const int *col, const double *lambda, const double *x,
                                  double *g) {
    PBCG_ELEMENTS(i, n) {
        const double li = lambda[i];
        for (int k = rowptr[i]; k < rowptr[i + 1]; ++k) g[k] = -li * x[PBCG_SAFE(col[k], n)];
    }
}

}  // namespace pbcg
