// Parts of the kernels that also compile for the host.
#pragma once

#ifdef __CUDACC__
#define PBCG_HD __host__ __device__ __forceinline__
#else
#define PBCG_HD inline
#endif

// The elements below count (at most 2^31) that belong to a thread of a kernel:
// every (threads of the grid)-th. The steps are unsigned: the index after the
// last may lie above 2^31, and a signed one would wrap below the bound again.
#define PBCG_ELEMENTS(i, count)                                                              \
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); (unsigned)i < (unsigned)(count); \
         i = (int)((unsigned)i + gridDim.x * blockDim.x))
