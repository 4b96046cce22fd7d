// Parts of the kernels that also compile for the host.
#pragma once

#ifdef __CUDACC__
#define PBCG_HD __host__ __device__ __forceinline__
#else
#define PBCG_HD inline
#endif

// Whether a counter that starts at 0 and wraps at 2^32 has reached `target`,
// which is never 2^31 or more away from it.
PBCG_HD bool reached(unsigned counter, unsigned target) { return (int)(counter - target) >= 0; }

// Groups of g that n elements make, the last perhaps smaller (n + g - 1 may pass 2^31).
PBCG_HD int groups_of(int n, int g) { return n / g + (n % g != 0); }

// The elements below count (at most 2^31) that belong to a thread of a kernel:
// every (threads of the grid)-th. The steps are unsigned: the index after the
// last may lie above 2^31, and a signed one would wrap below the bound again.
#define PBCG_ELEMENTS(i, count)                                                              \
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); (unsigned)i < (unsigned)(count); \
         i = (int)((unsigned)i + gridDim.x * blockDim.x))
