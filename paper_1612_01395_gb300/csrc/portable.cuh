// Parts of the kernels that also compile for the host.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define PBCG_HD __host__ __device__ __forceinline__
#else
#define PBCG_HD inline
#endif

namespace pbcg {

PBCG_HD uint64_t bits_of(double v) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t u;
    memcpy(&u, &v, 8);
    return u;
#endif
}
// Neither zero, subnormal, infinite nor NaN, without an FP64 instruction.
PBCG_HD bool is_normal(double v) {
    const int e = (int)(bits_of(v) >> 52) & 0x7ff;
    return e != 0 && e != 0x7ff;
}
// (alpha / rho) (1 / omega) from its two factors, or 0 where a factor or the
// product left the normal range: a subnormal factor has lost bits that the
// product, normal again, does not show.
PBCG_HD double beta_gain(double alpha_rho, double inv_omega) {
#ifdef __CUDA_ARCH__
    const double g = __dmul_rn(alpha_rho, inv_omega);
#else
    const double g = alpha_rho * inv_omega;
#endif
    return is_normal(alpha_rho) && is_normal(inv_omega) && is_normal(g) ? g : 0.0;
}

// Whether a counter that starts at 0 and wraps at 2^32 has reached `target`,
// which is never 2^31 or more away from it.
PBCG_HD bool reached(unsigned counter, unsigned target) { return (int)(counter - target) >= 0; }

// Groups of g that n elements make, the last perhaps smaller (n + g - 1 may pass 2^31).
PBCG_HD int groups_of(int n, int g) { return n / g + (n % g != 0); }

}  // namespace pbcg

// The elements below count (at most 2^31) that belong to a thread of a kernel:
// every (threads of the grid)-th. The steps are unsigned: the index after the
// last may lie above 2^31, and a signed one would wrap below the bound again.
#define PBCG_ELEMENTS(i, count)                                                              \
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); (unsigned)i < (unsigned)(count); \
         i = (int)((unsigned)i + gridDim.x * blockDim.x))
