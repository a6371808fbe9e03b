// quotient.h -- a division by the same number many times over (device, and plain C++ on the host).
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define MHC_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MHC_HOST_DEVICE inline
#endif

namespace mhc {

// a / b, correctly rounded, with y = 1 / b correctly rounded: Markstein's quotient iteration (P. Markstein, Computation
// of elementary functions on the IBM RISC System/6000 processor, 1990): the first correction leaves q within one unit in
// the last place, the second, with its exact remainder, rounds it.  It holds while remainders and quotients are normal
// numbers: an |a| outside of 1e-20 .. 1e20 (zeros with their signs, infinities) and a b outside of 1e-12 .. 1e12 (whose
// reciprocal may be infinite, or zero: 0 x infinity is no number) take the division.
MHC_HOST_DEVICE float quotient(float a, float b, float y) {
    float q = a * y;
    q = fmaf(fmaf(-q, b, a), y, q);
    q = fmaf(fmaf(-q, b, a), y, q);
    return fabsf(a) > 1e-20f && fabsf(a) < 1e20f && fabsf(y) > 1e-12f && fabsf(y) < 1e12f ? q : a / b;
}

}  // namespace mhc
