// A division by a number whose reciprocal is at hand. Plain C++ too, so that it
// can be compared with the division without a GPU.
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define BSVD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define BSVD_HOST_DEVICE inline
#endif

namespace bsvd {

// a / b, rounded to nearest, given inv = 1 / b rounded to nearest (Markstein's
// theorem, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990: with the remainder a - b q of a quotient q within one unit
// in the last place, exact in a fused multiply-add, q + r inv rounds to the
// nearest). The first correction makes q that close. For operands whose
// quotient and remainder do not underflow; a quotient of 0 has no sign.
BSVD_HOST_DEVICE float quotient(float a, float b, float inv) {
  float q = a * inv;
  q = fmaf(fmaf(-b, q, a), inv, q);
  return fmaf(fmaf(-b, q, a), inv, q);
}

}  // namespace bsvd
