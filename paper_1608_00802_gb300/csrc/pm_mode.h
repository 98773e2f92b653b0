// |m| of an integer mode, for the P(k) kernel and for its host test.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define PM_HD __host__ __device__ __forceinline__
#else
#define PM_HD inline
#endif

namespace pm {

// sqrt(m2) in fp64 from s = sqrtf(m2), m2 < 2^20 (exact in fp32), without the fp64 pipe's square root: the root is
// s + c with c = (m2 - s^2 - c^2) / (2 s).  The residual of s is exact (fma), so c to first order (hi) and
// its own residual with the second-order term (lo) are good to 2^-24 of 2^-24 of 2^-24, far below the
// last bit of the fp64 sum: the value is the fp64 square root's for every m2 up to 3 * 512^2.
PM_HD double mode_norm(uint32_t m2, float s) {
  const float res = fmaf(-s, s, float(m2));
  const float hi = 0.5f * res / s;
  const float lo = fmaf(-hi, hi, fmaf(-(s + s), hi, res)) * (0.5f / s);
  return double(s) + (double(hi) + double(lo));
}

}  // namespace pm
