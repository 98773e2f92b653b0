// |m| of an integer mode, for the P(k) kernel and for its host test.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define PM_HD __host__ __device__ __forceinline__
#else
#define PM_HD inline
#endif

namespace pm {

// sqrt(m2) in fp64 from s = sqrtf(m2), 0 < m2 < 2^20 (exact in fp32), without the fp64 pipe: the root is
// s + c with c = (m2 - s^2 - c^2) / (2 s).  The residual of s is exact (fma), so c to first order (hi) and
// its own residual with the second-order term (lo) are good to 2^-24 of 2^-24 of 2^-24 of s.  c is counted in units of
// the fp64 value's last place (hi a whole number and an exact rest, at most 2^28 of them) and added to the bits of s: the
// fp64 square root's value for every m2 up to 3 * 512^2.
PM_HD double mode_norm(uint32_t m2, float s) {
  const float res = fmaf(-s, s, float(m2));
  const float hi = 0.5f * res / s;
  const float lo = fmaf(-hi, hi, fmaf(-(s + s), hi, res)) * (0.5f / s);
  uint32_t sb;
  memcpy(&sb, &s, 4);
  const uint32_t unit_bits = (127u + 52u + 127u - (sb >> 23)) << 23;  // 2^52 over the binade of s
  float unit;
  memcpy(&unit, &unit_bits, 4);
  const float t = hi * unit, whole = rintf(t);
  const int ulps = int(whole) + int(rintf((t - whole) + lo * unit));
  const uint64_t b = (uint64_t(sb) << 29) + (uint64_t(896) << 52) + uint64_t(int64_t(ulps));
  double r;
  memcpy(&r, &b, 8);
  return r;
}

}  // namespace pm
