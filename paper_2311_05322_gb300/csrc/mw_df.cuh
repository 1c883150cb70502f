// Double-float pairs from FP64 values.
#pragma once
#include <cuda_runtime.h>

namespace mwk {

// v = hi + lo with hi the nearest float (ties to even) and lo the nearest float to v - hi, from the bits of v: the
// significand's upper 24 bits rounded, and the signed remainder (29 bits) converted and scaled.  The same
// values as conversions and a subtraction in FP64, whose pipe (1/64 of the FP32 rate) bounded this pass at a
// third of the copy bandwidth.  Exponents outside [-90, 126], where a part or its scale may not be exact, take that way.
__device__ __forceinline__ void split_double(double v, float& hi, float& lo) {
  const long long b = __double_as_longlong(v);
  const int e = (int)(b >> 52 & 0x7ff) - 1023;
  if ((b << 1) == 0) {   // zeros: most of a right-hand side (the FP64 way took 480 us for 525,329 x 64 of them)
    hi = __int_as_float((int)(b >> 32));
    lo = 0.f;
    return;
  }
  if (e < -90 || e > 126) {
    hi = __double2float_rn(v);
    lo = __double2float_rn(v - (double)hi);
    return;
  }
  const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;      // 53 bits, value m 2^(e - 52)
  const int up = (int)((m + 0xfffffffll + (m >> 29 & 1)) >> 29);          // 24 bits (or 2^24)
  const int rem = (int)(m - ((long long)up << 29));
  const float s = __int_as_float((e + 127 - 23) << 23 | (int)(b >> 32 & 0x80000000ll));
  hi = (float)up * s;                                                     // exact
  // the conversion rounds, the scaling is exact: s 2^-29 is a power of two, at least 2^-142 (denormals are on).  rem s
  // alone, with |rem| up to 2^28, would overflow from exponent 123 on.
  lo = (float)rem * (s * 0x1p-29f);
}

// (re_hi, re_lo, im_hi, im_lo) of a complex FP64 value.
__device__ __forceinline__ float4 split_df2(double2 v) {
  float4 r;
  split_double(v.x, r.x, r.y);
  split_double(v.y, r.z, r.w);
  return r;
}

}  // namespace mwk
