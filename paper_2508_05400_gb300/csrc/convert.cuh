// Conversions between FP64 and double-float (hi + lo) that spare the FP64 pipe,
// which is 60 times slower than the others on sm_103a and runs the hardware's
// conversions too.  Both give the bits of the plain conversions.
#pragma once
#include <cuda_runtime.h>

namespace rks {

// (double)f from the bits; zeros, subnormals, infinities and NaNs by the hardware
__device__ __forceinline__ double widen(float f) {
  const unsigned b = __float_as_uint(f), e = b & 0x7F800000u;
  if (e == 0u || e == 0x7F800000u) return (double)f;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// hi + lo rounded to FP64: one FP64 add instead of two conversions and an add
__device__ __forceinline__ double df_to_double(float2 v) { return widen(v.x) + widen(v.y); }

// hi = RN(x), lo = RN(x - hi): x's 53 bits cut by integer operations where hi
// and lo are normal floats
__device__ __forceinline__ float2 df_from_double(double x) {
  const int xh = __double2hiint(x), xl = __double2loint(x);
  const int E = (xh >> 20) & 0x7FF;
  if (E < 950 || E > 1023 + 126) {
    const float h = __double2float_rn(x);
    return make_float2(h, __double2float_rn(x - (double)h));
  }
  const int m = ((xh & 0xFFFFF) << 3) | (int)((unsigned)xl >> 29), low = xl & 0x1FFFFFFF;
  const int up = low > 0x10000000 || (low == 0x10000000 && (m & 1)) ? 1 : 0;
  const int sg = xh & 0x80000000;
  const float l = __int2float_rn(low - (up << 29)) * __int_as_float(((E - 948) << 23) | sg);
  return make_float2(__int_as_float(((((E - 896) << 23) | m) + up) | sg), l);
}

}  // namespace rks
