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

// hi + lo rounded to FP64.  Where the sum keeps hi's exponent (always for a
// normalised pair, unless hi is a power of two and lo points inwards, even by
// less than half a unit: the binade below has twice the resolution), its 53
// bits are hi's 24 and lo rounded to 2^-29 of hi's last place: an integer add;
// the rest by one FP64 add of the widened words.  With the add everywhere the
// scaled conversion of 80 columns of n = 1e6 took 595 us, now 179 us (HBM).
__device__ __forceinline__ double df_to_double(float2 v) {
  const unsigned h = __float_as_uint(v.x);
  const int E = (int)((h >> 23) & 0xFFu);
  const float t = __uint_as_float(__float_as_uint(v.y) ^ (h & 0x80000000u)) *
                  __int_as_float(((306 - (E < 52 ? 52 : E)) & 0xFF) << 23);   // lo in those units, hi's sign taken off
  const int i = __float2int_rn(t);
  const long long m = ((long long)(0x800000u | (h & 0x7FFFFFu)) << 29) + i;
  if (E < 52 || E == 255 || !(fabsf(t) < 1073741824.f) || m < (1ll << 52) + (t < 0.f) || m >= (1ll << 53))
    return widen(v.x) + widen(v.y);
  const long long r = m + ((long long)(E + 1023 - 127 - 1) << 52);
  return __hiloint2double((int)(r >> 32) | (int)(h & 0x80000000u), (int)r);
}

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
  const int sg = xh & 0x80000000, rest = low - (up << 29);
  const float l = __int2float_rn(sg ? -rest : rest) * __int_as_float((E - 948) << 23);   // +0 where hi is all of x
  return make_float2(__int_as_float(((((E - 896) << 23) | m) + up) | sg), l);
}

}  // namespace rks
