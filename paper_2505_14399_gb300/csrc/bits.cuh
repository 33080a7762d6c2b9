// Conversions between double, float and double-float on the integer units.
//
// This GPU's FP64 pipe takes a warp's conversion in 16 cycles of the whole SM, so passes that only
// change a type were bound by it (100 MB of float fields to double: 98 us instead of the 44 us
// their bytes take).  Normal numbers are converted here by moving exponent and mantissa bits;
// everything else (zero, subnormal, infinite, NaN, out of the other type's normal range) takes the
// hardware instruction.  Results are those of the hardware conversions bit for bit, except that
// df_from_bits may split an exact tie the other way (hi, -lo), which is as good a double-float.
#pragma once

#include "df64.cuh"

namespace wmg {

__device__ __forceinline__ double f64_from_bits(float x) {
  const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)   // normal
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
  return (double)x;
}

// round to nearest even
__device__ __forceinline__ float f32_from_bits(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned ex = (h >> 20) & 0x7ffu;
  if (ex - 897u < 253u) {              // 2^-126 <= |x| < 2^127
    unsigned f = ((ex - 896u) << 23) | ((h & 0xfffffu) << 3) | (l >> 29);
    const unsigned t = l & 0x1fffffffu;
    f += (t > 0x10000000u || (t == 0x10000000u && (f & 1u))) ? 1u : 0u;
    return __uint_as_float((h & 0x80000000u) | f);
  }
  return (float)x;
}

__device__ __forceinline__ df df_from_bits(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned ex = (h >> 20) & 0x7ffu;
  if (ex - 949u < 201u) {              // 2^-74 <= |x| < 2^127: the low word is normal as well
    unsigned f = ((ex - 896u) << 23) | ((h & 0xfffffu) << 3) | (l >> 29);
    const unsigned t = l & 0x1fffffffu, up = t >> 28;
    f += up;
    const int r = (int)t - (int)(up << 29);   // in [-2^28, 2^28), units of 2^(e - 52)
    const float scale = __uint_as_float((h & 0x80000000u) | ((ex - 948u) << 23));
    return {__uint_as_float((h & 0x80000000u) | f), __int2float_rn(r) * scale};
  }
  return df_from(x);
}
__device__ __forceinline__ zdf zdf_from_bits(zd x) { return {df_from_bits(x.re), df_from_bits(x.im)}; }

// hi + lo, correctly rounded (|lo| <= ulp(hi) / 2)
__device__ __forceinline__ double df_val_bits(df v) {
  const unsigned u = __float_as_uint(v.hi), a = u & 0x7fffffffu, ex = a >> 23;
  if (ex - 80u < 150u) {
    // hi = +-m 2^29 and lo = r in units of 2^(ex - 127 - 52)
    const float scale = __uint_as_float((306u - ex) << 23 | (u & 0x80000000u));   // +-2^(179 - ex)
    const long long s = ((long long)((a & 0x7fffffu) | 0x800000u) << 29) + __float2int_rn(v.lo * scale);
    if (s >= 1ll << 52 && s < 1ll << 53) {
      const unsigned h = (unsigned)((unsigned long long)s >> 32) & 0xfffffu;
      return __hiloint2double((int)((u & 0x80000000u) | ((ex + 896u) << 20) | h), (int)(unsigned)s);
    }
  }
  return (double)v.hi + (double)v.lo;
}

}  // namespace wmg
