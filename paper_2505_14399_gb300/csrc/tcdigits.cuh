// Exact fixed-point digit products on the fp16 tensor pipe (an Ozaki-style split) for the
// Galerkin forward-hop kernel.
//
// A double-float value v with |v| < 2 is written as 7 base-256 digits,
//     v = sum_{i < 7} s_i 2^{-6-8i},  s_i integers, |s_i| <= 128  (remainder at most 2^-55),
// each digit exact in fp16 (kept as s_i 2^-8).  The product of two such expansions is a sum of integer digit
// products: fp16 x fp16 MMAs with FP32 accumulation are exact while the partial sums stay
// below 2^24, the digit pairs (i, j) with i + j = d share one FP32 accumulator of weight
// 2^{-12-8d}, and pairs with i + j >= 7 (weight below 2^-68) are dropped.  The exact FP32 sums
// are then scaled by their weights (exact) and added to double-float accumulators with
// error-free two-sums.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"
#include "df64.cuh"
#include "tma.cuh"

namespace wmg {

constexpr int TC_NS = 7;               // digits per value

// The base-256 digits of two values v (|v| < 2, normalised: |v.lo| <= ulp(v.hi) / 2), each as
// the fp16 number s_i 2^-8, packed (the low word's digit at the lower address).
// Adding 1.546875 2^k (and 128 units) leaves v to the nearest 16-bit multiple of a unit in the
// low mantissa bits of the sum: n + 128 with n in [-2^15, 2^15], whose low byte is the second
// digit + 128 and whose next 16 bits, 0x4600 + floor((n + 128) / 256), hold the first, in
// [-128, 128].  The remainder is exact and either 0 or at least twice the low word, so a fast
// two-sum renormalises it; units of 2^-14, 2^-30, 2^-46 give two digits each and 2^-54 the last.
// The 16 bits 0x4600 + s are the fp16 number 6 + s 2^-8, and the low byte under the sum's
// exponent byte (0x44, 0x3c, 0x34) is 4^-j (4 + byte 2^-8): one byte permute and one exact fp16
// operation per digit of both values.  (Through FP32 and bf16 it took three permutes and a packed
// addition; seven rounds of rint, subtract, renormalise and scale took 98 FP32 instructions.)
__device__ __forceinline__ void tc_digits2(df2 v, unsigned s[TC_NS]) {
  const f32x2 m1 = f2_dup(0x1.8cp9f + 0x1p-7f), m2 = f2_dup(0x1.8cp-7f + 0x1p-23f);
  const f32x2 m3 = f2_dup(0x1.8cp-23f + 0x1p-39f), m4 = f2_dup(0x1.8p-31f + 0x1.18p-40f);
  const f32x2 a = f2_add(v.hi, m1);
  f32x2 r = f2_sub(v.hi, f2_sub(a, m1));
  f32x2 h = f2_add(r, v.lo), l = f2_sub(v.lo, f2_sub(h, r));
  const f32x2 b = f2_add(h, m2);
  r = f2_sub(h, f2_sub(b, m2));
  h = f2_add(r, l);
  l = f2_sub(l, f2_sub(h, r));
  const f32x2 c = f2_add(h, m3);
  const f32x2 d = f2_add(f2_add(f2_sub(h, f2_sub(c, m3)), l), m4);
  auto dig = [](f32x2 x, unsigned sel, float scale, float off) {
    const unsigned w = __byte_perm((unsigned)x, (unsigned)(x >> 32), sel);
    const __half2 y = __hfma2(*reinterpret_cast<const __half2*>(&w), __float2half2_rn(scale),
                              __float2half2_rn(off));
    return *reinterpret_cast<const unsigned*>(&y);
  };
  s[0] = dig(a, 0x6521, 1.0f, -6.0f);
  s[1] = dig(a, 0x7430, 1.0f, -4.5f);
  s[2] = dig(b, 0x6521, 1.0f, -6.0f);
  s[3] = dig(b, 0x7430, 4.0f, -4.5f);
  s[4] = dig(c, 0x6521, 1.0f, -6.0f);
  s[5] = dig(c, 0x7430, 16.0f, -4.5f);
  s[6] = dig(d, 0x5410, 1.0f, -6.0f);
}

// s + e += v w with an error-free two-sum (v w exact: w a power of two)
__device__ __forceinline__ void acc_fma(dfacc2& a, f32x2 v, f32x2 w) {
  const f32x2 s = f2_fma(v, w, a.s);
  const f32x2 nb = f2_sub(a.s, s);
  a.e = f2_add(a.e, f2_add(f2_sub(a.s, f2_add(s, nb)), f2_fma(v, w, nb)));
  a.s = s;
}

__device__ __forceinline__ bool tc_in_range(df2 v) {   // false for NaN
  return fabsf(f2_lo(v.hi)) < 2.0f && fabsf(f2_hi(v.hi)) < 2.0f;
}

}  // namespace wmg
