// Exact fixed-point digit products on the bf16 tensor pipe (an Ozaki-style split) for the
// Galerkin forward-hop kernel.
//
// A double-float value v with |v| < 2 is written as 7 base-256 digits,
//     v = sum_{i < 7} s_i 2^{-6-8i},  s_i integers, |s_i| <= 128  (remainder at most 2^-55),
// each digit exact in bfloat16.  The product of two such expansions is a sum of integer digit
// products: bf16 x bf16 MMAs with FP32 accumulation are exact while the partial sums stay
// below 2^24, the digit pairs (i, j) with i + j = d share one FP32 accumulator of weight
// 2^{-12-8d}, and pairs with i + j >= 7 (weight below 2^-68) are dropped.  The exact FP32 sums
// are then scaled by their weights (exact) and added to double-float accumulators with
// error-free two-sums.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"
#include "df64.cuh"
#include "tma.cuh"

namespace wmg {

constexpr int TC_NS = 7;               // digits per value

__device__ __forceinline__ void ldm_x4t(unsigned r[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldm_x2t(unsigned r[2], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(smem_addr(p)));
}

// c += a b, 16x16 (row) x 16x8 (col) bf16, FP32 accumulators
__device__ __forceinline__ void mma_bf16(float c[4], const unsigned a[4], const unsigned b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// The base-256 digits of two values v (|v| < 2, normalised: |v.lo| <= ulp(v.hi) / 2).  Adding
// 1.5 2^k (and 128 units) leaves v to the nearest 16-bit multiple of a unit in the low mantissa
// bits of the sum: n + 128 with n in [-2^15, 2^15], whose low byte is the second digit + 128 and
// whose rest, floor((n + 128) / 256), is the first, in [-128, 128].  The remainder is exact and
// either 0 or at least twice the low word, so a fast two-sum renormalises it; units of 2^-14,
// 2^-30, 2^-46 give two digits each and 2^-54 the last.  A byte becomes a float as the low
// mantissa byte of 2^23 + byte: 24 packed FP32 instructions and 14 byte permutes per two values
// instead of 98 FP32 instructions for seven rounds of rint, subtract, renormalise and scale.
__device__ __forceinline__ void tc_digits2(df2 v, f32x2 s[TC_NS]) {
  const f32x2 m1 = f2_dup(0x1.8p9f + 0x1p-7f), m2 = f2_dup(0x1.8p-7f + 0x1p-23f);
  const f32x2 m3 = f2_dup(0x1.8p-23f + 0x1p-39f), m4 = f2_dup(0x1.8p-31f + 0x1p-40f);
  const f32x2 a = f2_add(v.hi, m1);
  f32x2 r = f2_sub(v.hi, f2_sub(a, m1));
  f32x2 h = f2_add(r, v.lo), l = f2_sub(v.lo, f2_sub(h, r));
  const f32x2 b = f2_add(h, m2);
  r = f2_sub(h, f2_sub(b, m2));
  h = f2_add(r, l);
  l = f2_sub(l, f2_sub(h, r));
  const f32x2 c = f2_add(h, m3);
  const f32x2 d = f2_add(f2_add(f2_sub(h, f2_sub(c, m3)), l), m4);
  // 2^23 + 2^14 + first digit; 2^23 + 128 + second digit; 2^23 + 2^14 + last digit
  const f32x2 off16 = f2_dup(-(0x1p23f + 0x1p14f)), off8 = f2_dup(-(0x1p23f + 128.0f));
  auto bytes = [](f32x2 x, unsigned sel) {
    return f2_pack(__uint_as_float(__byte_perm((unsigned)x, 0x4b000000u, sel)),
                   __uint_as_float(__byte_perm((unsigned)(x >> 32), 0x4b000000u, sel)));
  };
  s[0] = f2_add(bytes(a, 0x7621), off16);
  s[1] = f2_add(bytes(a, 0x7640), off8);
  s[2] = f2_add(bytes(b, 0x7621), off16);
  s[3] = f2_add(bytes(b, 0x7640), off8);
  s[4] = f2_add(bytes(c, 0x7621), off16);
  s[5] = f2_add(bytes(c, 0x7640), off8);
  s[6] = f2_add(bytes(d, 0x7610), off16);
}

// Two digits (integers, |d| <= 128: at most 8 significant bits, so the low 16 bits of their
// FP32 words are zero and the high halves are their exact bfloat16 encodings) packed as the
// bf16 pair (the low word's digit at the lower address).
__device__ __forceinline__ unsigned tc_pack(f32x2 d) {
  return __byte_perm((unsigned)d, (unsigned)(d >> 32), 0x7632);
}

// s + e += v with an error-free two-sum (v exact)
__device__ __forceinline__ void acc_add(dfacc2& a, f32x2 v) {
  const df2 s = df2_two_sum(a.s, v);
  a.s = s.hi;
  a.e = f2_add(a.e, s.lo);
}

__device__ __forceinline__ bool tc_in_range(df2 v) {   // false for NaN
  return fabsf(f2_lo(v.hi)) < 2.0f && fabsf(f2_hi(v.hi)) < 2.0f;
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace wmg
