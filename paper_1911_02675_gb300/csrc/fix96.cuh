// fix96.cuh -- FP64 additions on the integer pipe: 96-bit block fixed point.
//
// The FP64 pipe of this part does ~1.75 additions per clock per SM, the integer pipe 64 to 114.
// Where a sum only adds and subtracts FP64 values (the Hadamard transform), a block of values is
// written as integers on one scale, added exactly, and rounded back to FP64 once:
//   V = M 2^(31 - (emax - e)),  x = V 2^(emax - 1106),
// M the 53-bit mantissa and e the exponent field of x, emax the largest exponent field of the
// block.  |V| < 2^84, so 2^11 of them add without overflow; a value loses only bits below 2^-84 of
// the block's largest, where an FP64 evaluation rounds at 2^-53 of every partial sum that the largest
// element is in.
#pragma once

#include <stdint.h>

namespace lsq_fix {

constexpr int EXP_SPECIAL = 0x7FF;  // exponent field of infinities and NaNs

struct i96 {
  uint32_t w0, w1, w2;
};

__device__ __forceinline__ i96 add(i96 a, i96 b) {
  i96 r;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=r"(r.w0), "=r"(r.w1), "=r"(r.w2)
      : "r"(a.w0), "r"(a.w1), "r"(a.w2), "r"(b.w0), "r"(b.w1), "r"(b.w2));
  return r;
}

__device__ __forceinline__ i96 sub(i96 a, i96 b) {
  i96 r;
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
      : "=r"(r.w0), "=r"(r.w1), "=r"(r.w2)
      : "r"(a.w0), "r"(a.w1), "r"(a.w2), "r"(b.w0), "r"(b.w1), "r"(b.w2));
  return r;
}

// v, or -v where mask is all ones
__device__ __forceinline__ i96 negate_if(i96 v, uint32_t mask) {
  return sub(i96{v.w0 ^ mask, v.w1 ^ mask, v.w2 ^ mask}, i96{mask, mask, mask});
}

// magnitude bits whose maximum over a block gives its scale (one word: the order of the high
// words is that of the exponents), and the scale of that maximum: the exponent field on the FP64
// scale, 1 for a block of zeros and subnormals, EXP_SPECIAL if an infinity or a NaN is there
__device__ __forceinline__ uint32_t mag_bits(double x) { return (uint32_t)__double2hiint(x) & 0x7FFFFFFFu; }
__device__ __forceinline__ uint32_t mag_bits(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
template <typename T>
__device__ __forceinline__ int scale_of(uint32_t mag) {
  if (sizeof(T) == 8) return max((int)(mag >> 20), 1);
  const int e = (int)(mag >> 23);
  return e == 0xFF ? EXP_SPECIAL : max(e, 1) + 896;
}

// v >> delta; the elements of a block within 2^31 of its largest take the short way
__device__ __forceinline__ i96 shift_right(i96 v, int delta) {
  if (delta >= 32) {
    if (delta & 64) v = i96{v.w2, 0u, 0u};
    if (delta & 32) v = i96{v.w1, v.w2, 0u};
    if (delta >= 128) v = i96{0u, 0u, 0u};
  }
  return i96{__funnelshift_r(v.w0, v.w1, delta), __funnelshift_r(v.w1, v.w2, delta), v.w2 >> (delta & 31)};
}

// a finite x on the scale emax >= exp_field(x), negated where flip is all ones
__device__ __forceinline__ i96 to_fix(double x, int emax, uint32_t flip) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7FFu);
  const uint32_t mh = (hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
  const i96 v{lo << 31, (mh << 31) | (lo >> 1), mh >> 1};
  return negate_if(shift_right(v, emax - max(e, 1)), flip ^ (uint32_t)((int32_t)hi >> 31));
}
__device__ __forceinline__ i96 to_fix(float x, int emax, uint32_t flip) {
  const uint32_t u = __float_as_uint(x);
  const int e = (int)((u >> 23) & 0xFFu);
  const uint32_t m = (u & 0x7FFFFFu) | (e ? 0x800000u : 0u);
  const i96 v{0u, m << 28, m >> 4};
  return negate_if(shift_right(v, emax - (max(e, 1) + 896)), flip ^ (uint32_t)((int32_t)u >> 31));
}

// v 2^(emax - 1106) rounded to FP64 (nearest, ties to even), negated where flip is all ones
__device__ __forceinline__ double from_fix(i96 v, int emax, uint32_t flip) {
  const uint32_t sg = (uint32_t)((int32_t)v.w2 >> 31);
  v = negate_if(v, sg);
  if ((v.w0 | v.w1 | v.w2) == 0u) return 0.0;
  const bool top2 = v.w2 != 0u, top1 = v.w1 != 0u;
  const uint32_t x2 = top2 ? v.w2 : (top1 ? v.w1 : v.w0);
  const uint32_t x1 = top2 ? v.w1 : (top1 ? v.w0 : 0u);
  const uint32_t x0 = top2 ? v.w0 : 0u;
  const int s = __clz((int)x2);
  const uint32_t h = __funnelshift_l(x1, x2, s), l = __funnelshift_l(x0, x1, s), rest = x0 << s;
  // exponent field of the leading bit (bit 95 - s, 32 lower per empty word)
  const int be = 95 - s - (top2 ? 0 : (top1 ? 32 : 64)) + emax - 83;
  const uint32_t rb = l & 0x7FFu;
  unsigned long long m = (((unsigned long long)h << 32) | l) >> 11;
  m += (rb > 0x400u || (rb == 0x400u && (rest != 0u || (m & 1ull)))) ? 1ull : 0ull;
  const unsigned long long sign = (unsigned long long)((sg ^ flip) & 0x80000000u) << 32;
  if (be <= 0)  // subnormal: scaled up by 2^128 and back
    return __longlong_as_double((long long)(sign | (((unsigned long long)(be + 127) << 52) + m))) * 0x1p-128;
  const unsigned long long bits = ((unsigned long long)(be - 1) << 52) + m;
  return __longlong_as_double((long long)(sign | (bits < 0x7FF0000000000000ull ? bits : 0x7FF0000000000000ull)));
}

}  // namespace lsq_fix
