// Exact fixed-point multiply-adds on the integer pipes, beside the FP64 pipe.
//
// GB300 issues two FP64 multiply-adds per clock and SM, so a sweep that does
// one per streamed 8-byte entry is bound by that pipe at 74 % of the HBM copy
// rate.  The integer pipes are idle meanwhile.  The level products therefore
// take 3 of every 8 columns' multiply-adds there: each product is the exact
// integer product of the two 53-bit significands, shifted to a common scale
// and added into a 128-bit accumulator per row (a long accumulator in
// Kulisch's sense, cut to 128 bits), rounded to FP64 once per block.  The sum
// of those columns then carries one rounding instead of one per column.
//
// Conditions, all checked, else the block goes through the FP64 pipe alone:
//   * block entries >= 0, finite, largest exponent not tiny: the block's largest
//     exponent field, known from set-up (block_exp);
//   * the same of the vector's entries: found while the vector is staged.
// A term is truncated below 2^-115 of (largest entry of the block) x (largest
// entry of the vector); a row whose sum is below 2^-51 of that product
// without being exactly zero cannot be rounded to FP64 accuracy from the
// window, and the level is then recomputed by FP64 multiply-adds alone.
#pragma once
#include <stdint.h>

#include "mc_internal.cuh"

namespace mc {
namespace dev {

// Smallest biased exponent of a block's (vector's) largest entry for which
// everything below the window is negligible, subnormal entries included.
constexpr int kMinFixedExp = 200;

// acc += (M * v) >> s, M = significand of the entry, v = (vh:vl) the 53-bit
// significand shifted left by 11, s = b - exponent(M) with b = exponent(block)
// + exponent(vector) - exponent(v) (clamped: the product is below 2^117, so
// 127 removes it; zero and subnormal entries have exponent 0 and land there).
// seen collects whether any entry was nonzero.
__device__ __forceinline__ void fixed_fma(uint32_t (&a)[4], uint32_t& seen, double M, uint32_t vl,
                                          uint32_t vh, int b) {
  const uint32_t hi = (uint32_t)__double2hiint(M), lo = (uint32_t)__double2loint(M);
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  const int s = min(b - (int)(hi >> 20), 127);
  seen |= hi | lo;
  const uint64_t t0 = (uint64_t)lo * vl;
  const uint64_t t1 = (uint64_t)mh * vl + (t0 >> 32);
  const uint64_t t2 = (uint64_t)lo * vh + (uint32_t)t1;
  const uint64_t t3 = (uint64_t)mh * vh + (t1 >> 32) + (t2 >> 32);
  uint32_t p0 = (uint32_t)t0, p1 = (uint32_t)t2, p2 = (uint32_t)t3, p3 = (uint32_t)(t3 >> 32);
  if (s & 64) {
    p0 = p2;
    p1 = p3;
    p2 = 0u;
    p3 = 0u;
  }
  if (s & 32) {
    p0 = p1;
    p1 = p2;
    p2 = p3;
    p3 = 0u;
  }
  p0 = __funnelshift_r(p0, p1, s);   // shifts by s mod 32
  p1 = __funnelshift_r(p1, p2, s);
  p2 = __funnelshift_r(p2, p3, s);
  p3 = __funnelshift_r(p3, 0u, s);
  asm("add.cc.u32 %0, %0, %4;\n\t"
      "addc.cc.u32 %1, %1, %5;\n\t"
      "addc.cc.u32 %2, %2, %6;\n\t"
      "addc.u32 %3, %3, %7;"
      : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
      : "r"(p0), "r"(p1), "r"(p2), "r"(p3));
}

// The accumulator as a double (one rounding); etot = exponent(block) +
// exponent(vector), biased both.  bad is set when the window cannot give FP64
// accuracy or the result leaves the normal range.
__device__ __forceinline__ double fixed_value(const uint32_t (&a)[4], uint32_t seen, int etot,
                                              bool& bad) {
  const uint64_t h = ((uint64_t)a[3] << 32) | a[2], l = ((uint64_t)a[1] << 32) | a[0];
  if (h == 0) {
    bad = bad || seen != 0u;
    return 0.0;
  }
  const int c = __clzll((long long)h);
  const uint64_t x = c ? (h << c) | (l >> (64 - c)) : h;
  const int e = etot - 1011 - c;          // biased exponent of the leading bit
  bad = bad || e < 1 || e > 2045;
  const uint64_t r = (x >> 11) + ((x >> 10) & 1u);   // 53 bits, rounded to nearest
  return __longlong_as_double((long long)(((uint64_t)(uint32_t)(e - 1) << 52) + r));
}

// Integer form of one vector entry: significand << 11 with the biased
// exponent in the low 11 bits.
__device__ __forceinline__ uint64_t fixed_entry(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint64_t s = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  return (s << 11) | ((hi >> 20) & 0x7ffu);
}

// e: largest exponent field (sign bit included: a negative entry reads as >= 2048)
// of a block's or a vector's entries.
__device__ __forceinline__ bool fixed_ok(int e) { return e >= kMinFixedExp && e < 2047; }

}  // namespace dev
}  // namespace mc
