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
// Conditions, decided before a block is streamed, else it goes through the FP64
// pipe alone (fixed_safe):
//   * entries of block and vector >= 0 and finite;
//   * no row can leave the window.  A term is truncated below 2^-115 of (largest
//     entry of the block) x (largest entry of the vector), so a row's sum must
//     be zero or at least 2^-52 of that product.  The exponents of the block
//     (block_exp) and of the vector (found while it is staged) bound it: a row
//     has its largest entry times the vector's smallest, or, where the vector
//     has zeros, no nonzero term below the smallest entries' product.
// So a block is never streamed twice (a row found short used to send its block
// through the FP64 pipe after all), and nothing is tested per entry.  16 sweeps of
// 6000 levels of 64, inverse: phases in geometric proportion over 2^149 3.20 -> 1.95 ms
// (one warp per level on the FP64 pipe alone: 2.03), half the phases of zero
// probability 2.31 -> 1.41 (2.03); 64 sweeps of 32768 x 64 29.92 -> 29.48 ms.
#pragma once
#include <stdint.h>

#include "mc_internal.cuh"

namespace mc {
namespace dev {

// acc += (M * v) >> s, M = significand of the entry, v = (vh:vl) the 53-bit
// significand shifted left by 11, s = b - exponent(M) with b = exponent(block)
// + exponent(vector) - exponent(v) (clamped: the product is below 2^117, so
// 127 removes it; zero and subnormal entries have exponent 0 and land there).
// seen (optional) collects whether any entry was nonzero.
__device__ __forceinline__ void fixed_fma(uint32_t (&a)[4], double M, uint32_t vl, uint32_t vh,
                                          int b, uint32_t* seen = nullptr) {
  const uint32_t hi = (uint32_t)__double2hiint(M), lo = (uint32_t)__double2loint(M);
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
  const int s = min(b - (int)(hi >> 20), 127);
  if (seen) *seen |= hi | lo;
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
// exponent(vector), biased both.  bad is set when entries were seen and the window
// cannot give FP64 accuracy, or the result leaves the normal range.
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

// The same as one part of a row that fixed_safe allows: nothing to report, and no
// branch (lanes without a row have empty accumulators: 20000 levels of 24, inverse, 16
// sweeps 1.45 -> 1.42 ms).
__device__ __forceinline__ double fixed_part(const uint32_t (&a)[4], int etot) {
  const uint64_t a1 = ((uint64_t)a[3] << 32) | a[2], a0 = ((uint64_t)a[1] << 32) | a[0];
  const bool low = a1 == 0;
  const uint64_t h = low ? a0 : a1, l = low ? 0ull : a0;
  const int c = __clzll((long long)h), e = (low ? etot - 64 : etot) - 1011 - c;
  const uint64_t x = (h << (c & 63)) | ((l >> 1) >> (63 - (c & 63)));
  const uint64_t r = (x >> 11) + ((x >> 10) & 1u);
  return h == 0 ? 0.0 : __longlong_as_double((long long)(((uint64_t)(uint32_t)(e - 1) << 52) + r));
}

// Integer form of one vector entry: significand << 11 with the biased
// exponent in the low 11 bits.
__device__ __forceinline__ uint64_t fixed_entry(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint64_t s = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  return (s << 11) | ((hi >> 20) & 0x7ffu);
}

// Exponents of a set of entries, packed: the largest exponent field (sign bit
// included: a negative entry reads as >= 2048) in bits 0..11, 4096 - the smallest one
// of a nonzero entry in bits 12..24 (0: no nonzero entry), whether there is a zero
// in bit 25.  Maxima and ors only, so sets join field by field.
__device__ __forceinline__ unsigned exp_field(double x) {
  return (unsigned)__double2hiint(x) >> 20;
}
__device__ __forceinline__ bool is_zero(double x) {   // (-0 is left to the sign)
  return (__double2hiint(x) | __double2loint(x)) == 0;
}
__device__ __forceinline__ unsigned exp_low(double x) {
  return is_zero(x) ? 0u : 4096u - exp_field(x);
}
__device__ __forceinline__ int exp_pack(unsigned most, unsigned low, bool zero) {
  return (int)(most | low << 12 | (zero ? 1u << 25 : 0u));
}
__device__ __forceinline__ int exp_join(int a, int b) {
  return max(a & 0xfff, b & 0xfff) | max(a & 0x1fff000, b & 0x1fff000) | ((a | b) & (1 << 25));
}

// Whether no row of block * vector can leave the window or the normal range
// (block: its block_exp).
__device__ __forceinline__ bool fixed_safe(int2 block, int vec) {
  const int most = block.x, vmost = vec & 0xfff, vlow = (vec >> 12) & 0x1fff;
  const int rows = block.y >> 16, low = (vec >> 25) || rows == 0 ? block.y & 0xffff : rows;
  return most < 2047 && vmost < 2047 && low > 0 && vlow > 0 &&
         most + low + vmost + vlow <= 8192 + 51 &&   // row >= 2^64 units of the accumulator
         low + vlow <= 8192 - 1030 && most + vmost <= 3040;
}

// As above for one sum of products of two blocks' entries (coupled operators, which
// test each entry): both largest entries.
__device__ __forceinline__ bool fixed_ok(int e) { return e >= 200 && e < 2047; }

}  // namespace dev
}  // namespace mc
