// FP64 contractions on the tensor cores by exact integer slices (the error-free splitting of Ozaki,
// Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, in fixed point).
//
// Why: GB300 retires two FP64 FMAs per clock and SM, and the FP64 operator at p = 7 spends 77% of
// its FP64 instructions in the six 8 x 8 derivative passes.  Here a pass leaves that pipe:
//  * the values of a line v_m (m < Q <= 8) become integers X_m = v_m 2^(61 - E), |X_m| < 2^62, with E
//    the exponent of the line's largest value, and so does the matrix (once, at mesh setup);
//  * both are written in eight balanced base-256 digits (|digit| <= 128), which FP16 holds exactly;
//  * mma.sync m16n8k16 forms all digit products of equal weight: order s = sum over a + b = s of
//    X-digit a times M-digit b.  A sum has at most 8 * 8 products of at most 2^14, so FP32
//    accumulation is exact.  Orders 0 .. 7 are formed; the rest lies below 2^-60 of the result's scale
//    (seven digits and orders measured 4 to 10 times the error of the FMA chain, eight a third of it);
//  * the accumulators start at 1.5 * 2^23, so that their bit patterns are the integer sums plus a
//    constant, and one 64-bit integer sum of the eight orders, normalised and rounded once, is the
//    FP64 result: everything but the products runs on the integer pipe.
// The error is that of a dot product with the line cut at 62 bits below its largest value and one
// final rounding, smaller than that of the chain of FP64 FMAs (one rounding per term and fold).
// A line that holds an infinity or a NaN, or whose largest value is not zero and lies outside 2^-895 .. 2^877, takes
// plain FP64 FMAs instead.
//
// Fragments: a warp holds 16 lines; lane 4 g + t owns entries 2t, 2t+1 of lines g and g + 8, on the way
// in (A fragment: the digit of the pair as one half2) and on the way out (C fragment), so a pass
// needs no data exchange beyond the line maximum over four lanes.
#pragma once

#include <cuda_fp16.h>

#include "internal.h"

namespace ceedgb {

// Digit tables of one matrix for the B fragments: word [j * 32 + lane] holds digit j of M[g][2t]
// (low half) and M[g][2t + 1], g = lane / 4, t = lane % 4; M = integer * 2^-scale.
struct FixMat {
  uint32_t d[FIX_DIGITS];
  int scale;
};

__device__ __forceinline__ void fix_load(FixMat &M, const uint32_t *tab, int lane) {
#pragma unroll
  for (int j = 0; j < FIX_DIGITS; ++j) M.d[j] = __ldg(tab + j * 32 + lane);
  M.scale = (int)__ldg(tab + FIX_DIGITS * 32);
}

// The value as a 62-bit integer relative to 2^E (biased exponent E of the line's largest value),
// truncated, plus 128 in each digit, so that byte 7 - a of the result is digit a + 128.
__device__ __forceinline__ uint64_t fix_in(double v, int E) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const int sgn = hi >> 31;
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const uint64_t m = (((uint64_t)mh << 32) | (uint32_t)__double2loint(v)) << 9;
  const uint64_t x = m >> min(E - e, 63);
  const uint64_t s = ((uint64_t)(uint32_t)sgn << 32) | (uint32_t)sgn;
  return (x ^ s) + 0x8080808080808080ull;
}

// digit a of two values as half2 (1024 + 128 + digit, then the bias taken off: exact)
template <int A>
__device__ __forceinline__ uint32_t fix_digit(uint64_t y0, uint64_t y1) {
  constexpr int b = 7 - A;
  const uint32_t w0 = b >= 4 ? (uint32_t)(y0 >> 32) : (uint32_t)y0, w1 = b >= 4 ? (uint32_t)(y1 >> 32) : (uint32_t)y1;
  constexpr uint32_t k = b & 3;
  const uint32_t p = (__byte_perm(w0, w1, k | (k << 4) | ((4 + k) << 8) | ((4 + k) << 12)) & 0x00ff00ffu) | 0x64006400u;
  const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
  const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&p), bias);
  return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ void fix_digits(uint32_t (&d)[8], uint64_t y0, uint64_t y1) {
  d[0] = fix_digit<0>(y0, y1);
  d[1] = fix_digit<1>(y0, y1);
  d[2] = fix_digit<2>(y0, y1);
  d[3] = fix_digit<3>(y0, y1);
  d[4] = fix_digit<4>(y0, y1);
  d[5] = fix_digit<5>(y0, y1);
  d[6] = fix_digit<6>(y0, y1);
  d[7] = fix_digit<7>(y0, y1);
}

// exponent field of v 2^(61 - E) M 2^scale, the orders' sum at weight 2^(47 - 8 s) and the leading
// one at bit 62 (whose place in the field adds one): E - scale + 65
constexpr int FIX_EXP_OUT = 65;
constexpr uint32_t FIX_MAGIC = 0x4B400000u;  // bits of 1.5 * 2^23: bits(magic + n) = bits(magic) + n

// Eight orders (bit patterns of magic + sum) to FP64: sum_s u_s 2^(47 - 8 s), rounded once; eb is the
// exponent field of the sum's unit plus 62.  The sum stays below 2^63 if the table's entries of one product sum
// to less than 2^66 (eight entries always do).  Orders 6 and 7 are rounded to whole units, without bias
// and a zero to zero.
__device__ __forceinline__ double fix_out(const uint32_t (&u)[FIX_DIGITS], int eb) {
  constexpr uint64_t K = (uint64_t)FIX_MAGIC * ((1ull << 47) + (1ull << 39) + (1ull << 31) + (1ull << 23) + (1ull << 15) + (1ull << 7)) +
                         (uint64_t)((FIX_MAGIC + (FIX_MAGIC >> 8)) >> 1);
  uint64_t S = (uint64_t)((u[6] + (u[7] >> 8) + 1u) >> 1) + (uint64_t)u[5] * (1u << 7);
  S += (uint64_t)u[4] * (1u << 15);
  S += (uint64_t)u[3] * (1u << 23);
  S += (uint64_t)u[2] * (1u << 31);
  const uint64_t A = S + ((uint64_t)((u[1] << 7) + (u[0] << 15)) << 32) - K;
  const int64_t sgn = (int64_t)A >> 63;
  const uint64_t B = (A ^ (uint64_t)sgn) - (uint64_t)sgn;  // |A|
  uint32_t hi = (uint32_t)(B >> 32), lo = (uint32_t)B;
  const bool low = hi == 0u;
  if (low) {  // below 2^32: its last bit, 2^-63 of the sum's range, is dropped
    hi = lo >> 1;
    lo = 0u;
  }
  const int n = __clz(hi) - 1;  // top bit to bit 62
  uint64_t N = (((uint64_t)hi << 32) | lo) << n;
  N += 0x200u;                                   // half of the last kept bit: round to nearest
  const int e = (low ? eb - 31 : eb) - n;
  const uint32_t dh = (uint32_t)(N >> 42) + ((uint32_t)e << 20);
  const uint32_t dl = (uint32_t)(N >> 10);
  return hi == 0u ? 0.0 : __hiloint2double((int)(dh | ((uint32_t)(sgn >> 32) & 0x80000000u)), (int)dl);
}

// Biased exponent E of the largest of the values whose high words' magnitudes have the maximum m (64 for
// all zero: every digit is then zero), and whether it lies outside the integer range (128 .. 1900).  High words all zero
// are zeros or subnormals below 2^-1042; the latter (fix_tiny) lie outside as well.
__device__ __forceinline__ int fix_exponent(int m) { return max(m >> 20, 64); }
__device__ __forceinline__ bool fix_odd_or_zero(int m) { return (uint32_t)(m - (128 << 20)) >= (uint32_t)(1901 - 128) << 20; }
__device__ __forceinline__ int fix_mag(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ bool fix_tiny(double v0, double v1) { return (__double2loint(v0) | __double2loint(v1)) != 0; }

// maximum over the four lanes that hold a line
__device__ __forceinline__ int fix_quad_max(int m) {
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
  return max(m, __shfl_xor_sync(0xffffffffu, m, 2));
}

__device__ __forceinline__ void fix_mma_start(uint32_t (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(FIX_MAGIC));
}

__device__ __forceinline__ void fix_mma(uint32_t (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// acc[s] (+)= the digit products of order s (digits a of x times s - a of b) over eight entries: x0, x1 the
// digits of lines g and g + 8, b the table's.  One product takes two digits of x: a in k slots 0..7,
// a + 1 in slots 8..15.  FIRST: the sums start here, from the magic constant (as the product's own addend:
// 32 register moves less than setting the accumulators beforehand).
template <bool FIRST>
__device__ __forceinline__ void fix_products(uint32_t (&acc)[FIX_DIGITS][4], const uint32_t (&x0)[8], const uint32_t (&x1)[8],
                                             const uint32_t (&b)[FIX_DIGITS]) {
#pragma unroll
  for (int s = 0; s < FIX_DIGITS; ++s)
#pragma unroll
    for (int a = 0; a <= s; a += 2) {
      const uint32_t lo = b[s - a], hi = s > a ? b[s - a - 1] : 0u;
      if (FIRST && a == 0) fix_mma_start(acc[s], x0[a], x1[a], x0[a + 1], x1[a + 1], lo, hi);
      else fix_mma(acc[s], x0[a], x1[a], x0[a + 1], x1[a + 1], lo, hi);
    }
}

// out = M v (M NO x NI, both at most 8) on the warp's 16 lines: v[0], v[1] = entries 2t, 2t+1 of line g, v[2], v[3] of line g + 8
// (zero past the line's length); out laid out alike.  full(n, m): M's entry in FP64, for lines outside
// the integer range.  Every lane of the warp takes part.
template <int NI, int NO, typename Full>
__device__ __forceinline__ void fix_pass(const FixMat &M, const double (&v)[4], double (&out)[4], Full full) {
  const int m0 = fix_quad_max(max(fix_mag(v[0]), fix_mag(v[1]))), m1 = fix_quad_max(max(fix_mag(v[2]), fix_mag(v[3])));
  const int E0 = fix_exponent(m0), E1 = fix_exponent(m1);
  // (in two steps: lines of zeros are common, and the second is left out where there is none)
  if (__any_sync(0xffffffffu, fix_odd_or_zero(m0) || fix_odd_or_zero(m1)) &&
      __any_sync(0xffffffffu, (fix_odd_or_zero(m0) && (m0 != 0 || fix_tiny(v[0], v[1]))) ||
                                  (fix_odd_or_zero(m1) && (m1 != 0 || fix_tiny(v[2], v[3]))))) {
    const int lane = threadIdx.x & 31, t = lane & 3, q = lane & ~3;
    double r[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int m = 0; m < NI; ++m) {
      const double a0 = __shfl_sync(0xffffffffu, (m & 1) ? v[1] : v[0], q + (m >> 1));
      const double a1 = __shfl_sync(0xffffffffu, (m & 1) ? v[3] : v[2], q + (m >> 1));
      const double f0 = 2 * t < NO ? full(2 * t, m) : 0.0, f1 = 2 * t + 1 < NO ? full(2 * t + 1, m) : 0.0;
      r[0] = fma(f0, a0, r[0]);
      r[1] = fma(f1, a0, r[1]);
      r[2] = fma(f0, a1, r[2]);
      r[3] = fma(f1, a1, r[3]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = r[k];
    return;
  }
  uint32_t x0[8], x1[8];
  fix_digits(x0, fix_in(v[0], E0), fix_in(v[1], E0));
  fix_digits(x1, fix_in(v[2], E1), fix_in(v[3], E1));
  uint32_t acc[FIX_DIGITS][4];
  fix_products<true>(acc, x0, x1, M.d);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    uint32_t u[FIX_DIGITS];
#pragma unroll
    for (int s = 0; s < FIX_DIGITS; ++s) u[s] = acc[s][k];
    out[k] = fix_out(u, (k < 2 ? E0 : E1) - M.scale + FIX_EXP_OUT);
  }
}

}  // namespace ceedgb
