// Non-tensor operator in FP64 with both basis contractions on the tensor cores as exact integer slices
// (fixmma.cuh), fused: gather, G u, pointwise D, G^T v, element vectors out.
//
// Why: at degree 4 on tetrahedra (35 nodes, 125 points) an element costs 26,250 FP64 FMAs in the two
// contractions and 1,125 in the pointwise step, at two per clock and SM; with the contractions off the
// FP64 pipe, the digit products (about 600 mma.sync m16n8k16 per element) and the integer work that
// splits inputs and joins orders (about 50 thousand lane instructions) bound it.
//
// A warp holds 16 elements; the lines of fixmma.cuh are its elements.  It walks the points in groups of
// eight: forward, three 8-point tiles (one per derivative) over the nodes in chunks of eight, all against
// one exponent per element; a thread then has the three derivatives at two points of two elements,
// applies the pointwise D to them, and has the operands of the transposed product in place: the group's
// 24 values per element, against one exponent per element and group, times five 8-node tiles.  Each
// group's result is joined to FP64 and added to the nodes' sums in registers.  Digits of the inputs are kept in
// shared memory, the tables come through L1 (each block's warps walk them together).
// Integer sums stay below 2^22: forward at most 35 nodes (6 pairs of digits of at most 128, 2 with a
// leading digit of at most 64), transposed 24 values.
//
// Precision: the slices' error is relative to the largest value and the largest table entry, that of a chain of FP64
// FMAs to the sum S of its terms' magnitudes.  A basis may be any, with zeros or small entries where an element's
// large values are, so S is measured: the leading digits' magnitudes, multiplied by one more mma per product.  Both errors
// emulated in exact arithmetic on random digits, root mean square: slices 2.2, 2.6, 3.3, 4.8 x 2^-60 of (largest value x
// largest entry, as powers of two) for 2, 4, 8, 35 terms; chain 0.48 x 2^-53 S.  They meet at S = 0.04 to 0.08 of that
// product (leading digits of 32 to 63 stand for the largest values: at 40 to 80).  What counts is a node's result: the
// points' margins (the smallest of the derivatives' S less that bound, times D's diagonal) go through the transposed
// product with the table's magnitudes, and an element in which a node's sum of them falls below the groups' own errors is
// put on a list and computed again by nt_fused_kernel, as are those with values outside the integers' range.
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "fixmma.cuh"
#include "nontensor.h"

namespace ceedgb {

constexpr int NTF_WARPS = 4;
// Blocks per SM by node chunks: the warps of a group's chain of passes wait on one another's results most of the time, so
// more of them pay for some spilled registers (diffusion of degree 4: 1.58 ms with two blocks, 1.09 with three, 1.21 with four;
// degrees 1 to 3: 0.57, 0.65, 0.76 ms with three, 0.49, 0.59, 0.69 with four).
constexpr int ntf_blocks(int nc) { return nc > 4 ? 3 : 4; }

bool nt_fix_supported(ceed_nt_t h, int op) { return h->d_fix[op == CEED_OP_MASS ? 0 : 1] != nullptr; }

// Leading-digit sums below which an element is computed by FMAs: a product over the element's nodes; and over all groups,
// relative to the root of the sum of the groups' squared scales (a group's error is independent of the others').
constexpr float ntf_least(int terms) { return 40.f + 1.2f * (float)terms; }
constexpr float NTF_LEAST_GROUPS = 72.f;
constexpr int NTF_GROUP_SPREAD = 60;  // a group's scale may exceed the first one's by this power of two

struct NtFixArgs {
  int64_t E, Es;
  int P, Q, ngroups;
  const uint32_t *rmap;   // [P][E]
  const double *x;
  const uint4 *fwd, *bwd; // [group][D][chunk][lane][2]: eight digit words of the B fragments
  int fwd_scale, bwd_scale;
  uint32_t *again;        // [1 + E]: number and list of the elements to be computed by FMAs
  const double *qd;       // [D == 1 ? 1 : 6][Q][Es]
  double *Ye;             // [P][E]
  int masked;
};

__device__ __forceinline__ void ntf_load(uint32_t (&b)[FIX_DIGITS], const uint4 *p) {
  const uint4 lo = __ldg(p), hi = __ldg(p + 1);
  b[0] = lo.x, b[1] = lo.y, b[2] = lo.z, b[3] = lo.w;
  b[4] = hi.x, b[5] = hi.y, b[6] = hi.z, b[7] = hi.w;
}

__device__ __forceinline__ double ntf_node(const NtFixArgs &a, int n, int64_t e) {
  const uint32_t m = __ldg(a.rmap + (int64_t)n * a.E + e);
  return (a.masked && (m & FLAG_DIR)) ? 0.0 : __ldg(a.x + (m & DOF_MASK));
}

// D at point q of element e: v becomes the flux (mass: the weighted value); diag: D's diagonal.
template <int D>
__device__ __forceinline__ void ntf_pointwise(const NtFixArgs &a, int q, int64_t e, double (&v)[D], float (&diag)[D]) {
  const double *qd = a.qd + (int64_t)q * a.Es + e;
  const int64_t cs = (int64_t)a.Q * a.Es;
  if constexpr (D == 1) {
    const double c = __ldg(qd);
    v[0] *= c;
    diag[0] = fabsf((float)c);
  } else {
    const double c0 = __ldg(qd), c1 = __ldg(qd + cs), c2 = __ldg(qd + 2 * cs), c3 = __ldg(qd + 3 * cs);
    const double c4 = __ldg(qd + 4 * cs), c5 = __ldg(qd + 5 * cs);
    const double g0 = v[0], g1 = v[1], g2 = v[2];
    v[0] = c0 * g0 + c1 * g1 + c2 * g2;
    v[1] = c1 * g0 + c3 * g1 + c4 * g2;
    v[2] = c2 * g0 + c4 * g1 + c5 * g2;
    diag[0] = fabsf((float)c0);
    diag[1] = fabsf((float)c3);
    diag[2] = fabsf((float)c5);
  }
}

// c (+)= x0, x1 (FP16 pairs of lines g and g + 8) times the magnitudes of the leading digits of b.
template <bool FIRST>
__device__ __forceinline__ void ntf_magnitudes(float (&c)[4], uint32_t x0, uint32_t x1, uint32_t b) {
  if (FIRST) c[0] = c[1] = c[2] = c[3] = 0.f;
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(x0), "r"(x1), "r"(b & 0x7fff7fffu));
}

__device__ __forceinline__ float ntf_pow2(int n) { return __int_as_float((127 + max(-126, min(n, 127))) << 23); }

// two values as an FP16 pair, within its range
__device__ __forceinline__ uint32_t ntf_pair(float a, float b) {
  const __half2 h = __floats2half2_rn(fmaxf(-6e4f, fminf(a, 6e4f)), fmaxf(-6e4f, fminf(b, 6e4f)));
  return *reinterpret_cast<const uint32_t *>(&h);
}

template <int NC>
constexpr size_t ntf_smem() {
  return (size_t)NTF_WARPS * NC * 5 * 32 * sizeof(uint4);
}

template <int D, int NC>
__global__ void __launch_bounds__(32 * NTF_WARPS, ntf_blocks(NC)) nt_fix_kernel(const NtFixArgs a) {
  extern __shared__ __align__(128) uint4 ntf_sh[];
  uint4 (*dig_sh)[NC][4][32] = reinterpret_cast<uint4 (*)[NC][4][32]>(ntf_sh);   // digits of the inputs: lines g (words 0..7), g + 8
  float4 (*mag_sh)[NC][32] = reinterpret_cast<float4 (*)[NC][32]>(ntf_sh + NTF_WARPS * NC * 4 * 32);  // the nodes' sums of magnitudes
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t2 = (lane & 3) * 2;
  const int64_t e0 = ((int64_t)blockIdx.x * NTF_WARPS + warp) * 16;
  const int64_t e[2] = {e0 + g, e0 + g + 8};
  const bool valid[2] = {e[0] < a.E, e[1] < a.E};
  int E0, E1;
  bool plain0, plain1;  // my elements to be computed by FMAs, as far as this lane knows
  {
    double u[NC][4];
    int m0 = 0, m1 = 0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int n = 8 * c + t2 + (k & 1);
        u[c][k] = (n < a.P && valid[k >> 1]) ? ntf_node(a, n, e[k >> 1]) : 0.0;
      }
      m0 = max(m0, max(fix_mag(u[c][0]), fix_mag(u[c][1])));
      m1 = max(m1, max(fix_mag(u[c][2]), fix_mag(u[c][3])));
    }
    m0 = fix_quad_max(m0);
    m1 = fix_quad_max(m1);
    E0 = fix_exponent(m0);
    E1 = fix_exponent(m1);
    bool t0 = false, t1 = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      t0 |= fix_tiny(u[c][0], u[c][1]);
      t1 |= fix_tiny(u[c][2], u[c][3]);
    }
    const int tiny0 = fix_quad_max(t0), tiny1 = fix_quad_max(t1);
    plain0 = fix_odd_or_zero(m0) && (m0 != 0 || tiny0 != 0);
    plain1 = fix_odd_or_zero(m1) && (m1 != 0 || tiny1 != 0);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      mag_sh[warp][c][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      uint32_t x0[8], x1[8];
      fix_digits(x0, fix_in(u[c][0], E0), fix_in(u[c][1], E0));
      fix_digits(x1, fix_in(u[c][2], E1), fix_in(u[c][3], E1));
      dig_sh[warp][c][0][lane] = make_uint4(x0[0], x0[1], x0[2], x0[3]);
      dig_sh[warp][c][1][lane] = make_uint4(x0[4], x0[5], x0[6], x0[7]);
      dig_sh[warp][c][2][lane] = make_uint4(x1[0], x1[1], x1[2], x1[3]);
      dig_sh[warp][c][3][lane] = make_uint4(x1[4], x1[5], x1[6], x1[7]);
    }
  }
  double y[NC][4];
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) y[c][k] = 0.0;
  const float least = ntf_least(a.P);
  int R0 = 0, R1 = 0;            // exponents of the first groups that are not zero: the magnitudes' unit
  float ww0 = 0.f, ww1 = 0.f;    // sums of the groups' squared scales

#pragma unroll 1
  for (int i = 0; i < a.ngroups; ++i) {
    __syncthreads();  // the block's warps read the same tables at the same time
    const uint4 *tf = a.fwd + ((int64_t)i * D * NC * 32 + lane) * 2, *tb = a.bwd + ((int64_t)i * D * NC * 32 + lane) * 2;
    double v[D][4];
    float margin[4], flux[D][4];   // of my points: the smallest S less the bound; that times D's diagonal
#pragma unroll
    for (int d = 0; d < D; ++d) {
      uint32_t acc[FIX_DIGITS][4];
      float mag[4];
      const auto chunk = [&](auto first, int c) {
        const uint4 q0 = dig_sh[warp][c][0][lane], q1 = dig_sh[warp][c][1][lane];
        const uint4 q2 = dig_sh[warp][c][2][lane], q3 = dig_sh[warp][c][3][lane];
        const uint32_t x0[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
        const uint32_t x1[8] = {q2.x, q2.y, q2.z, q2.w, q3.x, q3.y, q3.z, q3.w};
        uint32_t b[FIX_DIGITS];
        ntf_load(b, tf + (d * NC + c) * 64);
        fix_products<decltype(first)::value>(acc, x0, x1, b);
        ntf_magnitudes<decltype(first)::value>(mag, x0[0] & 0x7fff7fffu, x1[0] & 0x7fff7fffu, b[0]);
      };
      chunk(std::true_type(), 0);
#pragma unroll 1
      for (int c = 1; c < NC; ++c) chunk(std::false_type(), c);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t w[FIX_DIGITS];
#pragma unroll
        for (int s = 0; s < FIX_DIGITS; ++s) w[s] = acc[s][k];
        v[d][k] = fix_out(w, (k < 2 ? E0 : E1) - a.fwd_scale + FIX_EXP_OUT);
        margin[k] = d == 0 ? mag[k] : fminf(margin[k], mag[k]);
      }
    }
    // pointwise D at my two points of my two elements
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = 8 * i + t2 + (k & 1);
      double p[D];
      float diag[D];
#pragma unroll
      for (int d = 0; d < D; ++d) p[d] = v[d][k];
      if (q < a.Q && valid[k >> 1]) {
        ntf_pointwise<D>(a, q, e[k >> 1], p, diag);
      } else {
#pragma unroll
        for (int d = 0; d < D; ++d) p[d] = 0.0, diag[d] = 0.f;
      }
      const float over = margin[k] - least;  // (below the bound all of D's row spreads the error: three times)
#pragma unroll
      for (int d = 0; d < D; ++d) {
        v[d][k] = p[d];
        flux[d][k] = diag[d] * (over < 0.f ? 3.f * over : over);
      }
    }
    // transposed product of the group
    int m0 = 0, m1 = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      m0 = max(m0, max(fix_mag(v[d][0]), fix_mag(v[d][1])));
      m1 = max(m1, max(fix_mag(v[d][2]), fix_mag(v[d][3])));
    }
    m0 = fix_quad_max(m0);
    m1 = fix_quad_max(m1);
    const bool o0 = fix_odd_or_zero(m0), o1 = fix_odd_or_zero(m1);
    if (__any_sync(0xffffffffu, o0 || o1)) {  // (lanes whose own values are zero leave it to the others)
#pragma unroll
      for (int d = 0; d < D; ++d) {
        plain0 = plain0 || (o0 && (m0 != 0 || fix_tiny(v[d][0], v[d][1])));
        plain1 = plain1 || (o1 && (m1 != 0 || fix_tiny(v[d][2], v[d][3])));
      }
    }
    {
      const int F0 = fix_exponent(m0), F1 = fix_exponent(m1);
      // the groups' scales in units of the first one's; a group of zeros adds nothing, one far below the first
      // neither magnitudes nor error
      if (R0 == 0 && m0 != 0) R0 = F0;
      if (R1 == 0 && m1 != 0) R1 = F1;
      const int s0 = F0 - R0, s1 = F1 - R1;
      plain0 = plain0 || (m0 != 0 && s0 > NTF_GROUP_SPREAD);
      plain1 = plain1 || (m1 != 0 && s1 > NTF_GROUP_SPREAD);
      const float w0 = m0 != 0 && s0 > -NTF_GROUP_SPREAD ? ntf_pow2(min(s0, NTF_GROUP_SPREAD)) : 0.f;
      const float w1 = m1 != 0 && s1 > -NTF_GROUP_SPREAD ? ntf_pow2(min(s1, NTF_GROUP_SPREAD)) : 0.f;
      ww0 = fmaf(w0, w0, ww0);
      ww1 = fmaf(w1, w1, ww1);
      // margins in the unit of the group's leading digits
      const float unit0 = ntf_pow2(E0 - F0 + 56 - a.fwd_scale), unit1 = ntf_pow2(E1 - F1 + 56 - a.fwd_scale);
      uint32_t x0[D][8], x1[D][8], f0[D], f1[D];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        f0[d] = ntf_pair(flux[d][0] * unit0, flux[d][1] * unit0);
        f1[d] = ntf_pair(flux[d][2] * unit1, flux[d][3] * unit1);
        fix_digits(x0[d], fix_in(v[d][0], F0), fix_in(v[d][1], F0));
        fix_digits(x1[d], fix_in(v[d][2], F1), fix_in(v[d][3], F1));
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        uint32_t acc[FIX_DIGITS][4];
        float mag[4];
#pragma unroll
        for (int d = 0; d < D; ++d) {
          uint32_t b[FIX_DIGITS];
          ntf_load(b, tb + (d * NC + c) * 64);
          if (d == 0) {
            fix_products<true>(acc, x0[d], x1[d], b);
            ntf_magnitudes<true>(mag, f0[d], f1[d], b[0]);
          } else {
            fix_products<false>(acc, x0[d], x1[d], b);
            ntf_magnitudes<false>(mag, f0[d], f1[d], b[0]);
          }
        }
        float4 &sum = mag_sh[warp][c][lane];
        sum = make_float4(fmaf(mag[0], w0, sum.x), fmaf(mag[1], w0, sum.y), fmaf(mag[2], w1, sum.z), fmaf(mag[3], w1, sum.w));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint32_t w[FIX_DIGITS];
#pragma unroll
          for (int s = 0; s < FIX_DIGITS; ++s) w[s] = acc[s][k];
          y[c][k] += fix_out(w, (k < 2 ? F0 : F1) - a.bwd_scale + FIX_EXP_OUT);
        }
      }
    }
  }
  const float least0 = NTF_LEAST_GROUPS * sqrtf(ww0), least1 = NTF_LEAST_GROUPS * sqrtf(ww1);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const float4 sum = mag_sh[warp][c][lane];
    const int n = 8 * c + t2;
    plain0 = plain0 || (n < a.P && sum.x < least0) || (n + 1 < a.P && sum.y < least0);
    plain1 = plain1 || (n < a.P && sum.z < least1) || (n + 1 < a.P && sum.w < least1);
  }
  const int p0 = fix_quad_max(plain0 && valid[0]), p1 = fix_quad_max(plain1 && valid[1]);
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int n = 8 * c + t2 + (k & 1);
      if (n < a.P && valid[k >> 1] && !(k < 2 ? p0 : p1)) a.Ye[(int64_t)n * a.E + e[k >> 1]] = y[c][k];
    }
  if ((lane & 3) == 0) {  // (the order of the list does not matter: an element's result is its own)
    if (p0) a.again[1 + atomicAdd(a.again, 1u)] = (uint32_t)e[0];
    if (p1) a.again[1 + atomicAdd(a.again, 1u)] = (uint32_t)e[1];
  }
}

// Whether the slices serve a D x Q x P table, and its scales: forward (sums over an element's nodes) and transposed (sums
// over a group's points and derivatives).  Entries of one product sum to less than 2^66 (fix_out's sum below 2^63).  Not
// served: tables whose entries are not finite or so large or small that results could leave fix_out's exponents, and
// those in which a row has fewer than two entries within a factor of 16 of the table's largest (a nodal basis at its own
// nodes): most elements would be computed twice.
static bool nt_fix_scales(const double *M, int D, int Q, int P, int *fwd, int *bwd) {
  double most = 0, row = 0, col = 0;
  for (size_t k = 0; k < (size_t)D * Q * P; ++k) {
    if (!std::isfinite(M[k])) return false;
    most = std::max(most, std::fabs(M[k]));
  }
  if (most == 0) return false;
  for (int d = 0; d < D; ++d)
    for (int q = 0; q < Q; ++q) {
      double sum = 0;
      int large = 0;
      for (int n = 0; n < P; ++n) {
        const double v = std::fabs(M[((size_t)d * Q + q) * P + n]);
        sum += v;
        large += v >= most / 16;
      }
      row = std::max(row, sum);
      if (large < 2) return false;
    }
  for (int q0 = 0; q0 < Q; q0 += 8)
    for (int n = 0; n < P; ++n) {
      double sum = 0;
      for (int d = 0; d < D; ++d)
        for (int q = q0; q < std::min(Q, q0 + 8); ++q) sum += std::fabs(M[((size_t)d * Q + q) * P + n]);
      col = std::max(col, sum);
    }
  int most_ex = 0, row_ex = 0, col_ex = 0;
  std::frexp(most, &most_ex);
  std::frexp(row * 1.01, &row_ex);
  std::frexp(col * 1.01, &col_ex);
  if (!std::isfinite(row) || !std::isfinite(col)) return false;
  *fwd = std::min(62 - most_ex, 66 - row_ex);
  *bwd = std::min(62 - most_ex, 66 - col_ex);
  return std::min(*fwd, *bwd) >= 0 && std::max(*fwd, *bwd) <= 100;
}

// Digit tables of both operators (interp: D = 1; grad: D = 3), tab64 = [4][Q][P] on the host.
static int nt_fix_tables(ceed_nt_t h, const double *tab64, cudaStream_t s) {
  const int P = h->P, Q = h->Q, NC = (P + 7) / 8, NG = (Q + 7) / 8;
  for (int op = 0; op < 2; ++op) {
    const int D = op ? 3 : 1;
    const double *M = tab64 + (op ? (size_t)Q * P : 0);
    int *scale = h->fix_scale[op];
    if (!nt_fix_scales(M, D, Q, P, &scale[0], &scale[1])) continue;
    const size_t words = (size_t)NG * D * NC * 32 * FIX_DIGITS;
    std::vector<uint32_t> w(2 * words, 0u);
    for (int d = 0; d < D; ++d)
      for (int q = 0; q < Q; ++q)
        for (int n = 0; n < P; ++n) {
          uint16_t fd[FIX_DIGITS], bd[FIX_DIGITS];
          fix_digits_host(M[((size_t)d * Q + q) * P + n], scale[0], fd);
          if (scale[1] == scale[0]) std::copy(fd, fd + FIX_DIGITS, bd);
          else fix_digits_host(M[((size_t)d * Q + q) * P + n], scale[1], bd);
          const size_t tile = ((size_t)(q / 8) * D + d) * NC + n / 8;
          // forward: output point = lane / 4, input node pair = lane % 4; transposed: the other way round
          const size_t f = (tile * 32 + (q % 8) * 4 + (n % 8) / 2) * FIX_DIGITS;
          const size_t b = words + (tile * 32 + (n % 8) * 4 + (q % 8) / 2) * FIX_DIGITS;
          for (int j = 0; j < FIX_DIGITS; ++j) {
            w[f + j] |= (uint32_t)fd[j] << (16 * (n & 1));
            w[b + j] |= (uint32_t)bd[j] << (16 * (q & 1));
          }
        }
    CEED_CUDA_CHECK(cudaMalloc(&h->d_fix[op], w.size() * 4));
    if (!h->d_again) CEED_CUDA_CHECK(cudaMalloc(&h->d_again, (size_t)(1 + h->E) * 4));
    CEED_CUDA_CHECK(cudaMemcpyAsync(h->d_fix[op], w.data(), w.size() * 4, cudaMemcpyHostToDevice, s));
    CEED_CUDA_CHECK(cudaStreamSynchronize(s));  // w lives in this scope
  }
  return CEED_OK;
}

int nt_fix_prepare(ceed_nt_t h, const double *tab64, cudaStream_t s) {
  if (h->P > NTF_MAX_P) return CEED_OK;
  try {
    return nt_fix_tables(h, tab64, s);
  } catch (const std::bad_alloc &) {
    return fail(CEED_ERR_OOM, "host allocation of the digit tables");
  }
}

template <int D, int NC>
static int launch_nt_fix_nc(const NtFixArgs &a, cudaStream_t s) {
  if (int st = ensure_dynamic_smem((const void *)nt_fix_kernel<D, NC>, ntf_smem<NC>())) return st;
  const unsigned grid = (unsigned)((a.E + 16 * NTF_WARPS - 1) / (16 * NTF_WARPS));
  nt_fix_kernel<D, NC><<<grid, 32 * NTF_WARPS, ntf_smem<NC>(), s>>>(a);
  CEED_CUDA_CHECK(cudaGetLastError());
  return CEED_OK;
}

template <int D>
static int launch_nt_fix(const NtFixArgs &a, cudaStream_t s) {
  switch ((a.P + 7) / 8) {
    case 1: return launch_nt_fix_nc<D, 1>(a, s);
    case 2: return launch_nt_fix_nc<D, 2>(a, s);
    case 3: return launch_nt_fix_nc<D, 3>(a, s);
    case 4: return launch_nt_fix_nc<D, 4>(a, s);
    case 5: return launch_nt_fix_nc<D, 5>(a, s);
    default: return fail(CEED_ERR_UNSUPPORTED, "slice kernel: too many basis functions");
  }
}

int nt_fix_apply(ceed_nt_t h, int op, const double *qd, const double *x, double *Ye, int masked, cudaStream_t s) {
  const int k = op == CEED_OP_MASS ? 0 : 1, D = k ? 3 : 1, NC = (h->P + 7) / 8, NG = (h->Q + 7) / 8;
  NtFixArgs a;
  a.E = h->E;
  a.Es = h->Es;
  a.P = h->P;
  a.Q = h->Q;
  a.ngroups = NG;
  a.rmap = h->d_rmap;
  a.x = x;
  a.fwd = reinterpret_cast<const uint4 *>(h->d_fix[k]);
  a.bwd = a.fwd + (size_t)NG * D * NC * 32 * (FIX_DIGITS / 4);
  a.fwd_scale = h->fix_scale[k][0];
  a.bwd_scale = h->fix_scale[k][1];
  a.again = h->d_again;
  a.qd = qd;
  a.Ye = Ye;
  a.masked = masked;
  CEED_CUDA_CHECK(cudaMemsetAsync(h->d_again, 0, 4, s));
  return k ? launch_nt_fix<3>(a, s) : launch_nt_fix<1>(a, s);
}

}  // namespace ceedgb
