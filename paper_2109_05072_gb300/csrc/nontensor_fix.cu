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
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fixmma.cuh"
#include "nontensor.h"

namespace ceedgb {

constexpr int NTF_WARPS = 4;
// Blocks per SM by node chunks: the warps of a group's chain of passes wait on one another's results most of the time, so
// more of them pay for some spilled registers (degree 4: 1.55 ms with two blocks, 1.19 with three, 1.26 with four;
// degrees 1 to 3: 0.47, 0.68, 0.78 ms with three, 0.41, 0.54, 0.67 with four).
constexpr int ntf_blocks(int nc) { return nc > 4 ? 3 : 4; }

bool nt_fix_supported(int P) { return P <= NTF_MAX_P; }

struct NtFixArgs {
  int64_t E, Es;
  int P, Q, ngroups;
  const uint32_t *rmap;   // [P][E]
  const double *x;
  const uint4 *fwd, *bwd; // [group][D][chunk][lane][2]: eight digit words of the B fragments
  int scale;
  const double *tab;      // [D][Q][P] FP64, for values outside the integer range
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

template <int D, int NC>
__global__ void __launch_bounds__(32 * NTF_WARPS, ntf_blocks(NC)) nt_fix_kernel(const NtFixArgs a) {
  __shared__ uint4 dig_sh[NTF_WARPS][NC][4][32];   // digits of the inputs: lines g (words 0..7), g + 8
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t2 = (lane & 3) * 2;
  const int64_t e0 = ((int64_t)blockIdx.x * NTF_WARPS + warp) * 16;
  const int64_t e[2] = {e0 + g, e0 + g + 8};
  const bool valid[2] = {e[0] < a.E, e[1] < a.E};
  int E0, E1;
  bool odd0, odd1, odd;  // my elements' inputs outside the integer range; any of the warp's
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
    odd0 = fix_odd_or_zero(m0) && (m0 != 0 || tiny0 != 0);
    odd1 = fix_odd_or_zero(m1) && (m1 != 0 || tiny1 != 0);
    odd = __any_sync(0xffffffffu, odd0 || odd1);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
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

#pragma unroll 1
  for (int i = 0; i < a.ngroups; ++i) {
    __syncthreads();  // the block's warps read the same tables at the same time
    const uint4 *tf = a.fwd + ((int64_t)i * D * NC * 32 + lane) * 2, *tb = a.bwd + ((int64_t)i * D * NC * 32 + lane) * 2;
    double v[D][4];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      uint32_t acc[FIX_DIGITS][4];
      const auto chunk = [&](auto first, int c) {
        const uint4 q0 = dig_sh[warp][c][0][lane], q1 = dig_sh[warp][c][1][lane];
        const uint4 q2 = dig_sh[warp][c][2][lane], q3 = dig_sh[warp][c][3][lane];
        const uint32_t x0[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
        const uint32_t x1[8] = {q2.x, q2.y, q2.z, q2.w, q3.x, q3.y, q3.z, q3.w};
        uint32_t b[FIX_DIGITS];
        ntf_load(b, tf + (d * NC + c) * 64);
        fix_products<decltype(first)::value>(acc, x0, x1, b);
      };
      chunk(std::true_type(), 0);
#pragma unroll 1
      for (int c = 1; c < NC; ++c) chunk(std::false_type(), c);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t w[FIX_DIGITS];
#pragma unroll
        for (int s = 0; s < FIX_DIGITS; ++s) w[s] = acc[s][k];
        v[d][k] = fix_out(w, (k < 2 ? E0 : E1) - a.scale + FIX_EXP_OUT);
      }
    }
    if (odd) {
#pragma unroll
      for (int d = 0; d < D; ++d)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (!(k < 2 ? odd0 : odd1)) continue;
          const int q = 8 * i + t2 + (k & 1);
          double s = 0.0;
          if (q < a.Q && valid[k >> 1])
            for (int n = 0; n < a.P; ++n) s = fma(__ldg(a.tab + ((int64_t)d * a.Q + q) * a.P + n), ntf_node(a, n, e[k >> 1]), s);
          v[d][k] = s;
        }
    }
    // pointwise D at my two points of my two elements
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int q = 8 * i + t2 + (k & 1);
      if (q < a.Q && valid[k >> 1]) {
        const double *qd = a.qd + (int64_t)q * a.Es + e[k >> 1];
        const int64_t cs = (int64_t)a.Q * a.Es;
        if constexpr (D == 1) {
          v[0][k] *= __ldg(qd);
        } else {
          const double c0 = __ldg(qd), c1 = __ldg(qd + cs), c2 = __ldg(qd + 2 * cs), c3 = __ldg(qd + 3 * cs);
          const double c4 = __ldg(qd + 4 * cs), c5 = __ldg(qd + 5 * cs);
          const double g0 = v[0][k], g1 = v[1][k], g2 = v[2][k];
          v[0][k] = c0 * g0 + c1 * g1 + c2 * g2;
          v[1][k] = c1 * g0 + c3 * g1 + c4 * g2;
          v[2][k] = c2 * g0 + c4 * g1 + c5 * g2;
        }
      } else {
#pragma unroll
        for (int d = 0; d < D; ++d) v[d][k] = 0.0;
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
    bool o0 = fix_odd_or_zero(m0), o1 = fix_odd_or_zero(m1);
    const bool any_o = __any_sync(0xffffffffu, o0 || o1);
    if (any_o) {  // every lane of the warp
      bool t0 = false, t1 = false;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        t0 |= fix_tiny(v[d][0], v[d][1]);
        t1 |= fix_tiny(v[d][2], v[d][3]);
      }
      const int tiny0 = fix_quad_max(t0), tiny1 = fix_quad_max(t1);
      o0 = o0 && (m0 != 0 || tiny0 != 0);
      o1 = o1 && (m1 != 0 || tiny1 != 0);
    }
    {
      const int F0 = fix_exponent(m0), F1 = fix_exponent(m1);
      uint32_t x0[D][8], x1[D][8];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        fix_digits(x0[d], fix_in(v[d][0], F0), fix_in(v[d][1], F0));
        fix_digits(x1[d], fix_in(v[d][2], F1), fix_in(v[d][3], F1));
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        uint32_t acc[FIX_DIGITS][4];
#pragma unroll
        for (int d = 0; d < D; ++d) {
          uint32_t b[FIX_DIGITS];
          ntf_load(b, tb + (d * NC + c) * 64);
          if (d == 0) fix_products<true>(acc, x0[d], x1[d], b);
          else fix_products<false>(acc, x0[d], x1[d], b);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint32_t w[FIX_DIGITS];
#pragma unroll
          for (int s = 0; s < FIX_DIGITS; ++s) w[s] = acc[s][k];
          const double r = fix_out(w, (k < 2 ? F0 : F1) - a.scale + FIX_EXP_OUT);
          y[c][k] += (k < 2 ? o0 : o1) ? 0.0 : r;
        }
      }
    }
    if (any_o) {
#pragma unroll
      for (int d = 0; d < D; ++d)
#pragma unroll 1
        for (int p = 0; p < 8; ++p) {
          const int q = 8 * i + p;
          const double a0 = __shfl_sync(0xffffffffu, (p & 1) ? v[d][1] : v[d][0], (lane & ~3) + (p >> 1));
          const double a1 = __shfl_sync(0xffffffffu, (p & 1) ? v[d][3] : v[d][2], (lane & ~3) + (p >> 1));
#pragma unroll
          for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int n = 8 * c + t2 + (k & 1);
              if ((k < 2 ? o0 : o1) && q < a.Q && n < a.P)
                y[c][k] = fma(__ldg(a.tab + ((int64_t)d * a.Q + q) * a.P + n), k < 2 ? a0 : a1, y[c][k]);
            }
        }
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int n = 8 * c + t2 + (k & 1);
      if (n < a.P && valid[k >> 1]) a.Ye[(int64_t)n * a.E + e[k >> 1]] = y[c][k];
    }
}

// Digit tables of both operators (interp: D = 1; grad: D = 3), tab64 = [4][Q][P] on the host.
int nt_fix_prepare(ceed_nt_t h, const double *tab64, cudaStream_t s) {
  const int P = h->P, Q = h->Q, NC = (P + 7) / 8, NG = (Q + 7) / 8;
  for (int op = 0; op < 2; ++op) {
    const int D = op ? 3 : 1;
    const double *M = tab64 + (op ? (size_t)Q * P : 0);
    const size_t words = (size_t)NG * D * NC * 32 * FIX_DIGITS;
    std::vector<uint32_t> w(2 * words, 0u);
    const std::vector<long double> big(M, M + (size_t)D * Q * P);
    h->fix_scale[op] = fix_scale_host(big.data(), big.size());
    // the entries of one product (a point's nodes; a group's points and derivatives) sum to less than 2^65
    long double most = 0;
    for (int d = 0; d < D; ++d)
      for (int q = 0; q < Q; ++q) {
        long double sum = 0;
        for (int n = 0; n < P; ++n) sum += std::fabs(M[((size_t)d * Q + q) * P + n]);
        most = std::max(most, sum);
      }
    for (int q0 = 0; q0 < Q; q0 += 8)
      for (int n = 0; n < P; ++n) {
        long double sum = 0;
        for (int d = 0; d < D; ++d)
          for (int q = q0; q < std::min(Q, q0 + 8); ++q) sum += std::fabs(M[((size_t)d * Q + q) * P + n]);
        most = std::max(most, sum);
      }
    int ex = 0;
    std::frexp(most, &ex);
    h->fix_scale[op] = std::min(h->fix_scale[op], 65 - ex);
    for (int d = 0; d < D; ++d)
      for (int q = 0; q < Q; ++q)
        for (int n = 0; n < P; ++n) {
          uint16_t dig[FIX_DIGITS];
          fix_digits_host(M[((size_t)d * Q + q) * P + n], h->fix_scale[op], dig);
          const size_t tile = ((size_t)(q / 8) * D + d) * NC + n / 8;
          // forward: output point = lane / 4, input node pair = lane % 4; transposed: the other way round
          const size_t f = (tile * 32 + (q % 8) * 4 + (n % 8) / 2) * FIX_DIGITS;
          const size_t b = words + (tile * 32 + (n % 8) * 4 + (q % 8) / 2) * FIX_DIGITS;
          for (int j = 0; j < FIX_DIGITS; ++j) {
            w[f + j] |= (uint32_t)dig[j] << (16 * (n & 1));
            w[b + j] |= (uint32_t)dig[j] << (16 * (q & 1));
          }
        }
    CEED_CUDA_CHECK(cudaMalloc(&h->d_fix[op], w.size() * 4));
    CEED_CUDA_CHECK(cudaMemcpyAsync(h->d_fix[op], w.data(), w.size() * 4, cudaMemcpyHostToDevice, s));
    CEED_CUDA_CHECK(cudaStreamSynchronize(s));  // w lives in this scope
  }
  return CEED_OK;
}

template <int D>
static int launch_nt_fix(const NtFixArgs &a, cudaStream_t s) {
  const unsigned grid = (unsigned)((a.E + 16 * NTF_WARPS - 1) / (16 * NTF_WARPS));
  switch ((a.P + 7) / 8) {
    case 1: nt_fix_kernel<D, 1><<<grid, 32 * NTF_WARPS, 0, s>>>(a); break;
    case 2: nt_fix_kernel<D, 2><<<grid, 32 * NTF_WARPS, 0, s>>>(a); break;
    case 3: nt_fix_kernel<D, 3><<<grid, 32 * NTF_WARPS, 0, s>>>(a); break;
    case 4: nt_fix_kernel<D, 4><<<grid, 32 * NTF_WARPS, 0, s>>>(a); break;
    case 5: nt_fix_kernel<D, 5><<<grid, 32 * NTF_WARPS, 0, s>>>(a); break;
    default: return fail(CEED_ERR_UNSUPPORTED, "slice kernel: too many basis functions");
  }
  CEED_CUDA_CHECK(cudaGetLastError());
  return CEED_OK;
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
  a.scale = h->fix_scale[k];
  a.tab = h->d_tab64 + (k ? (size_t)h->Q * h->P : 0);
  a.qd = qd;
  a.Ye = Ye;
  a.masked = masked;
  return k ? launch_nt_fix<3>(a, s) : launch_nt_fix<1>(a, s);
}

}  // namespace ceedgb
