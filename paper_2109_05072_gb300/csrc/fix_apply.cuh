// The FP64 operators of apply_kernel.cuh with their 1D passes on the tensor cores (fixmma.cuh), for lines of up to
// FIX_MAX_Q points.
#pragma once

#include "fixmma.cuh"

namespace ceedgb {

// Shared-memory tile of one element: (t, s, r) at t * TP + s * 10 + r.  Pitch 10 and TP = 2 or 6 (mod 8)
// put the quarter-warps' accesses of the s and t passes and of the pointwise step on distinct banks.
template <int Q>
constexpr int fix_tp() {
  int tp = 10 * (Q - 1) + Q;
  while (tp % 8 != 2 && tp % 8 != 6) ++tp;
  return tp;
}
template <int Q>
constexpr int fix_warps() {
  return (Q * Q + 15) / 16;
}
// one element's tiles: three for diffusion, one for the mass operator
template <int P, int Q, int OP>
constexpr size_t fix_smem() {
  return ((size_t)(OP == CEED_OP_MASS ? 1 : 3) * Q * fix_tp<Q>() * sizeof(double) + 127) & ~(size_t)127;
}

// The elements' results r at a thread's nodes added to y (E -> L): first writer stores, later ones
// load-add-store; with a fused dot, x . y over the nodes whose final value this block writes, in a fixed order.
template <bool XCG>
__device__ __forceinline__ void fix_scatter(const ApplyArgs &a, const uint32_t (&idx)[4], const bool (&on)[4], const double (&r)[4],
                                            int col, int64_t blk) {
  double dot = 0.0;
  double yold[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    yold[k] = 0.0;
    if (on[k] && !(idx[k] & FLAG_FIRST) && !(a.masked && (idx[k] & FLAG_DIR)))
      yold[k] = __ldcg(a.y + (int64_t)(idx[k] & DOF_MASK) * a.ncol + col);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!on[k]) continue;
    const int64_t o = (int64_t)(idx[k] & DOF_MASK) * a.ncol + col;
    if (a.masked && (idx[k] & FLAG_DIR)) {
      if (idx[k] & FLAG_FIRST) {
        const double v = XCG ? __ldcg(a.x + o) : __ldg(a.x + o);
        a.y[o] = v;
        dot += v * v;
      }
    } else {
      const double v = (idx[k] & FLAG_FIRST) ? r[k] : yold[k] + r[k];
      a.y[o] = v;
      if ((idx[k] & FLAG_LAST) && (a.dot_part || a.dot_sh)) dot += (XCG ? __ldcg(a.x + o) : __ldg(a.x + o)) * v;
    }
  }
  if (a.dot_part || a.dot_sh) {
    __shared__ double dsum[APPLY_MAX_THREADS / 32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_down_sync(0xffffffffu, dot, off);
    if ((threadIdx.x & 31) == 0) dsum[threadIdx.x >> 5] = dot;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += dsum[w];
      if (a.dot_sh) *a.dot_sh += s;
      else a.dot_part[a.dot_base + blk] = s;
    }
  }
}

// fix_scatter in the element's turn; false if the wait for it gave up (nothing is then written).
template <bool XCG, typename WaitY>
__device__ __forceinline__ bool fix_turn(const ApplyArgs &a, const uint32_t (&idx)[4], const bool (&on)[4], const double (&r)[4],
                                         int64_t e, int col, bool first_col, int64_t blk, const WaitY &wait_y) {
  if constexpr (std::is_same<WaitY, ClusterOrder>::value) {
    wait_y.in_turn(e, [&](bool turn) {
      const bool now[4] = {turn && on[0], turn && on[1], turn && on[2], turn && on[3]};
      fix_scatter<XCG>(a, idx, now, r, col, blk);
    });
    return true;
  } else {
    if (first_col && !wait_y()) return false;
    fix_scatter<XCG>(a, idx, on, r, col, blk);
    return true;
  }
}

// One element of the collocated diffusion operator, FP64: fix_warps<Q>() warps, warp w on lines
// 16 w .. 16 w + 15 of every direction.  A thread keeps its t-lines in registers (gather, pointwise
// step, scatter: nodes t * Q^2 + line); r- and s-lines go through shared memory.  The FP64 pipe keeps
// the pointwise step (9 instructions a point) and the final sums (3).
template <int Q, bool XCG, typename WaitY>
__device__ __forceinline__ void fix_block(const ApplyArgs &a, const OpTab<double> &tab, const uint32_t *ftab, int64_t blk,
                                          unsigned char *smem_raw, const WaitY &wait_y) {
  constexpr int NQ = Q * Q * Q, TP = fix_tp<Q>();
  constexpr int NT = 32 * fix_warps<Q>();
  const int el = threadIdx.x / NT, tid = threadIdx.x % NT, lane = tid & 31, g = lane >> 2, t2 = (lane & 3) * 2;
  const unsigned eb = (unsigned)blk / (unsigned)a.cgroups, cg = (unsigned)blk - eb * (unsigned)a.cgroups;
  const int col0 = (int)cg * a.cpb, col1 = min(a.ncol, col0 + a.cpb);
  const int64_t e = a.e_begin + (int64_t)eb * a.ne + el;
  const bool active = el < a.ne && e < a.e_begin + a.e_count;
  double *su = (double *)(smem_raw + el * fix_smem<Q, Q, CEED_OP_DIFFUSION>()), *sr = su + Q * TP, *ss = sr + Q * TP;
  const double *sq = (const double *)a.qdata + e * a.estride;
  if (tid == 0 && active) l2_prefetch_bulk(sq, (uint32_t)(a.estride * sizeof(double)));
  // my lines (two per direction) and entries (two per line)
  const int l[2] = {(tid >> 5) * 16 + g, (tid >> 5) * 16 + g + 8};
  bool on[4];
  int at[4];   // tile position of my points: entry k & 1 of t-line l[k >> 1]
  int qp[4];   // their point number
  int lr[2], ls[2];  // tile positions of entry t2 of my r-lines and s-lines
  uint32_t idx[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int h = k >> 1, t = t2 + (k & 1);
    on[k] = active && l[h] < Q * Q && t < Q;
    at[k] = t * TP + (l[h] / Q) * 10 + l[h] % Q;
    qp[k] = t * Q * Q + l[h];
    idx[k] = on[k] ? __ldg(a.emap + e * NQ + qp[k]) : 0u;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    lr[h] = (l[h] / Q) * TP + (l[h] % Q) * 10 + t2;
    ls[h] = (l[h] / Q) * TP + t2 * 10 + l[h] % Q;
  }
  FixMat D;
  fix_load(D, ftab, lane);
  for (int col = col0; col < col1; ++col) {
    double u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      u[k] = 0.0;
      if (on[k] && !(a.masked && (idx[k] & FLAG_DIR))) {
        const double *x = a.x + (int64_t)(idx[k] & DOF_MASK) * a.ncol + col;
        u[k] = XCG ? __ldcg(x) : __ldg(x);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (on[k]) su[at[k]] = u[k];
    const auto full = [&](int n, int m) { return tab.D[n * Q + m]; };
    const auto full_t = [&](int n, int m) { return tab.D[m * Q + n]; };
    double gt[4];
    fix_pass<Q, Q>(D, u, gt, full);
    __syncthreads();
    {
      double v[4], w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = on[k] ? su[lr[k >> 1] + (k & 1)] : 0.0;
      fix_pass<Q, Q>(D, v, w, full);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (on[k]) sr[lr[k >> 1] + (k & 1)] = w[k];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = on[k] ? su[ls[k >> 1] + (k & 1) * 10] : 0.0;
      fix_pass<Q, Q>(D, v, w, full);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (on[k]) ss[ls[k >> 1] + (k & 1) * 10] = w[k];
    }
    __syncthreads();
    double wt[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      wt[k] = 0.0;
      if (on[k]) {
        const double *G = sq + qp[k];
        const double grr = __ldg(G), grs = __ldg(G + NQ), grt = __ldg(G + 2 * NQ);
        const double gss = __ldg(G + 3 * NQ), gst = __ldg(G + 4 * NQ), gtt = __ldg(G + 5 * NQ);
        const double ur = sr[at[k]], us = ss[at[k]];
        sr[at[k]] = grr * ur + grs * us + grt * gt[k];
        ss[at[k]] = grs * ur + gss * us + gst * gt[k];
        wt[k] = grt * ur + gst * us + gtt * gt[k];
      }
    }
    FixMat DT;
    fix_load(DT, ftab + FIX_TAB_WORDS, lane);
    double y[4];
    fix_pass<Q, Q>(DT, wt, y, full_t);
    __syncthreads();
    {
      double v[4], w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = on[k] ? sr[lr[k >> 1] + (k & 1)] : 0.0;
      fix_pass<Q, Q>(DT, v, w, full_t);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (on[k]) sr[lr[k >> 1] + (k & 1)] = w[k];  // in place: this thread's own entries
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = on[k] ? ss[ls[k >> 1] + (k & 1) * 10] : 0.0;
      fix_pass<Q, Q>(DT, v, w, full_t);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (on[k]) ss[ls[k >> 1] + (k & 1) * 10] = w[k];
    }
    __syncthreads();
    double r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) r[k] = on[k] ? y[k] + sr[at[k]] + ss[at[k]] : 0.0;
    if (!fix_turn<XCG>(a, idx, on, r, e, col, col == col0, blk, wait_y)) return;
    if (col + 1 < col1) __syncthreads();
  }
}

// The same with Gauss quadrature (Q = P + 1 points), mass or diffusion: interpolation along t, s, r, the
// quadrature-point operator on r-lines in registers, and the transposed way back; the node values of a
// thread are those of its t-lines.  A pass reads and writes the same entries of the tile, so it works in place.
template <int P, int Q, int OP, bool XCG, typename WaitY>
__device__ __forceinline__ void fix_gauss_block(const ApplyArgs &a, const OpTab<double> &tab, const uint32_t *ftab, int64_t blk,
                                                unsigned char *smem_raw, const WaitY &wait_y) {
  constexpr int NQ = Q * Q * Q, ND = P * P * P, TP = fix_tp<Q>(), NT = 32 * fix_warps<Q>();
  const int el = threadIdx.x / NT, tid = threadIdx.x % NT, lane = tid & 31, g = lane >> 2, t2 = (lane & 3) * 2;
  const unsigned eb = (unsigned)blk / (unsigned)a.cgroups, cg = (unsigned)blk - eb * (unsigned)a.cgroups;
  const int col0 = (int)cg * a.cpb, col1 = min(a.ncol, col0 + a.cpb);
  const int64_t e = a.e_begin + (int64_t)eb * a.ne + el;
  const bool active = el < a.ne && e < a.e_begin + a.e_count;
  double *s0 = (double *)(smem_raw + el * fix_smem<P, Q, OP>()), *s1 = s0 + Q * TP, *s2 = s1 + Q * TP;
  const double *sq = (const double *)a.qdata + (active ? e : a.e_begin) * a.estride;
  if (tid == 0 && active) l2_prefetch_bulk(sq, (uint32_t)(a.estride * sizeof(double)));
  const int l[2] = {(tid >> 5) * 16 + g, (tid >> 5) * 16 + g + 8};
  // entries t2, t2 + 1 (below n) of my lines (below nl) in a tile: line at base(l), entries `step` apart
  const auto get = [&](const double *s, double (&v)[4], int nl, int n, int step, auto base) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = (l[k >> 1] < nl && t2 + (k & 1) < n) ? s[base(l[k >> 1]) + (t2 + (k & 1)) * step] : 0.0;
  };
  const auto put = [&](double *s, const double (&v)[4], int nl, int n, int step, auto base) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (l[k >> 1] < nl && t2 + (k & 1) < n) s[base(l[k >> 1]) + (t2 + (k & 1)) * step] = v[k];
  };
  const auto r_line = [](int i) { return (i / Q) * TP + (i % Q) * 10; };  // (t, s) of Q x Q
  const auto s_line = [](int i) { return (i / Q) * TP + i % Q; };         // (t, r) of Q x Q
  const auto t_line = [](int i) { return (i / Q) * 10 + i % Q; };         // (s, r) of Q x Q
  const auto s_part = [](int i) { return (i / P) * TP + i % P; };         // (t, r) of Q x P
  const auto t_part = [](int i) { return (i / P) * 10 + i % P; };         // (s, r) of P x P
  const auto full_b = [&](int n, int m) { return tab.B[n * P + m]; };
  const auto full_bt = [&](int n, int m) { return tab.B[m * P + n]; };
  const auto full_d = [&](int n, int m) { return tab.D[n * Q + m]; };
  const auto full_dt = [&](int n, int m) { return tab.D[m * Q + n]; };
  bool on[4];
  uint32_t idx[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int t = t2 + (k & 1);
    on[k] = active && l[k >> 1] < P * P && t < P;
    idx[k] = on[k] ? __ldg(a.emap + e * ND + t * P * P + l[k >> 1]) : 0u;
  }
  FixMat M;
  for (int col = col0; col < col1; ++col) {
    double v[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = 0.0;
      if (on[k] && !(a.masked && (idx[k] & FLAG_DIR))) {
        const double *x = a.x + (int64_t)(idx[k] & DOF_MASK) * a.ncol + col;
        v[k] = XCG ? __ldcg(x) : __ldg(x);
      }
    }
    fix_load(M, ftab + 2 * FIX_TAB_WORDS, lane);
    fix_pass<P, Q>(M, v, w, full_b);
    put(s0, w, P * P, Q, TP, t_part);
    __syncthreads();
    get(s0, v, Q * P, P, 10, s_part);
    fix_pass<P, Q>(M, v, w, full_b);
    put(s0, w, Q * P, Q, 10, s_part);
    __syncthreads();
    get(s0, v, Q * Q, P, 1, r_line);
    fix_pass<P, Q>(M, v, w, full_b);
    // w: the column's values at my points (r-lines, entries t2 and t2 + 1)
    const auto point = [&](int k) { return l[k >> 1] * Q + t2 + (k & 1); };
    const auto at_point = [&](int k) { return active && l[k >> 1] < Q * Q && t2 + (k & 1) < Q; };
    if constexpr (OP == CEED_OP_MASS) {
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = at_point(k) ? __ldg(sq + point(k)) * w[k] : 0.0;
    } else {
      fix_load(M, ftab, lane);
      double ur[4];
      fix_pass<Q, Q>(M, w, ur, full_d);
      put(s0, w, Q * Q, Q, 1, r_line);
      __syncthreads();
      get(s0, v, Q * Q, Q, 10, s_line);
      fix_pass<Q, Q>(M, v, w, full_d);
      put(s1, w, Q * Q, Q, 10, s_line);
      get(s0, v, Q * Q, Q, TP, t_line);
      fix_pass<Q, Q>(M, v, w, full_d);
      put(s2, w, Q * Q, Q, TP, t_line);
      __syncthreads();
      get(s1, v, Q * Q, Q, 1, r_line);
      get(s2, w, Q * Q, Q, 1, r_line);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double us = v[k], ut = w[k], u0 = ur[k];
        ur[k] = v[k] = w[k] = 0.0;
        if (at_point(k)) {
          const double *G = sq + point(k);
          const double grr = __ldg(G), grs = __ldg(G + NQ), grt = __ldg(G + 2 * NQ);
          const double gss = __ldg(G + 3 * NQ), gst = __ldg(G + 4 * NQ), gtt = __ldg(G + 5 * NQ);
          ur[k] = grr * u0 + grs * us + grt * ut;
          v[k] = grs * u0 + gss * us + gst * ut;
          w[k] = grt * u0 + gst * us + gtt * ut;
        }
      }
      put(s1, v, Q * Q, Q, 1, r_line);
      put(s2, w, Q * Q, Q, 1, r_line);
      fix_load(M, ftab + FIX_TAB_WORDS, lane);
      double yr[4];
      fix_pass<Q, Q>(M, ur, yr, full_dt);
      __syncthreads();
      get(s1, v, Q * Q, Q, 10, s_line);
      fix_pass<Q, Q>(M, v, w, full_dt);
      put(s1, w, Q * Q, Q, 10, s_line);
      get(s2, v, Q * Q, Q, TP, t_line);
      fix_pass<Q, Q>(M, v, w, full_dt);
      put(s2, w, Q * Q, Q, TP, t_line);
      __syncthreads();
      get(s1, v, Q * Q, Q, 1, r_line);
      get(s2, w, Q * Q, Q, 1, r_line);
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = yr[k] + v[k] + w[k];
    }
    fix_load(M, ftab + 3 * FIX_TAB_WORDS, lane);
    fix_pass<Q, P>(M, w, v, full_bt);
    put(s0, v, Q * Q, P, 1, r_line);
    __syncthreads();
    get(s0, v, Q * P, Q, 10, s_part);
    fix_pass<Q, P>(M, v, w, full_bt);
    put(s0, w, Q * P, P, 10, s_part);
    __syncthreads();
    get(s0, v, P * P, Q, TP, t_part);
    fix_pass<Q, P>(M, v, w, full_bt);
    if (!fix_turn<XCG>(a, idx, on, w, e, col, col == col0, blk, wait_y)) return;
    if (col + 1 < col1) __syncthreads();
  }
}

// Measured (GB300, before -> after): diffusion p = 7 at 40^3 2.97 -> 1.21 ms (308 us is the traffic's share, 640 us the FP64
// pipe's: 12 instructions a point), p = 5 at 13 x 11 x 9 49 -> 35 us, mass p = 6 Gauss on 15,525 elements 503 -> 249 us.
// FP64 operators that run on the slices, whatever variant of the apply is asked for: collocated diffusion with 6 to
// 8 points per direction, and mass and diffusion with 7 or 8 Gauss points.  A line costs the integer pipe the same
// whatever its length, so shorter lines gain nothing (8 entries: 24 clocks of the FP64 pipe against 8 of the
// integer pipe; 5: 10 against 8 and the tile's unused lines); longer ones do not fit the tile.
template <int P, int Q, int OP, typename T>
constexpr bool fix_covers() {
  return std::is_same<T, double>::value && slice_operator(P, Q, OP);
}

template <int P, int Q, int OP, bool XCG, typename WaitY>
__device__ __forceinline__ void fix_any_block(const ApplyArgs &a, const OpTab<double> &tab, const uint32_t *ftab, int64_t blk,
                                              unsigned char *smem_raw, const WaitY &wait_y) {
  if constexpr (P == Q) fix_block<Q, XCG>(a, tab, ftab, blk, smem_raw, wait_y);
  else fix_gauss_block<P, Q, OP, XCG>(a, tab, ftab, blk, smem_raw, wait_y);
}

struct FixArgs {
  ApplyArgs a;
  const uint32_t *tab;
};

// Blocks per SM: with neither the FP64 nor the integer pipe full (51 and 46% at p = 7 with four blocks) warps wait on
// one another's results, so a fifth block pays for some spilled registers (40^3 at p = 7: 1.26 -> 1.20 ms; 24^3 at p = 5: 238 ->
// 223 us), except at p = 6 (24^3: 260 with four, 269 us with five).  Staging the quadrature data in shared memory by
// cp.async was slower than reading it at the pointwise step (p = 7: 1.34 ms): it takes L1 from the tables.
template <int P, int Q>
constexpr int fix_min_blocks() {
  return P == 7 && Q == 7 ? 4 : 5;
}

template <int P, int Q, int OP>
__global__ void __launch_bounds__(32 * fix_warps<Q>(), fix_min_blocks<P, Q>()) fix_kernel(const FixArgs f, const OpTab<double> tab) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  ColourWait wait_y;
  colour_open_next();
  fix_any_block<P, Q, OP, false>(f.a, tab, f.tab, blockIdx.x, smem_raw, wait_y);
}

template <int P, int Q, int OP>
__global__ void __launch_bounds__(APPLY_MAX_THREADS) fix_cluster_kernel(const FixArgs f, const OpTab<double> tab, const ClusterOrder order) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  fix_any_block<P, Q, OP, false>(f.a, tab, f.tab, blockIdx.x, smem_raw, order);
}

}  // namespace ceedgb
