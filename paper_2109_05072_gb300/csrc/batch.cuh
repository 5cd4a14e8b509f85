// Batched apply: several independent meshes (different polynomial orders allowed) in ONE persistent
// launch.  The blocks of a persistent grid take pieces of work (element blocks) colour by colour over
// all meshes; a piece touches y once its mesh's previous colour is in memory (ColourOrder), so that the
// atomic-free scatter stays race-free.  The grid is sized to what is co-resident on the GPU; the wait
// is bounded (a timeout is recorded instead of hanging).
#pragma once

#include <algorithm>
#include <cstring>

#include "apply_kernel.cuh"
#include "progress.h"

namespace ceedgb {

struct BatchMesh {
  ApplyArgs a;                              // e_begin / e_count set per colour inside the kernel
  int P, Q, ncolors;
  const uint32_t *fix;                      // digit tables of the slice kernels, if the mesh has them
  int64_t cstart[BATCH_MAX_COLORS + 1];     // colour-sorted element ranges
};

template <typename T>
struct BatchArgs {
  int n, max_colors;
  unsigned *sync;                           // [BATCH_SYNC_WORDS], zero before a launch and after it
  int *err;
  long long grid_wait;                      // polls of a wait between colours before it gives up
  BatchMesh m[BATCH_MAX];
  OpTab<T> tab[BATCH_MAX];
};

// Pause between two polls of a grid barrier or of a colour's counter.  Shorter ones gain nothing (64 ns: the same times at
// 16^3 and 24^3, p = 7, all operators, and in the batch), and the waits' limits are counted in polls.
constexpr unsigned POLL_NS = 100;

// Bounded grid barrier (sense by generation counter).  Returns false on timeout.
__device__ __forceinline__ bool grid_barrier(unsigned *sync, int *err, long long limit, int *ok_sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned *vgen = sync + SYNC_LINE;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(sync, 1u) + 1u;
    if (arrived == gridDim.x) {
      atomicExch(sync, 0u);
      __threadfence();
      atomicAdd(sync + SYNC_LINE, 1u);
    } else {
      long long it = 0;
      while (*vgen == gen) {
        if (++it > limit) {
          ok = 0;
          *err = CEED_ERR_TIMEOUT;
          break;
        }
        __nanosleep(POLL_NS);
      }
    }
    __threadfence();
    *ok_sh = ok;
  }
  __syncthreads();
  return *ok_sh != 0;
}

// The 1D tables of the mesh being processed, copied from the parameter block to the start of shared memory
// (indexing the parameter block by a run-time mesh slot would cost registers in every pass).
template <typename T>
constexpr size_t batch_tab_bytes() {
  return (sizeof(OpTab<T>) + 127) & ~(size_t)127;
}

// Pieces of work (element blocks times column groups) of mesh m's colour c.
template <typename T>
__device__ __forceinline__ int64_t pieces(const BatchArgs<T> &b, int c, int m) {
  if (c >= b.m[m].ncolors) return 0;
  const ApplyArgs &a = b.m[m].a;
  return (b.m[m].cstart[c + 1] - b.m[m].cstart[c] + a.ne - 1) / a.ne * a.cgroups;
}

// Order between the colours of a persistent apply without a grid barrier.  done[c] counts the work of
// colour c that is in memory: the batch's pieces (element blocks), or in the fused PCG iteration the blocks that
// have finished their share of the colour.  Work of colour c touches y once
// done[c - 1] has reached its total -- all of colour c - 1 waited for colour c - 2, so all
// earlier colours are then in memory.  Blocks take pieces in colour order, so the earliest unfinished
// piece never waits, and all that a piece does before its scatter (gather, contractions) overlaps the
// colour before.  The wait is bounded like the grid barrier's.
struct ColourOrder {
  static constexpr bool OPEN = false;
  const unsigned *prev;   // counter of the colour before; null: nothing to wait for, or waited for already
  unsigned target;
  long long limit;
  int *err;
  int *ok_sh;             // shared word: thread 0's verdict for the block
  __device__ __forceinline__ bool operator()() const {
    if (!prev) return true;
    if (threadIdx.x == 0) {
      int ok = 1;
      const volatile unsigned *v = prev;
      long long it = 0;
      while (!progress_reached(*v, target)) {
        if (++it > limit) {
          ok = 0;
          *err = CEED_ERR_TIMEOUT;
          break;
        }
        __nanosleep(POLL_NS);
      }
      __threadfence();
      *ok_sh = ok;
    }
    __syncthreads();
    return *ok_sh != 0;
  }
};

// The block's work counted here is done (its writes included): called by every thread.
__device__ __forceinline__ void colour_done(unsigned *done) {
  __syncthreads();  // also frees shared memory for the next piece
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(done, 1u);
  }
}

// One piece of work of one order: a function of its own, so that the orders' register needs do not add up (inlined
// together under the cap of 128 registers they spill 1.8 KB per thread; here 48 bytes at most).  It copies its arguments:
// through the caller's references every use of one is a load from local memory (double-float, p = 3, 5, 7 on 48^3, 40^3,
// 32^3 elements, 3 / 12 columns: 10.8 / 39.2 ms, 9.5 / 35.2 with copies).
template <int P, int Q, int OP, typename T, typename TQ, bool STAGE>
__device__ __noinline__ void batch_piece(const ApplyArgs &args, const uint32_t *fix, int64_t blk, const ColourOrder &order) {
  const ApplyArgs a = args;
  const ColourOrder wait_y = order;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // one copy barrier per element slot of the largest block, idle slots included (apply_block readies them all):
  // 64 at Q = 2, more than the APPLY_MAX_NE elements that a launch of its own may ask for
  __shared__ uint64_t bar[STAGE ? (APPLY_MAX_THREADS + Q * Q - 1) / (Q * Q) : 1];
  const OpTab<T> &tab = *reinterpret_cast<const OpTab<T> *>(smem_raw);
  if constexpr (fix_covers<P, Q, OP, T>()) fix_any_block<P, Q, OP, false>(a, tab, fix, blk, smem_raw + batch_tab_bytes<T>(), wait_y);
  else apply_block<P, Q, OP, T, TQ, STAGE>(a, tab, blk, smem_raw + batch_tab_bytes<T>(), bar, wait_y);
}

template <int OP, typename T, typename TQ, bool STAGE, bool COLLOC>
__device__ __forceinline__ void batch_body(const BatchArgs<T> &b, unsigned char *smem_raw) {
  __shared__ int ok_sh;
  T *tab_words = (T *)smem_raw;
  __shared__ int64_t next_sh;
  int cur_m = -1;
  int c = 0, m = 0;
  int64_t base = 0;       // pieces before those of (colour c, mesh m)
  int64_t cnt = pieces(b, 0, 0);
  // pieces are numbered colour by colour, mesh by mesh, and handed out in that order: the orders'
  // elements cost up to ten times one another, so a fixed share per block would leave blocks idle
  if (threadIdx.x == 0) ok_sh = 1;
  for (;;) {
    if (threadIdx.x == 0) next_sh = atomicAdd(b.sync, 1u);
    __syncthreads();
    const int64_t v = next_sh;
    if (v < base) {  // the counters went back under a running launch (the batch applied twice at once)
      if (threadIdx.x == 0) *b.err = CEED_ERR_TIMEOUT;
      return;
    }
    while (v >= base + cnt) {
      base += cnt;
      if (++m == b.n) {
        m = 0;
        if (++c == b.max_colors) break;
      }
      cnt = pieces(b, c, m);
    }
    if (c == b.max_colors) break;
    ApplyArgs a = b.m[m].a;
    a.e_begin = b.m[m].cstart[c];
    a.e_count = b.m[m].cstart[c + 1] - a.e_begin;
    unsigned *done = b.sync + (2 + m * BATCH_MAX_COLORS + c) * SYNC_LINE;
    const ColourOrder wait_y{c ? done - SYNC_LINE : nullptr, c ? (unsigned)pieces(b, c - 1, m) : 0u, b.grid_wait, b.err, &ok_sh};
    const int64_t blk = v - base;
    if (m != cur_m) {
      const T *src = reinterpret_cast<const T *>(&b.tab[m]);
      for (int w = threadIdx.x; w < (int)(sizeof(OpTab<T>) / sizeof(T)); w += blockDim.x) tab_words[w] = src[w];
      __syncthreads();
      cur_m = m;
    }
#define CEEDGB_BCASE(PP)                                                                       \
  case PP:                                                                                     \
    batch_piece<PP, COLLOC ? PP : PP + 1, OP, T, TQ, STAGE>(a, b.m[m].fix, blk, wait_y);       \
    break;
    switch (b.m[m].P) {
      CEEDGB_BCASE(2)
      CEEDGB_BCASE(3)
      CEEDGB_BCASE(4)
      CEEDGB_BCASE(5)
      CEEDGB_BCASE(6)
      CEEDGB_BCASE(7)
      CEEDGB_BCASE(8)
      CEEDGB_BCASE(9)
      default:
        break;
    }
#undef CEEDGB_BCASE
    if (!ok_sh) return;  // gave up: the later pieces' waits run out too; the host resets the counters
    colour_done(done);
  }
  // the last block to leave readies the counters for the next launch (no block waits any more)
  if (threadIdx.x == 0) ok_sh = atomicAdd(b.sync + SYNC_LINE, 1u) + 1u == gridDim.x;
  __syncthreads();
  if (ok_sh)
    for (int w = threadIdx.x * SYNC_LINE; w < BATCH_SYNC_WORDS; w += blockDim.x * SYNC_LINE) b.sync[w] = 0u;
}

template <int OP, typename T, typename TQ, bool STAGE, bool COLLOC>
__global__ void __launch_bounds__(APPLY_MAX_THREADS, std::is_same<T, DF>::value ? 1 : 2) batch_kernel(const BatchArgs<T> b) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  batch_body<OP, T, TQ, STAGE, COLLOC>(b, smem_raw);
}

// Threads of one element where the slice kernels run the mesh's operator, else 0.
template <int OP, typename T>
int batch_fix_threads(int P, int Q) {
#define CEEDGB_S(PP)                                                                                   \
  if (P == PP && Q == PP && fix_covers<PP, PP, OP, T>()) return 32 * fix_warps<PP>();                   \
  if (P == PP && Q == PP + 1 && fix_covers<PP, PP + 1, OP, T>()) return 32 * fix_warps<PP + 1>();
  CEEDGB_S(6) CEEDGB_S(7) CEEDGB_S(8)
#undef CEEDGB_S
  return 0;
}

// Shared memory per thread block for a mesh with P nodes / Q points when blocks have `threads` threads.
template <int OP, typename T, typename TQ, bool STAGE>
size_t batch_smem_for(int P, int Q, int threads) {
  if (const int per = batch_fix_threads<OP, T>(P, Q)) {
    size_t fb = 0;
#define CEEDGB_S(PP) \
  if (P == PP) fb = (Q == PP) ? fix_smem<PP, PP, OP>() : fix_smem<PP, PP + 1, OP>();
    CEEDGB_S(6) CEEDGB_S(7) CEEDGB_S(8)
#undef CEEDGB_S
    return (size_t)((threads + per - 1) / per) * fb;
  }
  const int slots = (threads + Q * Q - 1) / (Q * Q);
  size_t eb = 0;
#define CEEDGB_S(PP)                                                                              \
  if (P == PP) eb = (Q == PP) ? apply_elem_smem<PP, PP, OP, T, TQ, STAGE>()                       \
                              : apply_elem_smem<PP, PP + 1, OP, T, TQ, STAGE>();
  CEEDGB_S(2) CEEDGB_S(3) CEEDGB_S(4) CEEDGB_S(5) CEEDGB_S(6) CEEDGB_S(7) CEEDGB_S(8) CEEDGB_S(9)
#undef CEEDGB_S
  return (size_t)slots * eb;
}


// Launch one batched apply (host side).  `launch` lists the meshes' apply requests.
template <int OP, typename T, typename TQ>
int launch_batch(int n, ceed_mesh_t const *meshes, const ApplyReq *reqs, const OpTab<T> *const *tabs,
                 unsigned *sync, int *err, const BatchLaunch &L, cudaStream_t s, unsigned *grid_used) {
  BatchArgs<T> b;
  std::memset(&b, 0, sizeof(b));
  b.n = n;
  b.sync = sync;
  b.err = err;
  b.grid_wait = grid_wait_limit();
  size_t smem = 0;
  const bool colloc = meshes[0]->Q == meshes[0]->P;
  if (L.threads > APPLY_MAX_THREADS) return fail(CEED_ERR_INVALID, "batch blocks have at most 256 threads");
  for (int k = 0; k < n; ++k) {
    ceed_mesh_t m = meshes[k];
    if ((m->Q == m->P) != colloc) return fail(CEED_ERR_UNSUPPORTED, "a batch mixes quadrature rules");
    if (m->n_colors > BATCH_MAX_COLORS) return fail(CEED_ERR_UNSUPPORTED, "too many colours for a batch");
    BatchMesh &bm = b.m[k];
    bm.P = m->P;
    bm.Q = m->Q;
    bm.ncolors = 0;  // colours that hold elements (each waits for the one before)
    for (int c = 0; c < m->n_colors; ++c)
      if (m->color_start[c + 1] > m->color_start[c]) bm.cstart[++bm.ncolors] = m->color_start[c + 1];
    bm.a.emap = m->d_emap;
    bm.a.qdata = reqs[k].qdata;
    bm.a.x = reqs[k].x;
    bm.a.y = reqs[k].y;
    bm.a.ncol = reqs[k].ncol;
    bm.a.masked = reqs[k].masked;
    const int fix_threads = batch_fix_threads<OP, T>(m->P, m->Q);
    bm.fix = m->d_fix;
    bm.a.ne = L.threads / (fix_threads ? fix_threads : m->Q * m->Q);
    if (bm.a.ne < 1) return fail(CEED_ERR_INVALID, "block too small for this order");
    column_split(bm.a, (meshes[k]->E / std::max(1, bm.ncolors) + bm.a.ne - 1) / bm.a.ne);
    bm.a.err = err;
    bm.a.wait_limit = copy_wait_limit();
    bm.a.estride = qdata_estride(OP, sizeof(TQ), m->Q);
    bm.a.dot_part = nullptr;
    bm.a.dot_base = 0;
    bm.a.dot_sh = nullptr;
    b.tab[k] = *tabs[k];
    b.max_colors = std::max(b.max_colors, bm.ncolors);
    const size_t sm = L.stage ? batch_smem_for<OP, T, TQ, true>(m->P, m->Q, L.threads)
                              : batch_smem_for<OP, T, TQ, false>(m->P, m->Q, L.threads);
    smem = std::max(smem, batch_tab_bytes<T>() + sm);
  }
  auto go = [&](auto kernel) -> int {
    CEED_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0, dev = 0, nsm = 0;
    CEED_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, L.threads, smem));
    CEED_CUDA_CHECK(cudaGetDevice(&dev));
    CEED_CUDA_CHECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    if (per_sm < 1) return fail(CEED_ERR_UNSUPPORTED, "batched kernel does not fit on an SM");
    unsigned grid = (unsigned)(per_sm * nsm);
    if (L.grid > 0 && L.grid < grid) grid = L.grid;
    // cooperative launch: the runtime refuses it unless every block of the grid can be resident at
    // once (pieces are taken in order, so the waits between colours end with fewer, too; they are bounded all the same)
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(L.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    CEED_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kernel, b));
    if (grid_used) *grid_used = grid;
    return CEED_OK;
  };
  // (the double-float operator included: unlike its single-mesh kernel it runs fastest without a
  // register cap here -- 7.2 / 7.7 GDOF/s at 1 / 4 right-hand sides; 6.1 at 128 registers, the orders then inlined)
  if (colloc) return L.stage ? go(batch_kernel<OP, T, TQ, true, true>) : go(batch_kernel<OP, T, TQ, false, true>);
  return L.stage ? go(batch_kernel<OP, T, TQ, true, false>) : go(batch_kernel<OP, T, TQ, false, false>);
}

}  // namespace ceedgb
