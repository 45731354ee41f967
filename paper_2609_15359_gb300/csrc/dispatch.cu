// dispatch.cu -- global memory-aware dispatch (Sec. 3.3, Algorithm 1).
//
// Horizon SNAPSHOT.  For candidate j with live steps u_j and decoder k the
// peak is p_j + 1 + M_k(u_j) with M_k(u) = max_{t<u}(K[k][t] + t): one prefix
// maximum per decoder, shared by every candidate.  Writing A_k(u) =
// cap_k - 1 - M_k(u), decoder k is feasible for j iff p_j <= A_k(u_j) and the
// headroom is A_k(u_j) - p_j.  The rule (smallest Q among feasible decoders,
// else largest headroom, ties to the lowest index) then needs, per horizon
// column u, only
//   * PMq_u[i] = max over the first i+1 decoders in (Q, index) order of
//     A_k(u): the first position where it reaches p_j is the chosen decoder;
//   * max_k A_k(u) and its lowest arg-max for the fallback.
// So K is read at most once, tile by tile over the horizon (only the tiles
// holding some candidate's last live step), with all D rows of a tile staged
// in shared memory by one TMA copy; the carry of the prefix maximum into a
// tile comes from a per-decoder scan of the 16-step summary; per column the
// arg-max comes first, a candidate above every A_k is decided at once, and
// PMq is built only where some candidate fits, each of those then costing a
// binary search over D instead of D scores.  Candidates are first bucketed by
// the tile of their last live step so each tile serves its own.  Three
// launches: the carry scan and the bucket counts (independent, one launch),
// the bucket scatter, the scoring kernel.
//
// SEQUENTIAL (reservation after each choice) and the literal Algorithm 1
// modes are separate kernels below.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>

#include "maps_internal.cuh"
#include "maps_bench.h"

namespace maps {
namespace {

constexpr int kMaxD = 1024;
constexpr int kMainThreads = 256;
constexpr int kBoxRows = 256;  // TMA box height limit

// ---------------------------------------------------------------------------
// TMA / mbarrier primitives (inline PTX)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile(
      "{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(
          smem_u32(bar)),
      "r"(bytes)
      : "memory");
}
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for a barrier phase; false if the bound expired.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
  for (uint32_t spins = 0; !mbar_test_wait(bar, parity); ++spins) {
    if (spins > kSpinLimit) return false;
    __nanosleep(20);
  }
  return true;
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// ---------------------------------------------------------------------------
// SNAPSHOT preparation.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int candidate_steps(int32_t U, int H) {
  return U < 1 ? 1 : (U > H ? H : U);
}

constexpr int kSumBlock = 16;      // steps per kmax summary entry
constexpr int kUnitCands = 1024;   // candidates per work unit of the main kernel

// kmax[k][b] = max over the 16 steps of block b of K[k][t] + t, for callers
// that do not pass the summary from maps_project_occupancy.
__global__ void __launch_bounds__(256)
kmax_from_K_kernel(int D, int H, const int32_t *__restrict__ K, uint32_t *__restrict__ kmax,
                   int32_t *status) {
  pdl_prologue();
  const int64_t nb = (static_cast<int64_t>(H) + kSumBlock - 1) / kSumBlock;
  const int64_t total = nb * D;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  bool neg = false;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t k = i / nb, b = i - k * nb;
    const int32_t *row = K + k * H;
    const int64_t t0 = b * kSumBlock;
    uint32_t m = 0;
    for (int c = 0; c < kSumBlock; ++c) {
      const int64_t t = t0 + c;
      if (t >= H) break;
      const int32_t v = __ldg(row + t);
      if (v < 0) neg = true;
      const uint32_t x = static_cast<uint32_t>(v) + static_cast<uint32_t>(t);
      m = x > m ? x : m;
    }
    kmax[i] = m;
  }
  if (neg) flag_error(status, MAPS_E_RANGE);
}

// The same summary for the SEQUENTIAL walk, with the maxima of its 128-step chunks
// (eight blocks, eight lanes' maxima).
constexpr int kSeqChunk = 128;
__global__ void __launch_bounds__(256)
seq_summary_kernel(int D, int H, const int32_t *__restrict__ K, uint32_t *__restrict__ km,
                   uint32_t *__restrict__ cm, int32_t *status) {
  pdl_prologue();
  const int64_t nb = (static_cast<int64_t>(H) + kSumBlock - 1) / kSumBlock;
  const int64_t nch = (static_cast<int64_t>(H) + kSeqChunk - 1) / kSeqChunk;
  const int64_t total = 8 * nch * D;  // lanes: whole chunks
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int lane = threadIdx.x & 31;
  bool neg = false;
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x - lane; i0 < total; i0 += stride) {
    const int64_t i = i0 + lane, ch = i >> 3, k = ch / nch, b = (ch - k * nch) * 8 + (i & 7);
    uint32_t m = 0;
    if (i < total && b < nb) {
      const int32_t *row = K + k * H;
#pragma unroll
      for (int c = 0; c < kSumBlock; ++c) {
        const int64_t t = b * kSumBlock + c;
        const int32_t v = t < H ? __ldg(row + t) : 0;
        if (v < 0) neg = true;
        if (t < H) m = max(m, static_cast<uint32_t>(v) + static_cast<uint32_t>(t));
      }
      km[k * nb + b] = m;
    }
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 4));
    if (i < total && (lane & 7) == 0) cm[ch] = m;
  }
  if (neg) flag_error(status, MAPS_E_RANGE);
}

// A caller's summary is compared with K at four blocks of every row (the
// first, the last, the middle and one that varies with the decoder); a
// mismatch there is reported, any other gives unspecified results.
__device__ __forceinline__ bool summary_matches(const int32_t *__restrict__ K,
                                                const uint32_t *__restrict__ kmax, int H, int64_t nb,
                                                int k, int which) {
  const int64_t b = which == 0 ? 0 : which == 1 ? nb - 1 : which == 2 ? nb / 2 : (k * 7919LL) % nb;
  const int32_t *kr = K + static_cast<int64_t>(k) * H;
  const int64_t t_end = (b + 1) * kSumBlock < H ? (b + 1) * kSumBlock : static_cast<int64_t>(H);
  long long mx = -1;
  for (int64_t t = b * kSumBlock; t < t_end; ++t) {
    const long long v = static_cast<long long>(__ldg(kr + t)) + t;
    mx = v > mx ? v : mx;
  }
  return mx >= 0 && static_cast<uint32_t>(mx) == __ldg(kmax + k * nb + b);
}

// carry[k][i] = max of K[k][t] + t over t < i*W2 (0 for i = 0): the prefix
// maximum that horizon tile i inherits from the tiles before it.  One block
// per decoder; each thread reads 16 consecutive summary entries at once
// (whole tiles, as W2/16 divides 16), keeps its tiles' maxima in registers,
// and after a block scan writes its tiles' carries (the decoder's row of the
// carries is contiguous; a work unit later reads one word per decoder).
__device__ void carry_scan_block(int kk, int D, int H, int W2, int T2, const int32_t *__restrict__ K,
                                 bool check_kmax, const uint32_t *__restrict__ kmax,
                                 uint32_t *__restrict__ carry,
                                 const int32_t *__restrict__ Q, const int32_t *__restrict__ cap,
                                 int32_t *sig, int32_t *rank_of, int32_t *capq, int32_t *status) {
  __shared__ uint32_t s_w[8];
  __shared__ int s_rank;
  {
    // this decoder's position in (Q, index) order: the decoders before it
    const int32_t qk = __ldg(Q + kk);
    int r = 0;
    for (int k2 = threadIdx.x; k2 < D; k2 += blockDim.x) {
      const int32_t q2 = __ldg(Q + k2);
      r += (q2 < qk) || (q2 == qk && k2 < kk);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
    if (threadIdx.x == 0) s_rank = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_rank, r);
    __syncthreads();
    if (threadIdx.x == 0) {
      const int32_t ck = __ldg(cap + kk);
      if ((qk | ck) < 0) flag_error(status, MAPS_E_RANGE);
      sig[s_rank] = kk;
      rank_of[kk] = s_rank;
      capq[s_rank] = ck;
    }
  }
  constexpr int kPer = 16;
  const int k = kk;
  const int64_t nb = (static_cast<int64_t>(H) + kSumBlock - 1) / kSumBlock;
  const int bpt = W2 / kSumBlock;  // summary blocks per tile (1..16)
  const uint32_t *row = kmax + static_cast<int64_t>(k) * nb;
  uint32_t *out = carry + static_cast<int64_t>(k) * T2;  // carry[k][i], tile-contiguous per decoder
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool vec = (reinterpret_cast<uintptr_t>(row) % 16) == 0;
  uint32_t run = 0;
  for (int64_t c0 = 0; c0 < nb; c0 += 256 * kPer) {
    const int64_t b0 = c0 + threadIdx.x * kPer;
    uint32_t v[kPer];
    if (vec && b0 + kPer <= nb) {
#pragma unroll
      for (int q = 0; q < kPer; q += 4) {
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(row + b0 + q));
        v[q] = x.x, v[q + 1] = x.y, v[q + 2] = x.z, v[q + 3] = x.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < kPer; ++q) v[q] = b0 + q < nb ? __ldg(row + b0 + q) : 0u;
    }
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) m = v[q] > m ? v[q] : m;
    uint32_t incl = m;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl = y > incl ? y : incl;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    uint32_t r = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) r = 0;
    uint32_t all = 0;
    for (int w = 0; w < 8; ++w) {
      if (w < warp) r = s_w[w] > r ? s_w[w] : r;
      all = s_w[w] > all ? s_w[w] : all;
    }
    r = r > run ? r : run;
    // this thread's tiles: [b0 / bpt, (b0 + kPer) / bpt)
    const int64_t tile0 = b0 / bpt;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (q % bpt == 0) {
        const int64_t ti = tile0 + q / bpt;
        if (ti < T2) out[ti] = r;
      }
      r = v[q] > r ? v[q] : r;
    }
    run = all > run ? all : run;
    __syncthreads();
  }
  if (check_kmax && threadIdx.x < 4 && !summary_matches(K, kmax, H, nb, k, threadIdx.x))
    flag_error(status, MAPS_E_INVALID);
}

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Candidates are bucketed by the horizon tile holding their last live step
// u_j - 1.  When the tile count fits in shared memory each block first counts
// its candidates per tile locally and then adds one global count per
// non-empty tile; otherwise lanes with the same tile combine their atomic.
// Grid-stride loops run in whole warps.
constexpr int kBinSmem = 4096;

struct Unit {
  int32_t tile, start, count, pad;
};

__device__ void bin_scan_block(int T2, const uint32_t *tcount, uint32_t *toff, Unit *units,
                               uint32_t *nunits);

// Counting block b of nblk.
__device__ void bin_count_block(int b, int nblk, int64_t J, int H, int W2, int T2,
                                const int32_t *__restrict__ cp, const int32_t *__restrict__ cb,
                                uint32_t *tcount, int32_t *choice, int64_t *headroom,
                                int32_t *status, uint32_t *ticket, uint32_t *toff, Unit *units,
                                uint32_t *nunits) {
  __shared__ uint32_t s_h[kBinSmem];
  __shared__ bool s_last;
  const bool local = T2 <= kBinSmem;
  if (local)
    for (int i = threadIdx.x; i < T2; i += blockDim.x) s_h[i] = 0;
  __syncthreads();
  const int64_t stride = static_cast<int64_t>(nblk) * blockDim.x;
  bool bad = false;
  for (int64_t j0 = static_cast<int64_t>(b) * blockDim.x; j0 < J; j0 += stride) {
    const int64_t j = j0 + threadIdx.x;
    int tile = -1;
    if (j < J) {
      const int32_t p = cp[j], U = cb[j];
      if ((p | U) < 0) {
        bad = true;
        choice[j] = -1;
        if (headroom) headroom[j] = 0;
      } else {
        tile = (candidate_steps(U, H) - 1) / W2;
      }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, tile);
    if (tile >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1)
      atomicAdd(local ? &s_h[tile] : &tcount[tile], static_cast<uint32_t>(__popc(peers)));
  }
  if (bad) flag_error(status, MAPS_E_RANGE);
  if (local) {
    __syncthreads();
    // start each block's flush at a different tile so blocks do not collide
    const int rot = static_cast<int>((static_cast<int64_t>(b) * 97) % T2);
    for (int i = threadIdx.x; i < T2; i += blockDim.x) {
      const int t = (i + rot) % T2;
      if (s_h[t]) atomicAdd(&tcount[t], s_h[t]);
    }
  }
  // the last block to finish turns the counts into offsets and work units
  // (one thread publishes the block's counts: the barrier orders every
  // thread's atomics before its fence, as a grid barrier does)
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == static_cast<uint32_t>(nblk) - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    bin_scan_block(T2, tcount, toff, units, nunits);
  }
}

// The two independent first steps in one launch: blocks [0, D) scan the
// carries of decoder blockIdx.x, the others count the candidates per tile.
__global__ void __launch_bounds__(256)
dispatch_prep_kernel(int ncarry, int D, int H, int W2, int T2, const int32_t *__restrict__ K,
                     bool check_kmax, const uint32_t *__restrict__ kmax,
                     uint32_t *__restrict__ carry, const int32_t *__restrict__ Q,
                     const int32_t *__restrict__ cap, int32_t *sig, int32_t *rank_of,
                     int32_t *capq, int64_t J, const int32_t *__restrict__ cp,
                     const int32_t *__restrict__ cb, uint32_t *tcount, int32_t *choice,
                     int64_t *headroom, int32_t *status, uint32_t *ticket, uint32_t *toff,
                     Unit *units, uint32_t *nunits) {
  pdl_prologue();
  if (static_cast<int>(blockIdx.x) < ncarry)
    carry_scan_block(blockIdx.x, D, H, W2, T2, K, check_kmax, kmax, carry, Q, cap, sig, rank_of,
                     capq, status);
  else
    bin_count_block(blockIdx.x - ncarry, gridDim.x - ncarry, J, H, W2, T2, cp, cb, tcount, choice,
                    headroom, status, ticket, toff, units, nunits);
}

// Run by the last counting block (any multiple of 32 threads up to 1024):
// tile offsets toff[0..T2] and the work units (a tile with c candidates gives
// ceil(c / kUnitCands) units; the unit count goes to *nunits).
__device__ void bin_scan_block(int T2, const uint32_t *tcount, uint32_t *toff, Unit *units,
                               uint32_t *nunits) {
  __shared__ uint32_t s_w[2][32];
  const int nt = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // each thread takes a contiguous run of tiles: one block scan in all
  const int per = (T2 + nt - 1) / nt;
  const int i0 = min(T2, static_cast<int>(threadIdx.x) * per), i1 = min(T2, i0 + per);
  uint32_t sc = 0, su = 0;
  for (int i = i0; i < i1; ++i) {
    const uint32_t c = __ldcg(tcount + i);
    sc += c;
    su += (c + kUnitCands - 1) / kUnitCands;
  }
  uint32_t ic = sc, iu = su;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t yc = __shfl_up_sync(0xffffffffu, ic, off);
    const uint32_t yu = __shfl_up_sync(0xffffffffu, iu, off);
    if (lane >= off) {
      ic += yc;
      iu += yu;
    }
  }
  if (lane == 31) {
    s_w[0][warp] = ic;
    s_w[1][warp] = iu;
  }
  __syncthreads();
  uint32_t rc = ic - sc, ru = iu - su;  // exclusive starts of this thread's run
  for (int w = 0; w < warp; ++w) {
    rc += s_w[0][w];
    ru += s_w[1][w];
  }
  for (int i = i0; i < i1; ++i) {
    const uint32_t c = __ldcg(tcount + i);
    const uint32_t nu = (c + kUnitCands - 1) / kUnitCands;
    toff[i] = rc;
    for (uint32_t q = 0; q < nu; ++q) {
      Unit un;
      un.tile = i;
      un.start = static_cast<int32_t>(rc + q * kUnitCands);
      un.count = static_cast<int32_t>(min(static_cast<uint32_t>(kUnitCands), c - q * kUnitCands));
      un.pad = 0;
      units[ru + q] = un;
    }
    rc += c;
    ru += nu;
  }
  if (threadIdx.x == nt - 1) {  // the last thread's run ends at the totals
    toff[T2] = rc;
    *nunits = ru;
  }
}

// Place every valid candidate into its tile's bucket as (index, prompt,
// steps).  The order inside a bucket does not matter: each candidate's
// decision depends only on itself.
__global__ void __launch_bounds__(256)
bin_scatter_kernel(int64_t J, int H, int W2, int T2, const int32_t *__restrict__ cp,
                   const int32_t *__restrict__ cb, const uint32_t *toff, uint32_t *tcursor,
                   int32_t *ord, int32_t *sp, int32_t *su) {
  // The candidates are the caller's input and the grid before this one (the
  // counting kernel of the same call) writes only the workspace and the
  // call's outputs; it starts only once every earlier grid has completed.  So
  // this thread's first candidate is loaded before the wait on it.
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t b0 = static_cast<int64_t>(blockIdx.x) * blockDim.x;
  const int64_t j_first = b0 + threadIdx.x;
  const int32_t p_first = j_first < J ? cp[j_first] : -1;
  const int32_t u_first = j_first < J ? cb[j_first] : -1;
  pdl_prologue();
  __shared__ uint32_t s_h[kBinSmem];  // local counts, then local cursors
  __shared__ uint32_t s_b[kBinSmem];  // this block's base inside each bucket
  const bool local = T2 <= kBinSmem;
  if (local) {
    for (int i = threadIdx.x; i < T2; i += blockDim.x) s_h[i] = 0;
    __syncthreads();
    for (int64_t j0 = b0; j0 < J; j0 += stride) {
      const int64_t j = j0 + threadIdx.x;
      int tile = -1;
      if (j < J) {
        const int32_t U = j0 == b0 ? u_first : cb[j];
        if (((j0 == b0 ? p_first : cp[j]) | U) >= 0) tile = (candidate_steps(U, H) - 1) / W2;
      }
      const unsigned peers = __match_any_sync(0xffffffffu, tile);
      if (tile >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1)
        atomicAdd(&s_h[tile], static_cast<uint32_t>(__popc(peers)));
    }
    __syncthreads();
    const int rot = static_cast<int>((static_cast<int64_t>(blockIdx.x) * 97) % T2);
    for (int i = threadIdx.x; i < T2; i += blockDim.x) {
      const int t = (i + rot) % T2;
      const uint32_t c = s_h[t];
      s_b[t] = c ? toff[t] + atomicAdd(&tcursor[t], c) : 0u;
      s_h[t] = 0;
    }
    __syncthreads();
  }
  for (int64_t j0 = b0; j0 < J; j0 += stride) {
    const int64_t j = j0 + threadIdx.x;
    int tile = -1, u = 0;
    int32_t p = 0;
    if (j < J) {
      p = j0 == b0 ? p_first : cp[j];
      const int32_t U = j0 == b0 ? u_first : cb[j];
      if ((p | U) >= 0) {
        u = candidate_steps(U, H);
        tile = (u - 1) / W2;
      }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, tile);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if (tile >= 0 && (threadIdx.x & 31) == leader) {
      const uint32_t c = static_cast<uint32_t>(__popc(peers));
      base = local ? s_b[tile] + atomicAdd(&s_h[tile], c) : toff[tile] + atomicAdd(&tcursor[tile], c);
    }
    base = __shfl_sync(0xffffffffu, base, leader);
    if (tile >= 0) {
      const uint32_t pos = base + __popc(peers & lanemask_lt());
      ord[pos] = static_cast<int32_t>(j);
      sp[pos] = p;
      su[pos] = u;
    }
  }
}

// ---------------------------------------------------------------------------
// SNAPSHOT main kernel: one CTA per work unit, a unit being (tile, a slice of
// the tile's candidates).  Tiles without candidates are never read: their
// contribution reaches later tiles through the carry, built from the summary.
// Several CTAs share an SM, so one CTA's TMA wait overlaps another's work.
// ---------------------------------------------------------------------------
struct SnapArgs {
  int D, H, W2, T2, Drows, boxes, box_rows;  // Drows = rows per staged tile (>= D)
  int tile_stride;                           // elements of the tile buffer (1 KB multiple)
  int comp_off;                              // words from the tile buffer to comp
  int region;                                // words from the tile buffer to the small arrays
  bool alias;                                // comp overwrites the tile (one row per thread)
  bool use_tma;
  const int32_t *K;
  const int32_t *sig, *rank_of, *capq;  // queue order
  const uint32_t *carry;                // [D][T2]
  const Unit *units;
  const uint32_t *nunits;
  const int32_t *ord, *sp, *su;
  int32_t *choice;
  int64_t *headroom;
  int32_t *status;
};

template <int W2>
__global__ void __launch_bounds__(kMainThreads, 4)
dispatch_snapshot_kernel(const __grid_constant__ CUtensorMap tmap, SnapArgs a) {
  pdl_prologue();
  extern __shared__ __align__(1024) unsigned char smem[];
  const int unit = blockIdx.x;
  if (unit >= static_cast<int>(*a.nunits)) return;
  const int D = a.D, H = a.H;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarpsM = kMainThreads / 32;
  uint32_t *kb = reinterpret_cast<uint32_t *>(smem);
  // comp[slot][i]: M of decoder sig[i] at the slot's column, then rewritten
  // in place into the queue-ordered prefix maximum of A (clamped at -1).
  // Rows are D + 1 words apart so that one row's writes to several slots fall
  // on different banks.
  const int Dp = D + 1;
  uint32_t *comp = kb + a.comp_off;
  int32_t *s_capq = reinterpret_cast<int32_t *>(kb + a.region);
  int32_t *s_sig = s_capq + D;
  int32_t *s_rank = s_sig + D;
  uint32_t *s_carry = reinterpret_cast<uint32_t *>(s_rank + D);
  int32_t *s_slot = reinterpret_cast<int32_t *>(s_carry + D);  // [W2] column -> slot (-1 none)
  int32_t *s_argA = s_slot + W2;                               // [W2]
  long long *s_maxA = reinterpret_cast<long long *>(
      (reinterpret_cast<uintptr_t>(s_argA + W2) + 15) & ~uintptr_t(15));  // [W2]
  uint64_t *s_bar = reinterpret_cast<uint64_t *>(s_maxA + W2);
  long long *s_segA = reinterpret_cast<long long *>(s_bar + 1);      // [8][32]
  int32_t *s_segrun = reinterpret_cast<int32_t *>(s_segA + kWarpsM * 32);  // [8][32]
  int32_t *s_segK = s_segrun + kWarpsM * 32;                          // [8][32]
  int32_t *s_need = s_segK + kWarpsM * 32;                            // [W2] column needs PMq
  int32_t *s_needlist = s_need + W2;                                  // [W2]
  __shared__ int s_nslots, s_abort, s_nneed;

  const Unit un = a.units[unit];
  const int64_t t0 = static_cast<int64_t>(un.tile) * W2;
  if (tid == 0) {
    s_abort = 0;
    if (a.use_tma) {
      mbar_init(s_bar, 1);
      fence_mbar_init();
      // every box is credited in full, rows past D included (zero-filled)
      mbar_expect_tx(s_bar, static_cast<uint32_t>(a.boxes) * a.box_rows * W2 * 4u);
      for (int b = 0; b < a.boxes; ++b)
        tma_load_2d(kb + static_cast<size_t>(b) * a.box_rows * W2, &tmap, s_bar, un.tile * W2,
                    b * a.box_rows);
    }
  }
  // queue order, capacities and this tile's carries; columns this unit needs
  for (int k = tid; k < D; k += kMainThreads) {
    s_sig[k] = __ldg(a.sig + k);
    s_rank[k] = __ldg(a.rank_of + k);
    s_capq[k] = __ldg(a.capq + k);
    s_carry[k] = __ldg(a.carry + static_cast<int64_t>(k) * a.T2 + un.tile);
  }
  for (int c = tid; c < W2; c += kMainThreads) s_slot[c] = 0;
  __syncthreads();
  for (int q0 = 0; q0 < un.count; q0 += kMainThreads * 8) {
    int32_t uu[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {  // issue the loads together
      const int q = q0 + i * kMainThreads + tid;
      uu[i] = q < un.count ? __ldg(a.su + un.start + q) : 0;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (uu[i] > 0) s_slot[uu[i] - 1 - t0] = 1;
  }
  if (!a.use_tma) {
    for (int e = tid; e < D * W2; e += kMainThreads) {
      const int r = e / W2, c = e - (e / W2) * W2;
      const int64_t t = t0 + c;
      // 32-column tiles use the layout of a 128-byte swizzled TMA copy
      const int at = W2 == 32 ? r * 32 + ((((c >> 2) ^ (r & 7))) << 2) + (c & 3) : e;
      kb[at] = t < H ? static_cast<uint32_t>(a.K[static_cast<int64_t>(r) * H + t]) : 0u;
    }
  }
  __syncthreads();
  if (warp == 0) {  // compact the flagged columns (W2 <= 256)
    int run = 0;
    for (int c0 = 0; c0 < W2; c0 += 32) {
      const int c = c0 + lane;
      const bool f = c < W2 && s_slot[c] != 0;
      const unsigned bal = __ballot_sync(0xffffffffu, f);
      if (c < W2) s_slot[c] = f ? run + __popc(bal & lanemask_lt()) : -1;
      run += __popc(bal);
    }
    if (lane == 0) s_nslots = run;
  }
  if (a.use_tma && !mbar_wait_bounded(s_bar, 0)) {
    if (tid == 0) flag_error(a.status, MAPS_E_TIMEOUT);
    s_abort = 1;
  }
  __syncthreads();
  if (s_abort) {
    // a copy may still land: wait for it once more (bounded) before leaving
    mbar_wait_bounded(s_bar, 0);
    return;
  }
  const int nslots = s_nslots;

  // --- prefix maximum of K + t along each row; keep the needed columns ----
  bool neg = false;
  if (W2 == 32 && a.alias) {
    // One row per thread (D <= kMainThreads): every row is read into registers
    // first, then, after a barrier, comp is written over the tile.
    const int row = tid;
    const bool live = row < D;
    uint4 q[8];
    if (live) {
      const uint4 *rp = reinterpret_cast<const uint4 *>(kb + static_cast<size_t>(row) * 32);
#pragma unroll
      for (int ch = 0; ch < 8; ++ch) q[ch] = rp[ch ^ (row & 7)];
    }
    __syncthreads();  // the tile has been read: its space becomes comp
    if (live) {
      uint32_t run = s_carry[row];
      const int rk = s_rank[row];
#pragma unroll
      for (int ch = 0; ch < 8; ++ch) {
        const uint32_t raw[4] = {q[ch].x, q[ch].y, q[ch].z, q[ch].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int c = ch * 4 + e;
          const int64_t t = t0 + c;
          if (t < H) {
            if (static_cast<int32_t>(raw[e]) < 0) neg = true;
            const uint32_t x = raw[e] + static_cast<uint32_t>(t);  // K + t < 2^32
            run = x > run ? x : run;
          }
          const int sl = s_slot[c];
          if (sl >= 0) comp[static_cast<size_t>(sl) * Dp + rk] = run;
        }
      }
    }
  } else if constexpr (W2 == 32) {
    // One thread per row.  The tile is stored with 128-byte swizzling: the
    // 16-byte chunk ch of row r sits at chunk ch ^ (r & 7) of its 128-byte
    // row, so a warp loading one chunk of 32 rows hits every bank once per
    // quarter-warp.  The running maximum starts from the row's carry.
    for (int row = tid; row < D; row += kMainThreads) {
      const uint4 *rp = reinterpret_cast<const uint4 *>(kb + static_cast<size_t>(row) * 32);
      uint32_t run = s_carry[row];
      const int rk = s_rank[row];
#pragma unroll
      for (int ch = 0; ch < 8; ++ch) {
        const uint4 q = rp[ch ^ (row & 7)];
        const uint32_t raw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int c = ch * 4 + e;
          const int64_t t = t0 + c;
          if (t < H) {
            if (static_cast<int32_t>(raw[e]) < 0) neg = true;
            const uint32_t x = raw[e] + static_cast<uint32_t>(t);  // K + t < 2^32
            run = x > run ? x : run;
          }
          const int sl = s_slot[c];
          if (sl >= 0) comp[static_cast<size_t>(sl) * Dp + rk] = run;
        }
      }
    }
  } else {
    constexpr int seg = W2 / 16;  // cells per row segment; 16 segments per row
    const int items = ((D * 16 + kMainThreads - 1) / kMainThreads) * kMainThreads;
    for (int it = tid; it < items; it += kMainThreads) {
      const int row = it >> 4, sg = it & 15;
      const bool live_row = row < D;
      uint32_t v[seg];
      uint32_t run = 0;
#pragma unroll
      for (int j = 0; j < seg; ++j) {
        const int c = sg * seg + j;
        const int64_t t = t0 + c;
        uint32_t x = 0;
        if (live_row && t < H) {
          const uint32_t raw = kb[static_cast<size_t>(row) * W2 + c];
          if (static_cast<int32_t>(raw) < 0) neg = true;
          x = raw + static_cast<uint32_t>(t);  // K + t < 2^32
        }
        run = x > run ? x : run;
        v[j] = run;
      }
      uint32_t incl = run;
#pragma unroll
      for (int off = 1; off < 16; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off, 16);
        if (sg >= off) incl = y > incl ? y : incl;
      }
      uint32_t excl = __shfl_up_sync(0xffffffffu, incl, 1, 16);
      if (sg == 0) excl = 0;
      if (live_row) {
        const uint32_t cr = s_carry[row];
        const int rk = s_rank[row];
        excl = excl > cr ? excl : cr;
#pragma unroll
        for (int j = 0; j < seg; ++j) {
          const int sl = s_slot[sg * seg + j];
          if (sl >= 0) comp[static_cast<size_t>(sl) * Dp + rk] = v[j] > excl ? v[j] : excl;
        }
      }
    }
  }
  if (neg) flag_error(a.status, MAPS_E_RANGE);
  __syncthreads();

  // --- per needed column: arg-max of A, then (where some candidate can be
  // placed) the prefix maximum of A in queue order ---------------------------
  // Columns go 32 at a time, lane c taking column cb + c; warp w takes the
  // w-th eighth of the queue positions, in order.  Rows are D + 1 words apart,
  // so a warp's 32 columns fall on 32 banks.
  {
    const int L = (D + kWarpsM - 1) / kWarpsM;
    const int i0 = warp * L, i1 = min(D, i0 + L);
    // (1) the best (A, decoder) of each column: each segment's, then warp 0
    // combines the eight
    for (int cb = 0; cb < nslots; cb += 32) {
      const int sl = cb + lane;
      const bool live = sl < nslots;
      const uint32_t *col = comp + static_cast<size_t>(live ? sl : 0) * Dp;
      long long bA = LLONG_MIN;
      int bK = 0x7fffffff;
      if (live)
        for (int i = i0; i < i1; ++i) {
          const long long A = static_cast<long long>(s_capq[i]) - 1 - static_cast<long long>(col[i]);
          const int k = s_sig[i];
          if (A > bA || (A == bA && k < bK)) {
            bA = A;
            bK = k;
          }
        }
      s_segA[warp * 32 + lane] = bA;
      s_segK[warp * 32 + lane] = bK;
      __syncthreads();
      if (live && warp == 0) {
        for (int w = 1; w < kWarpsM; ++w) {
          const long long yA = s_segA[w * 32 + lane];
          const int yK = s_segK[w * 32 + lane];
          if (yA > bA || (yA == bA && yK < bK)) {
            bA = yA;
            bK = yK;
          }
        }
        s_maxA[sl] = bA;
        s_argA[sl] = bK;
        s_need[sl] = 0;
      }
      __syncthreads();  // the segment arrays serve the next 32 columns
    }
    // (2) a candidate that fits no decoder (p above its column's best A) is
    // decided here (most headroom); the others mark their column
    for (int q = tid; q < un.count; q += kMainThreads) {
      const int32_t p = __ldg(a.sp + un.start + q);
      const int sl = s_slot[__ldg(a.su + un.start + q) - 1 - t0];
      if (static_cast<long long>(p) <= s_maxA[sl]) {
        s_need[sl] = 1;
      } else {
        const int j = __ldg(a.ord + un.start + q);
        a.choice[j] = s_argA[sl];
        if (a.headroom) a.headroom[j] = s_maxA[sl] - p;
      }
    }
    __syncthreads();
    if (warp == 0) {  // compact them
      int run = 0;
      for (int c0 = 0; c0 < nslots; c0 += 32) {
        const int sl = c0 + lane;
        const bool f = sl < nslots && s_need[sl] != 0;
        const unsigned bal = __ballot_sync(0xffffffffu, f);
        if (f) s_needlist[run + __popc(bal & lanemask_lt())] = sl;
        run += __popc(bal);
      }
      if (lane == 0) s_nneed = run;
    }
    __syncthreads();
    // (3) for those: a running maximum of A (clamped at -1) per segment,
    // written in place, then each segment raised to the maximum of the
    // segments before it
    const int nneed = s_nneed;
    for (int cb = 0; cb < nneed; cb += 32) {
      const bool live = cb + lane < nneed;
      const int sl = live ? s_needlist[cb + lane] : 0;
      uint32_t *col = comp + static_cast<size_t>(sl) * Dp;
      int32_t run = -1;
      if (live)
        for (int i = i0; i < i1; ++i) {
          const long long A = static_cast<long long>(s_capq[i]) - 1 - static_cast<long long>(col[i]);
          const int32_t a32 = A < -1 ? -1 : static_cast<int32_t>(A);
          run = a32 > run ? a32 : run;
          col[i] = static_cast<uint32_t>(run);
        }
      s_segrun[warp * 32 + lane] = run;
      __syncthreads();
      if (live) {
        int32_t ex = -1;
        for (int w = 0; w < warp; ++w) ex = max(ex, s_segrun[w * 32 + lane]);
        if (ex > -1)
          for (int i = i0; i < i1; ++i) {
            const int32_t v = static_cast<int32_t>(col[i]);
            if (v < ex) col[i] = static_cast<uint32_t>(ex);
          }
      }
      __syncthreads();
    }
  }

  // --- the candidates that fit some decoder (loads issued together, then the
  // searches); the others were decided above ----------------------------------
  for (int q0 = 0; s_nneed > 0 && q0 < un.count; q0 += kMainThreads * 8) {
    int32_t pp[8], uu[8], jj[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int q = q0 + i * kMainThreads + tid;
      const bool ok = q < un.count;
      pp[i] = ok ? __ldg(a.sp + un.start + q) : 0;
      uu[i] = ok ? __ldg(a.su + un.start + q) : 0;
      jj[i] = ok ? __ldg(a.ord + un.start + q) : -1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (jj[i] < 0) continue;
      const int32_t p = pp[i];
      const int c = static_cast<int>(uu[i] - 1 - t0);
      const int sl = s_slot[c];
      if (s_maxA[sl] < p) continue;  // nothing feasible: decided above
      const int32_t *pm = reinterpret_cast<const int32_t *>(comp) + static_cast<size_t>(sl) * Dp;
      int l = 0, r = D - 1;  // first queue position whose prefix reaches p
      while (l < r) {
        const int mid = (l + r) >> 1;
        if (pm[mid] >= p)
          r = mid;
        else
          l = mid + 1;
      }
      a.choice[jj[i]] = s_sig[l];
      if (a.headroom) a.headroom[jj[i]] = static_cast<long long>(pm[l]) - p;
    }
  }
}

// ---------------------------------------------------------------------------
// SNAPSHOT of few candidates (direct_fits): one launch instead of a memset and
// three.  One to eight warps take a candidate and score its decoders, a slice
// each: per decoder M, the maximum of the 16-step summary below u by all the
// lanes, and of at most 15 cells.  Nothing is bucketed and nothing carried, at the
// price of reading each row's summary once a candidate, from L2.
//
// The grid also reads K once for negative values, and compares a caller's
// summary with K at four blocks of every row, as the bucketed form does.
// ---------------------------------------------------------------------------
constexpr int kDirectWarps = 8;
constexpr int kDirectRows = 8;

// At most this many (candidate, decoder) scores, decoders counted as whole groups of
// kDirectRows a warp, twice as many (without that) times the 2,048-step spans of the
// horizon, cells of K, and a horizon.
// Candidates of a few hundred steps decide where the lines lie; in brackets the
// same with all of them through the horizon, which no size tells the host.
// Measured, one launch against four: 4 decoders, H 4,096, 32 candidates 4.7
// against 13.1 us (5.2; 12.9); 16, 16,381, 1,021: 7.2 against 20.6 (11.2; 18.6);
// 100, 8,192, 600: 12.1 against 16.4 (19.2; 16.5); 64, 4,096, 2,048: 16.2 against
// 18.6; 1, 30,000, 8,192: 10.7 against 20.5 (25.9; 17.5).  Past the lines: 16,
// 2,048, 16,384: 25.9 against 20.7; 256, 2,048, 1,024: 22.6 against 18.4; 2, 100,
// 24,000: 19.9 against 17.5; 2, 256, 65,536: 40.9 against 19.1; 18, 104, 6,271: 24.6
// against 19.7; 12, 50,000, 100: 7.8 against 16.4, but 63 against 14.5.  Where the
// summary's rows are no whole 16-byte words (330 decoders, H 2,760, 256 candidates:
// 10.9 against 24.6) a lane has four words in flight as well; with one, 28.5.
constexpr int64_t kDirectScores = 1 << 17;
constexpr int64_t kDirectCells = 1 << 20;
constexpr int kDirectH = 32768;
// warps a candidate: as many as have kDirectRows rows each
int direct_share(int D) {
  int share = 1;
  while (share < kDirectWarps && share * kDirectRows < D) share *= 2;
  return share;
}
bool direct_fits(int D, int H, int64_t J) {
  const int step = direct_share(D) * kDirectRows;
  return J * ((D + step - 1) / step * step) <= kDirectScores &&
         J * D * std::max(1, H / 2048) <= 2 * kDirectScores && H <= kDirectH &&
         static_cast<int64_t>(D) * H <= kDirectCells;
}

template <bool VEC>
__global__ void __launch_bounds__(32 * kDirectWarps)
dispatch_direct_kernel(int D, int H, const int32_t *__restrict__ K, const uint32_t *__restrict__ kmax,
                       int check_kmax, const int32_t *__restrict__ cap, const int32_t *__restrict__ Q,
                       int64_t J, const int32_t *__restrict__ cp, const int32_t *__restrict__ cb,
                       int32_t *__restrict__ choice, int64_t *__restrict__ headroom, int32_t *status,
                       int share) {
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ unsigned long long s_key[kDirectWarps];
  __shared__ long long s_h[kDirectWarps];
  pdl_prologue();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nb = (static_cast<int64_t>(H) + kSumBlock - 1) / kSumBlock;
  // this warp's candidate of the block's, and its decoders [d0, d1)
  const int per = kDirectWarps / share, mine = warp / share, part = warp % share;
  const int slice = ((D + share - 1) / share + kDirectRows - 1) / kDirectRows * kDirectRows;
  const int d0 = min(D, part * slice), d1 = min(D, d0 + slice);
  for (int64_t j0 = static_cast<int64_t>(blockIdx.x) * per; j0 < J; j0 += static_cast<int64_t>(gridDim.x) * per) {
    const int64_t j = j0 + mine;
    const int32_t p = j < J ? __ldg(cp + j) : -1, U = j < J ? __ldg(cb + j) : -1;
    unsigned long long best = ~0ull;  // infeasible << 63 | Q or deficit << 10 | decoder
    long long best_h = 0;
    if ((p | U) >= 0) {
      const int u = candidate_steps(U, H);
      const int nfull = u / kSumBlock, rem = u - nfull * kSumBlock;
      // kDirectRows rows at a time, their loads in flight together; lane i
      // keeps the M of the i-th of 32 rows
      for (int k0 = d0; k0 < d1; k0 += 32) {
        uint32_t M = 0;
        for (int i0 = 0; i0 < 32 && k0 + i0 < d1; i0 += kDirectRows) {
          uint32_t m[kDirectRows];
#pragma unroll
          for (int i = 0; i < kDirectRows; ++i) {
            const int k = min(k0 + i0 + i, D - 1), t = nfull * kSumBlock + lane;
            m[i] = lane < rem ? static_cast<uint32_t>(__ldg(K + static_cast<int64_t>(k) * H + t)) +
                                    static_cast<uint32_t>(t)
                              : 0u;
          }
          const uint32_t *km = kmax + static_cast<int64_t>(k0 + i0) * nb;
          const int64_t rows = D - 1 - (k0 + i0);  // the last row's distance
          if (VEC) {  // rows are whole 16-byte words
            for (int b = 4 * lane; b < nfull; b += 128) {
              uint4 v[kDirectRows];
#pragma unroll
              for (int i = 0; i < kDirectRows; ++i)
                v[i] = __ldg(reinterpret_cast<const uint4 *>(km + (i < rows ? i : rows) * nb + b));
#pragma unroll
              for (int i = 0; i < kDirectRows; ++i) {
                m[i] = max(m[i], v[i].x);
                if (b + 1 < nfull) m[i] = max(m[i], v[i].y);
                if (b + 2 < nfull) m[i] = max(m[i], v[i].z);
                if (b + 3 < nfull) m[i] = max(m[i], v[i].w);
              }
            }
          } else {
            for (int b = lane; b < nfull; b += 128) {  // one by one: four in flight a lane, too
              uint32_t v[4][kDirectRows];
#pragma unroll
              for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < kDirectRows; ++i)
                  v[q][i] = b + 32 * q < nfull ? __ldg(km + (i < rows ? i : rows) * nb + b + 32 * q) : 0u;
#pragma unroll
              for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < kDirectRows; ++i) m[i] = max(m[i], v[q][i]);
            }
          }
#pragma unroll
          for (int i = 0; i < kDirectRows; ++i) {
            const uint32_t r = __reduce_max_sync(kAll, m[i]);
            if (lane == i0 + i) M = r;
          }
        }
        if (k0 + lane < d1) {
          const int k = k0 + lane;
          const long long h = static_cast<long long>(__ldg(cap + k)) - (static_cast<long long>(p) + 1 + M);
          const unsigned long long v =
              h >= 0 ? static_cast<unsigned long long>(__ldg(Q + k)) & 0xffffffffull
                     : (1ull << 53) | static_cast<unsigned long long>(-h);
          const unsigned long long key = (v << 10) | static_cast<unsigned>(k);
          if (key < best) {
            best = key;
            best_h = h;
          }
        }
      }
    }
    unsigned long long all = best;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long y = __shfl_xor_sync(kAll, all, off);
      all = y < all ? y : all;
    }
    if (best == all && (best != ~0ull || lane == 0)) {  // the best decoder's lane (keys are unique)
      s_key[warp] = best;
      s_h[warp] = best_h;
    }
    __syncthreads();
    if (part == 0 && lane == 0 && j < J) {
      int w = warp;
      for (int i = 1; i < share; ++i)
        if (s_key[warp + i] < s_key[w]) w = warp + i;
      const bool ok = (p | U) >= 0;
      if (!ok) flag_error(status, MAPS_E_RANGE);
      choice[j] = ok ? static_cast<int32_t>(s_key[w] & 1023u) : -1;
      if (headroom) headroom[j] = ok ? s_h[w] : 0;
    }
    __syncthreads();  // the keys serve the block's next candidates
  }
  bool bad = false;
  const int64_t gt = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t nt = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t k = gt; k < D; k += nt)
    if ((__ldg(cap + k) | __ldg(Q + k)) < 0) bad = true;
  if (check_kmax) {  // the summary pass of a call without one reports these
    const int64_t cells = static_cast<int64_t>(D) * H;
    int32_t any = 0;
    if ((reinterpret_cast<uintptr_t>(K) & 15) == 0) {
#pragma unroll 4
      for (int64_t i = gt; i < cells / 4; i += nt) {
        const int4 v = __ldg(reinterpret_cast<const int4 *>(K) + i);
        any |= v.x | v.y | v.z | v.w;
      }
      if (gt < cells % 4) any |= __ldg(K + cells - 1 - gt);
    } else {
      for (int64_t i = gt; i < cells; i += nt) any |= __ldg(K + i);
    }
    if (any < 0) bad = true;
    for (int64_t e = gt; e < 4ll * D; e += nt) {
      const int k = static_cast<int>(e >> 2);
      if (!summary_matches(K, kmax, H, nb, k, static_cast<int>(e & 3))) flag_error(status, MAPS_E_INVALID);
    }
  }
  if (bad) flag_error(status, MAPS_E_RANGE);
}

// ---------------------------------------------------------------------------
// SEQUENTIAL horizon dispatch: one block walks the candidates in order.
// With F_k(t) = K[k][t] + t, scoring decoder k needs M_k(u) = max_{t<u} F_k(t);
// reserving the footprint adds p + t + 1 to F_k*(t) for t < u.
//
// The walk is one chain of dependent decisions, so its cost is a decision's
// latency: the instructions and barriers on the chain, at five to six cycles
// an instruction for a warp.  A decision takes one barrier.  In phase j
//   * each row warp picks candidate j's decoder (all the same one) from the
//     scores of the phase before, adds the footprint to its chunk (128 steps)
//     of that row and takes the maximum of F below the next candidate's u over
//     it: together the chosen decoder's score for candidate j + 1.  A booking
//     warp picks too, and writes the outputs;
//   * the column warps, four lanes a decoder, meanwhile score every decoder for
//     candidate j + 1.  Only the row being written may be read half updated,
//     and its entry is the one that the row warps' maximum replaces.
// A score is the maximum of the chunk maxima below u, at most 7 maxima of 16
// steps, 3 of 4 and 3 cells: one kind to each of the four lanes.  The first P0
// steps of each row with these maxima live in shared memory, the steps past
// them in L2 (with maxima of 16 steps), where a candidate costs some L2 round
// trips; a warp of the chosen row has two of its chunks there in flight, four
// consecutive steps a lane.  (One chunk, with lanes on consecutive steps: 64 decoders,
// H 32,763, candidates of up to 6,000 steps 2.84 against 2.08 us a decision.)  Rows
// are loaded as far as a candidate reaches, and the chunks' maxima come from the
// summary's kernel: a single candidate through the horizon of 200 decoders, H 32,768,
// 37 us against 122 with them made here (and 42 by the walk in global memory alone).
//
// The 32-bit pick keys, the smallest wins: a feasible decoder is
// min(Q - q0, lim) << kb | k, an infeasible one 1 << 31 |
// min(M - cap - x0, lim) << kb | k, q0 and x0 lower bounds for the whole call
// (Q and K only grow, and M >= K[k][0]).  If even the smallest key is at lim
// the pick is made on 64-bit keys.
//
// Measured, occupancy and walk: 16 decoders, H 16,384, 1,024 candidates 3.51 ->
// 0.58 ms; 64 decoders, H 32,763, 2,003 candidates 8.1 -> 1.18 ms.  Before, one
// block scored every decoder from global memory with four barriers a decision
// (3.4 and 4.0 us each).  Forms in between: two warps a decoder, each scoring
// and reserving in lockstep, 1.58 and 4.44 ms (issue bound: every warp ran the
// whole pick); one chain warp reserving alone, 1.34 and 1.86 ms; a lane a
// decoder in the columns and the pick and its bookkeeping in every row warp,
// 0.93 and 1.68 ms.
// ---------------------------------------------------------------------------
constexpr int kRowWarps = 8;
constexpr int kColWarps = 16;  // at most
constexpr int kSeqWords = 9;    // per-decoder words beside the rows
__host__ __device__ constexpr int seq_dw(int D) { return (D + 31) / 32 * 32; }

struct SeqArgs {
  int D, H;
  int P0;              // resident steps of a row (whole chunks)
  int P2;              // chunks whose maxima are resident
  int ncol;            // column warps
  int kb, mc;
  int32_t *K;
  uint32_t *km;        // [D][ceil(H/16)]  max of F per 16 steps
  uint32_t *cm;        // [D][ceil(H/128)]  max of F per chunk; kept up to date from chunk P2 on
  const int32_t *cap;
  int32_t *Q;
  int64_t J;
  const int32_t *cp, *cb;
  int32_t *choice;
  int64_t *headroom;
  int32_t *status;
};

// Shared memory of a row: F, the maxima of 4, of 16 and of 128 steps, each with
// four words of padding (16-byte reads of eight rows then spread over the
// banks).  A score reads up to 8 words from any place of a row's part, hence
// the padding at the end of all of them.
constexpr int kSeqPad = 16;
__host__ __device__ constexpr int seq_ldc(int P2) { return (P2 + 3) / 4 * 4 + 4; }
__host__ __device__ constexpr int64_t seq_row_words(int64_t P0, int P2) {
  return P0 + P0 / 4 + P0 / 16 + 12 + seq_ldc(P2);
}

// The packed 64-bit decision key, the smallest wins: inf << 63 | v << 10 | k.
// mc (rank by headroom alone) puts every decoder in the infeasible class, by
// 2^33 - h (positive: h <= cap < 2^31).
__device__ __forceinline__ unsigned long long seq_key64(long long h, int32_t q, int k, int mc) {
  const bool feas = h >= 0 && !mc;
  const unsigned long long v = feas ? static_cast<unsigned long long>(q)
                               : mc ? static_cast<unsigned long long>((1ll << 33) - h)
                                    : static_cast<unsigned long long>(-h);
  return (feas ? 0ull : 1ull << 63) | (v << 10) | static_cast<unsigned>(k);
}

__device__ __forceinline__ void seq_bar(int warps) {
  asm volatile("bar.sync 1, %0;" ::"r"(32 * warps) : "memory");
}

__device__ __forceinline__ uint32_t max4(uint4 v) { return max(max(v.x, v.y), max(v.z, v.w)); }
// the larger of m and the first n of v (n may be below 0 or above 4)
__device__ __forceinline__ uint32_t max4_below(uint4 v, int n, uint32_t m) {
  if (n > 0) m = max(m, v.x);
  if (n > 1) m = max(m, v.y);
  if (n > 2) m = max(m, v.z);
  if (n > 3) m = max(m, v.w);
  return m;
}

// RD: decoders per lane of a pick, 0 for any number.
template <int RD>
__global__ void __launch_bounds__(1024, 1)
dispatch_sequential_kernel(const __grid_constant__ SeqArgs a) {
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ __align__(16) uint32_t seq_smem[];
  __shared__ int2 s_cand[64];           // (p, u) of candidate i at i mod 64; u = 0: none or invalid
  __shared__ __align__(16) uint32_t s_part[2][kRowWarps];  // the chosen row's maxima, per row warp
  __shared__ int4 s_crit[2];            // its (cap, Q, off)
  __shared__ int s_q0, s_umax, s_wide;
  __shared__ long long s_x0;
  pdl_prologue();
  const int D = a.D, H = a.H, P0 = a.P0, P2 = a.P2, mc = a.mc, kb = a.kb;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nwarp = 32;
  const int64_t nb = (static_cast<int64_t>(H) + kSumBlock - 1) / kSumBlock;
  const int64_t nch = (static_cast<int64_t>(H) + kSeqChunk - 1) / kSeqChunk;
  // per-decoder words first (Dw, D in whole warps): (key, M) of each decoder for a
  // candidate by its parity, the queue length behind that key, capacity, queue
  // length, and off (M + off is the infeasible key term)
  const int Dw = seq_dw(D);
  uint2 *const s_col = reinterpret_cast<uint2 *>(seq_smem);  // [2][Dw]
  int32_t *const words = reinterpret_cast<int32_t *>(seq_smem + 4 * Dw);
  int32_t *const s_colq = words;                              // [2][Dw]
  int32_t *const s_cap = words + 2 * Dw, *const s_q = words + 3 * Dw, *const s_off = words + 4 * Dw;
  // then the rows; offsets in words
  const int ldF = P0 + 4, ld4 = P0 / 4 + 4, ld16 = P0 / 16 + 4, ldc = seq_ldc(P2);
  const int o4 = D * ldF, o16 = o4 + D * ld4, oc = o16 + D * ld16;
  uint32_t *const F = seq_smem + kSeqWords * Dw;
  // --- capacities, the first candidates ---------------------------------------
  if (tid == 0) {
    s_q0 = 0x7fffffff;
    s_x0 = LLONG_MAX;
    s_umax = s_wide = 0;
  }
  for (int k = D + tid; k < Dw; k += blockDim.x) s_col[k] = s_col[Dw + k] = make_uint2(~0u, 0u);
  __syncthreads();
  bool bad = false;
  for (int k = tid; k < D; k += blockDim.x) {
    const int32_t ck = a.cap[k], qk = a.Q[k];
    if ((ck | qk) < 0) bad = true;  // K < 0 is reported by the summary pass
    s_cap[k] = ck;
    s_q[k] = qk;
    atomicMin(&s_q0, qk);
    atomicMin(&s_x0, static_cast<long long>(a.K[static_cast<int64_t>(k) * H]) - ck);
  }
  auto load_cand = [&](int64_t j) {
    const int32_t p = j < a.J ? __ldg(a.cp + j) : -1, U = j < a.J ? __ldg(a.cb + j) : -1;
    return (p | U) < 0 ? make_int2(0, 0) : make_int2(p, candidate_steps(U, H));
  };
  int umax = 0;
  for (int64_t j = tid; j < a.J; j += blockDim.x) {
    const int2 c = load_cand(j);
    umax = max(umax, c.y);
    if (c.y == 0) {
      bad = true;
      a.choice[j] = -1;
      if (a.headroom) a.headroom[j] = 0;
    }
  }
  umax = __reduce_max_sync(kAll, umax);
  if (lane == 0) atomicMax(&s_umax, umax);
  if (tid < 64) s_cand[tid] = load_cand(tid);
  __syncthreads();
  // --- the resident rows, as far as a candidate reaches, two chunks in flight ----
  const int rch = P0 / kSeqChunk;  // resident chunks of a row
  const int lch = min(rch, (s_umax + kSeqChunk - 1) / kSeqChunk);
  for (int e0 = warp; e0 < D * lch; e0 += 2 * nwarp) {
    uint32_t x[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = min(e0 + h * nwarp, D * lch - 1), k = e / lch, t0 = (e - k * lch) * kSeqChunk;
      const int32_t *row = a.K + static_cast<int64_t>(k) * H + t0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int t = 32 * i + lane;
        x[h][i] = t0 + t < H ? static_cast<uint32_t>(row[t]) + static_cast<uint32_t>(t0 + t) : 0u;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = e0 + h * nwarp, k = e / lch, t0 = (e - k * lch) * kSeqChunk;
      if (e >= D * lch) break;
      uint32_t *const f = F + k * ldF + t0;
#pragma unroll
      for (int i = 0; i < 4; ++i) f[32 * i + lane] = x[h][i];
      __syncwarp();
      uint32_t m = max4(reinterpret_cast<const uint4 *>(f)[lane]);
      F[o4 + k * ld4 + t0 / 4 + lane] = m;
      m = max(m, __shfl_xor_sync(kAll, m, 1));
      m = max(m, __shfl_xor_sync(kAll, m, 2));
      if ((lane & 3) == 0) F[o16 + k * ld16 + t0 / 16 + (lane >> 2)] = m;
    }
  }
  const int cmax = min(s_umax >> 7, P2);  // scores read the chunk maxima below this one
#pragma unroll 4
  for (int e = tid; e < cmax * D; e += blockDim.x) {
    const int k = e / cmax, c = e - k * cmax;
    F[oc + k * ldc + c] = __ldcg(a.cm + k * nch + c);
  }
  const long long x0 = s_x0;
  for (int k = tid; k < D; k += blockDim.x) {
    const long long off = -(x0 + s_cap[k]);
    s_off[k] = static_cast<int32_t>(off);
    // M < 2^31 + 2^28 while K is within int32: M + off cannot wrap
    if (off > (1ll << 30) || off < INT_MIN) s_wide = 1;
  }
  __syncthreads();
  const int32_t q0 = s_q0;
  const uint32_t kmask = (1u << kb) - 1u;
  // key terms stop at lim (no key is ~0); 0 where the terms need more bits
  const uint32_t lim = s_wide ? 0u : (1u << (31 - kb)) - 2u;
  const uint32_t lim_key = lim << kb;
  auto key32 = [&](uint32_t M, int32_t p, int32_t cap, int32_t q, int32_t off, int k) {
    const int32_t room = mc ? 0 : max(cap - p, 0);  // p + 1 + M <= cap: M < cap - p
    const bool feas = M < static_cast<uint32_t>(room);
    const uint32_t term = feas ? static_cast<uint32_t>(q - q0) : M + static_cast<uint32_t>(off);
    return (feas ? 0u : 0x80000000u) + (min(term, lim) << kb) + static_cast<uint32_t>(k);
  };
  // a column's lane: which maxima of its decoder it reads, as the first n words
  // from a place of the row's part: w = u >> sh, n = w & low, place w & ~low
  const int part = lane & 3;
  const int sh = part == 0 ? 7 : part == 1 ? 4 : part == 2 ? 2 : 0;
  const int low = part == 0 ? -1 : part == 1 ? 7 : 3;
  const int ldp = part == 0 ? ldc : part == 1 ? ld16 : part == 2 ? ld4 : ldF;
  const int op = part == 0 ? oc : part == 1 ? o16 : part == 2 ? o4 : 0;
  struct ColLane {  // what a lane keeps of its decoder
    int k, kc;
    int32_t cap, off;
    const uint32_t *part;  // its part of the decoder's row
  };
  auto col_lane = [&](int k) {
    ColLane c;
    c.k = k, c.kc = min(k, D - 1);
    c.cap = s_cap[c.kc], c.off = s_off[c.kc];
    c.part = F + op + c.kc * ldp;
    return c;
  };
  auto score_col = [&](int64_t j, const ColLane &cl) {  // four lanes a decoder
    const int2 cd = s_cand[j & 63];
    const int u = cd.y;
    const bool in = u < P0;  // its chunk is resident (P0 is whole chunks)
    const int w = u >> sh;
    const int n = part == 0 ? min(w, P2) : in ? w & low : 0;
    const uint32_t *b = cl.part + (in ? w & ~low : 0);
    const uint4 v0 = *reinterpret_cast<const uint4 *>(b), v1 = *reinterpret_cast<const uint4 *>(b + 4);
    uint32_t m = max4_below(v1, n - 4, max4_below(v0, n, 0u));
    if (n > 8)
      for (int i = 8; i < n; i += 4) m = max4_below(*reinterpret_cast<const uint4 *>(b + i), n - i, m);
    if (u >= P0) {
      if ((u & (kSeqChunk - 1)) != 0) {  // the last chunk in global memory
        const int c = u >> 7, n16 = (u >> 4) & 7, t0 = u & ~15;
        const uint32_t *bg = a.km + cl.kc * nb + c * 8;
        const int32_t *row = a.K + static_cast<int64_t>(cl.kc) * H + t0;
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (part + 4 * i < n16) m = max(m, bg[part + 4 * i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int t = part + 4 * i;
          if (t < (u & 15)) m = max(m, static_cast<uint32_t>(row[t]) + static_cast<uint32_t>(t0 + t));
        }
      }
      for (int c = P2 + part; c < (u >> 7); c += 4) m = max(m, a.cm[cl.kc * nch + c]);
    }
    m = max(m, __shfl_xor_sync(kAll, m, 1));
    m = max(m, __shfl_xor_sync(kAll, m, 2));
    const int32_t q = s_q[cl.kc];
    const uint32_t key = key32(m, cd.x, cl.cap, q, cl.off, cl.k);
    if (part == 0 && cl.k < D) {
      const int at = (j & 1) ? Dw + cl.k : cl.k;
      s_col[at] = make_uint2(key, m);
      s_colq[at] = q;
    }
  };
  for (int k0 = warp * 8; k0 < D; k0 += nwarp * 8) score_col(0, col_lane(k0 + (lane >> 2)));
  __syncthreads();

  // The pick of candidate j (with p) at phase parity par: the decoder, and this
  // lane's best key and its M; `best` is that key in the winner's lane alone.
  // The entry of decoder kprev, chosen before, comes from the row warps.
  auto pick = [&](int p, int par, int kprev, uint32_t &best, uint32_t &key, uint32_t &M) {
    const uint4 pa = *reinterpret_cast<const uint4 *>(&s_part[par ^ 1][0]);
    const uint4 pb = *reinterpret_cast<const uint4 *>(&s_part[par ^ 1][4]);
    const int4 cr = s_crit[par ^ 1];
    const uint32_t cM = max(max4(pa), max4(pb));
    const uint32_t ckey = key32(cM, p, cr.x, cr.y, cr.z, kprev);
    key = ~0u;
    M = 0;
    auto take = [&](int k) {
      uint2 e = s_col[par * Dw + k];
      if (k == kprev) e = make_uint2(ckey, cM);
      M = e.x < key ? e.y : M;
      key = min(key, e.x);
    };
    if (RD > 0) {
#pragma unroll
      for (int i = 0; i < (RD > 0 ? RD : 1); ++i) take(32 * i + lane);
    } else {
#pragma unroll 4
      for (int k = lane; k < D; k += 32) take(k);
    }
    best = __reduce_min_sync(kAll, key);
    if ((best & 0x7fffffffu) < lim_key) return static_cast<int>(best & kmask);
    unsigned long long k64 = ~0ull;  // the wide keys
    for (int k = lane; k < D; k += 32) {
      const uint32_t Mk = k == kprev ? cM : s_col[par * Dw + k].y;
      const int32_t qk = k == kprev ? cr.y : s_colq[par * Dw + k];
      const unsigned long long y =
          seq_key64(static_cast<long long>(s_cap[k]) - (static_cast<long long>(p) + 1 + Mk), qk, k, mc);
      if (y < k64) {
        k64 = y;
        M = Mk;
        key = static_cast<uint32_t>(k);  // this lane's best decoder
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long y = __shfl_xor_sync(kAll, k64, off);
      k64 = y < k64 ? y : k64;
    }
    best = static_cast<uint32_t>(k64 & 1023u);
    return static_cast<int>(best);
  };

  const int walkers = kRowWarps + 1 + a.ncol;  // warps of the per-decision barrier
  if (warp < kRowWarps) {
    int kprev = -1;  // the decoder chosen before
    int2 c1 = s_cand[0];
    const bool res0 = warp < rch;           // this warp's first chunk is resident
    const int tb = warp * kSeqChunk, tl = tb + 4 * lane;
    const int later = res0 ? tb + kRowWarps * kSeqChunk : tb;  // where its other chunks begin
    // its first chunk in global memory
    const int cg = (rch > warp ? (rch - warp + kRowWarps - 1) / kRowWarps * kRowWarps : 0) + warp;
    for (int64_t j = 0; j < a.J; ++j) {
      const int2 cd = c1;
      c1 = s_cand[(j + 1) & 63];
      const int p = cd.x, u = cd.y, u1 = c1.y, ue = max(u, u1);
      const int par = static_cast<int>(j & 1);
      int kk = -1;
      if (u > 0) {
        uint32_t best, key, M;
        kk = pick(p, par, kprev, best, key, M);
        uint32_t m1 = 0, bm0 = 0;
        uint32_t *const fr = F + kk * ldF + 4 * lane;
        auto add_to = [&](uint4 &v, int t) {  // the footprint on steps t.. t + 3 below u
          const uint32_t x = static_cast<uint32_t>(p) + 1u + static_cast<uint32_t>(t);
          const int n = u - t;
          v.x += n > 0 ? x : 0u;
          v.y += n > 1 ? x + 1u : 0u;
          v.z += n > 2 ? x + 2u : 0u;
          v.w += n > 3 ? x + 3u : 0u;
        };
        auto set_cm = [&](int c, uint32_t m) {
          if (c < P2)
            F[oc + kk * ldc + c] = m;
          else
            a.cm[kk * nch + c] = m;
        };
        auto fold = [&](int c, uint32_t bm) {  // the chunk's maxima, from its 4-step ones
          F[o4 + kk * ld4 + c * 32 + lane] = bm;
          bm = max(bm, __shfl_xor_sync(kAll, bm, 1));
          bm = max(bm, __shfl_xor_sync(kAll, bm, 2));
          if ((lane & 3) == 0) F[o16 + kk * ld16 + c * 8 + (lane >> 2)] = bm;
          bm = __reduce_max_sync(kAll, bm);
          if (lane == 0) set_cm(c, bm);
        };
        if (res0 && tb < ue) {
          uint4 v = *reinterpret_cast<const uint4 *>(fr + tb);
          add_to(v, tl);
          m1 = max4_below(v, u1 - tl, 0u);
          bm0 = max4(v);  // folded once the score is published
          if (tb < u) *reinterpret_cast<uint4 *>(fr + tb) = v;
        }
        // the later chunks of a long horizon: one branch on the chain of the others
        if (__builtin_expect(later < ue, 0)) {
          for (int c = warp + kRowWarps; c < rch && c * kSeqChunk < ue; c += kRowWarps) {
            const int t0 = c * kSeqChunk;
            uint4 v = *reinterpret_cast<const uint4 *>(fr + t0);
            add_to(v, t0 + 4 * lane);
            m1 = max4_below(v, u1 - (t0 + 4 * lane), m1);
            if (t0 < u) {
              *reinterpret_cast<uint4 *>(fr + t0) = v;
              fold(c, max4(v));
            }
          }
          // those in global memory, two in flight, four consecutive steps a lane
          for (int c0 = cg; c0 * kSeqChunk < ue; c0 += 2 * kRowWarps) {
            int32_t *const row = a.K + static_cast<int64_t>(kk) * H;
            uint4 v[2];
  #pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int t0 = (c0 + h * kRowWarps) * kSeqChunk, t = t0 + 4 * lane;
              v[h] = make_uint4(0, 0, 0, 0);
              if (t0 >= ue) continue;
              if (t < H) v[h].x = static_cast<uint32_t>(row[t]);
              if (t + 1 < H) v[h].y = static_cast<uint32_t>(row[t + 1]);
              if (t + 2 < H) v[h].z = static_cast<uint32_t>(row[t + 2]);
              if (t + 3 < H) v[h].w = static_cast<uint32_t>(row[t + 3]);
            }
  #pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int c = c0 + h * kRowWarps, t0 = c * kSeqChunk, t = t0 + 4 * lane;
              if (t0 >= ue) break;
              add_to(v[h], t);
              if (t0 < u) {
                if (t < u) row[t] = static_cast<int32_t>(v[h].x);
                if (t + 1 < u) row[t + 1] = static_cast<int32_t>(v[h].y);
                if (t + 2 < u) row[t + 2] = static_cast<int32_t>(v[h].z);
                if (t + 3 < u) row[t + 3] = static_cast<int32_t>(v[h].w);
              }
              // F = K + t on the steps within the horizon
              const uint32_t te = static_cast<uint32_t>(t);
              v[h].x += t < H ? te : 0u;
              v[h].y += t + 1 < H ? te + 1u : 0u;
              v[h].z += t + 2 < H ? te + 2u : 0u;
              v[h].w += t + 3 < H ? te + 3u : 0u;
              m1 = max4_below(v[h], u1 - t, m1);
              if (t0 < u) {
                uint32_t f = max4(v[h]);
                f = max(f, __shfl_xor_sync(kAll, f, 1));
                f = max(f, __shfl_xor_sync(kAll, f, 2));
                const int b = (t0 >> 4) + (lane >> 2);
                if ((lane & 3) == 0 && b * kSumBlock < H) a.km[kk * nb + b] = f;
                f = __reduce_max_sync(kAll, f);
                if (lane == 0) set_cm(c, f);
              }
            }
          }
        }
        // publish, and fold the first chunk's maxima: one reduction, shuffle
        // and store in flight with another's
        if (res0 && tb < u) {
          const uint32_t b1 = max(bm0, __shfl_xor_sync(kAll, bm0, 1));
          m1 = __reduce_max_sync(kAll, m1);
          const uint32_t cm0 = __reduce_max_sync(kAll, bm0);
          const uint32_t b2 = max(b1, __shfl_xor_sync(kAll, b1, 2));
          if (lane == 0) s_part[par][warp] = m1;
          F[o4 + kk * ld4 + warp * 32 + lane] = bm0;
          if ((lane & 3) == 0) F[o16 + kk * ld16 + warp * 8 + (lane >> 2)] = b2;
          if (lane == 0) set_cm(warp, cm0);
        } else {
          m1 = __reduce_max_sync(kAll, m1);
          if (lane == 0) s_part[par][warp] = m1;
        }
      }
      kprev = kk;
      seq_bar(walkers);
    }
  } else if (warp == kRowWarps) {
    int kprev = -1;
    for (int64_t j = 0; j < a.J; ++j) {
      const int2 cd = s_cand[j & 63];
      const int p = cd.x, par = static_cast<int>(j & 1);
      int kk = -1;
      if (cd.y > 0) {
        uint32_t best, key, M;
        kk = pick(p, par, kprev, best, key, M);
        if (key == best) {  // the chosen decoder's lane books the decision
          const int32_t cap = s_cap[kk], q = s_q[kk];
          const int32_t qn = q == 0x7fffffff ? q : q + 1;
          s_q[kk] = qn;
          s_crit[par] = make_int4(cap, qn, s_off[kk], 0);
          a.choice[j] = kk;
          if (a.headroom)
            a.headroom[j] = static_cast<long long>(cap) - (static_cast<long long>(p) + 1 + M);
          // the largest new cell, K + p + t + 1, is M + p + 1
          if (q == 0x7fffffff || static_cast<long long>(p) + 1 + M > 0x7fffffffLL) bad = true;
        }
      }
      kprev = kk;
      seq_bar(walkers);
    }
  } else if (warp < walkers) {
    const int cw = warp - kRowWarps - 1;
    int2 cn = make_int2(0, 0);  // column warp 0: the 32 candidates of the next ring refill
    if (cw == 0) cn = load_cand(64 + lane);
    const ColLane mine = col_lane(cw * 8 + (lane >> 2));  // every column warp has some decoder
    for (int64_t j = 0; j < a.J; ++j) {
      if (cw == 0 && (j & 31) == 0 && j > 0) {
        s_cand[(j + 32 + lane) & 63] = cn;
        cn = load_cand(j + 64 + lane);
      }
      score_col(j + 1, mine);
      for (int k0 = (cw + a.ncol) * 8; k0 < D; k0 += 8 * a.ncol) score_col(j + 1, col_lane(k0 + (lane >> 2)));
      seq_bar(walkers);
    }
  }
  __syncthreads();
  if (bad) flag_error(a.status, MAPS_E_RANGE);
  for (int k = tid; k < D; k += blockDim.x) a.Q[k] = s_q[k];
  for (int k = warp; k < D; k += nwarp) {
    int32_t *row = a.K + static_cast<int64_t>(k) * H;
#pragma unroll 8
    for (int t = lane; t < lch * kSeqChunk && t < H; t += 32)
      row[t] = static_cast<int32_t>(F[k * ldF + t] - static_cast<uint32_t>(t));
  }
}

// ---------------------------------------------------------------------------
// Algorithm 1, literal.  Budgets: B_eff = floor(cap/S) - blocks held or
// reserved by the ongoing requests.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
alg1_budget_kernel(int D, int S, const int64_t *res_off, int64_t R, const int32_t *prompt,
                   const int32_t *gen, const int32_t *bound, const int32_t *cap,
                   long long *B_eff, int32_t *status) {
  pdl_prologue();
  __shared__ long long s_red[8];
  const int k = blockIdx.x;
  int64_t lo = res_off[k], hi = res_off[k + 1];
  if (lo < 0 || hi < lo || hi > R) {
    if (threadIdx.x == 0) flag_error(status, MAPS_E_RANGE);
    lo = hi = 0;
  }
  long long held = 0;
  bool bad = false;
  for (int64_t r = lo + threadIdx.x; r < hi; r += blockDim.x) {
    const int32_t p = prompt[r], g = gen[r], U = bound[r];
    if ((p | g | U) < 0) {
      bad = true;
      continue;
    }
    const long long reserve = static_cast<long long>(U) > static_cast<long long>(g) + 1
                                  ? static_cast<long long>(U)
                                  : static_cast<long long>(g) + 1;
    held += (static_cast<long long>(p) + reserve + S - 1) / S;
  }
  if (bad) flag_error(status, MAPS_E_RANGE);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) held += __shfl_xor_sync(0xffffffffu, held, off);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = held;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long tot = 0;
    for (int w = 0; w < 8; ++w) tot += s_red[w];
    B_eff[k] = static_cast<long long>(cap[k]) / S - tot;
  }
}

// SNAPSHOT: every block rebuilds the queue-ordered prefix maximum of B_eff
// (D <= 1024) and serves a slice of the candidates by binary search.
__global__ void __launch_bounds__(256)
alg1_snapshot_kernel(int D, int S, const long long *B_eff, const int32_t *cap, const int32_t *Q,
                     int64_t J, const int32_t *cp, const int32_t *cb, int32_t *choice,
                     int64_t *headroom, int32_t *status) {
  pdl_prologue();
  __shared__ long long s_B[kMaxD];
  __shared__ long long s_pm[kMaxD];
  __shared__ int s_sig[kMaxD];
  __shared__ long long s_maxB;
  __shared__ int s_argB;
  const int tid = threadIdx.x;
  bool bad = false;
  for (int k = tid; k < D; k += blockDim.x) {
    s_B[k] = B_eff[k];
    if ((cap[k] | Q[k]) < 0) bad = true;
    const int32_t qk = Q[k];
    int rank = 0;
    for (int k2 = 0; k2 < D; ++k2) {
      const int32_t q2 = Q[k2];
      rank += (q2 < qk) || (q2 == qk && k2 < k);
    }
    s_sig[rank] = k;
  }
  if (bad) flag_error(status, MAPS_E_RANGE);
  __syncthreads();
  if (tid < 32) {
    // warp 0: prefix max in queue order and arg-max in index order
    const int per = (D + 31) / 32, lo = tid * per, hi = min(D, lo + per);
    long long run = LLONG_MIN, bB = LLONG_MIN;
    int bK = 0x7fffffff;
    for (int i = lo; i < hi; ++i) {
      const long long x = s_B[s_sig[i]];
      run = x > run ? x : run;
    }
    for (int k = lo; k < hi; ++k)
      if (s_B[k] > bB) {
        bB = s_B[k];
        bK = k;
      }
    long long incl = run;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, incl, off);
      if (tid >= off) incl = y > incl ? y : incl;
    }
    long long excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (tid == 0) excl = LLONG_MIN;
    long long r2 = excl;
    for (int i = lo; i < hi; ++i) {
      const long long x = s_B[s_sig[i]];
      r2 = x > r2 ? x : r2;
      s_pm[i] = r2;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const long long yB = __shfl_xor_sync(0xffffffffu, bB, off);
      const int yK = __shfl_xor_sync(0xffffffffu, bK, off);
      if (yB > bB || (yB == bB && yK < bK)) {
        bB = yB;
        bK = yK;
      }
    }
    if (tid == 0) {
      s_maxB = bB;
      s_argB = bK;
    }
  }
  __syncthreads();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  bool badc = false;
  for (int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + tid; j < J; j += stride) {
    const int32_t p = cp[j], U = cb[j];
    if ((p | U) < 0) {
      badc = true;
      choice[j] = -1;
      if (headroom) headroom[j] = 0;
      continue;
    }
    const long long need = (static_cast<long long>(p) + U + S - 1) / S;  // Eq. (feasibility)
    int k;
    long long h;
    if (s_pm[D - 1] < need) {
      k = s_argB;  // nothing feasible: argmax B_eff
      h = s_maxB - need;
    } else {
      int l = 0, r = D - 1;  // argmin Q over the feasible set
      while (l < r) {
        const int mid = (l + r) >> 1;
        if (s_pm[mid] >= need)
          r = mid;
        else
          l = mid + 1;
      }
      k = s_sig[l];
      h = s_B[k] - need;
    }
    choice[j] = k;
    if (headroom) headroom[j] = h;
  }
  if (badc) flag_error(status, MAPS_E_RANGE);
}

// SEQUENTIAL: after each choice B_eff[k*] -= B_need, Q[k*] += 1.  The walk is
// one chain of dependent decisions, so its cost is a decision's latency.  One
// warp walks it with every decoder's budget and queue length in registers
// (decoder 32 i + lane is entry i of its lane): a decision is R selects, one
// 32-bit warp minimum and the winner's update, with no barrier and no memory
// on the chain (outputs wait in shared memory, a chunk of candidates' terms are
// loaded one chunk ahead).  64 decoders, 8,192 candidates: 0.44 ms, 54 ns a
// decision (102 ns with the outputs written and invalid candidates branched
// over on the chain).  One block of 1,024 threads with the budgets in shared
// memory, Q in global memory and two block barriers a decision took 20.3 ms.
//
// The 32-bit keys, the smallest wins: a feasible decoder is
// (Q - q0) << kb | k, an infeasible one 1 << 31 | (b0 - B_eff) << kb | k, with
// q0 the smallest Q and b0 the largest B_eff when the keys were last based and
// kb the bits of an index.  Both terms only grow; a chunk of 32 candidates is
// walked on them when neither can pass 31 - kb bits within it, else the keys
// are based anew, and a chunk that still does not fit (budgets further apart
// than about 2^31 / D) takes the wide comparison, on 64-bit budgets.
template <int R>
__global__ void __launch_bounds__(32)
alg1_sequential_kernel(int D, int S, const long long *B_eff, const int32_t *cap, int32_t *Q, int64_t J,
                       const int32_t *__restrict__ cp, const int32_t *__restrict__ cb,
                       int32_t *choice, int64_t *headroom, int32_t *status) {
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ int2 s_out[32];  // a chunk's choices and the chosen budgets (less b0)
  const int lane = threadIdx.x;
  pdl_prologue();
  long long B[R];  // budgets, exact at chunk boundaries
  int32_t q[R];
  bool bad = false;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int k = 32 * i + lane;
    B[i] = k < D ? B_eff[k] : LLONG_MIN;
    q[i] = k < D ? Q[k] : 0x7fffffff;
    if (k < D && (cap[k] | q[i]) < 0) bad = true;
  }
  int kb = 0;
  while ((1 << kb) < D) ++kb;
  const uint32_t kmask = (1u << kb) - 1u;
  const long long lim = (1ll << (31 - kb)) - 1;  // key terms stay below this (no key is ~0)
  long long b0 = 0, q0 = 0;                // the keys' bases
  long long bspan = lim, qspan = lim;      // bounds of the key terms (lim: not based yet)
  int64_t j = lane;
  int32_t p_n = j < J ? __ldg(cp + j) : 0, U_n = j < J ? __ldg(cb + j) : 0;
  for (int64_t j0 = 0; j0 < J; j0 += 32) {
    const int n = J - j0 < 32 ? static_cast<int>(J - j0) : 32;
    const int32_t p = p_n, U = U_n;
    j = j0 + 32 + lane;  // the next chunk's loads are in flight during this one
    p_n = j < J ? __ldg(cp + j) : 0;
    U_n = j < J ? __ldg(cb + j) : 0;
    const bool valid = lane < n && (p | U) >= 0;
    const unsigned vm = __ballot_sync(kAll, valid);
    if (lane < n && !valid) {
      bad = true;
      choice[j0 + lane] = -1;
      if (headroom) headroom[j0 + lane] = 0;
    }
    // Eq. (feasibility); at most 2^32 + S - 2 before the division
    const long long need = valid ? (static_cast<long long>(p) + U + S - 1) / S : 0;
    const uint32_t nmax = __reduce_max_sync(kAll, static_cast<uint32_t>(need));  // need < 2^32
    const long long grow = 32ll * nmax;
    // every term within its bits, and no queue length past int32, in this chunk
    auto fits = [&] {
      return bspan + grow < lim && qspan + 32 < lim && q0 + qspan + 32 <= 0x7fffffff;
    };
    if (!fits()) {  // base the keys anew
      long long bh = LLONG_MIN, bl = LLONG_MAX;
      int32_t ql = 0x7fffffff, qh = INT_MIN;
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (32 * i + lane < D) {
          bh = max(bh, B[i]);
          bl = min(bl, B[i]);
          ql = min(ql, q[i]);
          qh = max(qh, q[i]);
        }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        bh = max(bh, __shfl_xor_sync(kAll, bh, off));
        bl = min(bl, __shfl_xor_sync(kAll, bl, off));
      }
      ql = __reduce_min_sync(kAll, ql);
      qh = __reduce_max_sync(kAll, qh);
      b0 = bh;
      q0 = ql;
      // budgets are sums of at most 2^31 terms below 2^33: no difference wraps
      bspan = bh - bl;
      qspan = static_cast<long long>(qh) - ql;
    }
    if (fits()) {
      bspan += grow;
      qspan += 32;
      const long long th64 = need - b0;  // feasible: B - b0 >= need - b0
      const int32_t th_l = th64 > INT_MAX ? INT_MAX : th64 < INT_MIN ? INT_MIN : static_cast<int32_t>(th64);
      const uint32_t need_l = static_cast<uint32_t>(need);
      int32_t b[R];
      uint32_t fk[R], ik[R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const uint32_t k = 32 * i + lane;
        const bool has = k < static_cast<uint32_t>(D);
        b[i] = has ? static_cast<int32_t>(B[i] - b0) : INT_MIN;
        fk[i] = has ? (static_cast<uint32_t>(q[i] - q0) << kb) | k : ~0u;
        ik[i] = has ? 0x80000000u | (static_cast<uint32_t>(b0 - B[i]) << kb) | k : ~0u;
      }
      // the chain holds no branch and no memory: the next candidate's terms
      // are fetched a step ahead, the outputs wait in shared memory
      int32_t th = __shfl_sync(kAll, th_l, 0);
      uint32_t nd = __shfl_sync(kAll, need_l, 0);
#pragma unroll 4
      for (int c = 0; c < n; ++c) {
        const int32_t th1 = __shfl_sync(kAll, th_l, (c + 1) & 31);
        const uint32_t nd1 = __shfl_sync(kAll, need_l, (c + 1) & 31);
        const bool ok = ((vm >> c) & 1u) != 0;
        uint32_t sel[R];
        uint32_t m = ~0u;
#pragma unroll
        for (int i = 0; i < R; ++i) {
          sel[i] = b[i] >= th ? fk[i] : ik[i];
          m = min(m, sel[i]);
        }
        m = __reduce_min_sync(kAll, m);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const bool win = sel[i] == m && ok;  // keys are unique, and ~0 only on absent decoders
          if (win) s_out[c] = make_int2(static_cast<int32_t>(m & kmask), b[i]);
          const uint32_t d = win ? nd : 0u;
          b[i] -= static_cast<int32_t>(d);
          ik[i] += d << kb;
          fk[i] += win ? 1u << kb : 0u;
        }
        th = th1;
        nd = nd1;
      }
      __syncwarp();
      if (valid) {
        choice[j0 + lane] = s_out[lane].x;
        if (headroom) headroom[j0 + lane] = b0 + s_out[lane].y - need;
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (32 * i + lane < D) {
          B[i] = b0 + b[i];
          q[i] = static_cast<int32_t>(q0 + (fk[i] >> kb));
        }
      continue;
    }
    // wide: the smallest Q among the decoders that fit, else the largest
    // budget, each then by index
    bspan = qspan = lim;
    for (int c = 0; c < n; ++c) {
      const long long nd = __shfl_sync(kAll, need, c);
      if (!((vm >> c) & 1u)) continue;
      uint32_t qm = ~0u;  // Q >= 0 here (a negative one is a range error)
      long long bm = LLONG_MIN;
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (32 * i + lane < D) {
          if (B[i] >= nd) qm = min(qm, static_cast<uint32_t>(q[i]));
          bm = max(bm, B[i]);
        }
      qm = __reduce_min_sync(kAll, qm);
      const bool fit = qm != ~0u;
      if (!fit) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) bm = max(bm, __shfl_xor_sync(kAll, bm, off));
      }
      uint32_t kk = ~0u;
#pragma unroll
      for (int i = R - 1; i >= 0; --i)
        if (32 * i + lane < D && (fit ? B[i] >= nd && static_cast<uint32_t>(q[i]) == qm : B[i] == bm))
          kk = 32 * i + lane;
      kk = __reduce_min_sync(kAll, kk);
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (kk == static_cast<uint32_t>(32 * i + lane)) {
          choice[j0 + c] = static_cast<int32_t>(kk);
          if (headroom) headroom[j0 + c] = B[i] - nd;
          B[i] -= nd;
          if (q[i] == 0x7fffffff)
            bad = true;
          else
            q[i] += 1;
        }
    }
  }
  if (bad) flag_error(status, MAPS_E_RANGE);
#pragma unroll
  for (int i = 0; i < R; ++i)
    if (32 * i + lane < D) Q[32 * i + lane] = q[i];
}

// Few candidates on many decoders: a thread a decoder, the block's choice by a vote, a
// maximum and the lowest index that has it, 0.6 to 1 us a decision.  The warp above
// first takes 16 or 32 decoders a lane into registers, which a few decisions do not
// repay: replayed calls of 4 and 8 candidates, this form against the warp, 257
// decoders 5.3 and 7.3 us against 7.2 and 8.9; 1,024 8.3 and 12.1 against 19.0 and
// 18.6 (with the block's shared memory and Q in global memory 15.6 and 28.2).
constexpr int kFewCands = 8;
constexpr int kFewD = 256;
__global__ void __launch_bounds__(kMaxD)
alg1_few_kernel(int D, int S, const long long *B_eff, const int32_t *cap, int32_t *Q, int64_t J,
                const int32_t *__restrict__ cp, const int32_t *__restrict__ cb, int32_t *choice,
                int64_t *headroom, int32_t *status) {
  constexpr unsigned kAll = 0xffffffffu;
  pdl_prologue();
  __shared__ long long s_v[32];
  __shared__ unsigned s_k[32];
  const int k = threadIdx.x, lane = k & 31, warp = k >> 5, nw = blockDim.x >> 5;
  const bool has = k < D;
  long long B = has ? B_eff[k] : 0;
  int32_t q = has ? Q[k] : 0;
  bool bad = has && (cap[k] | q) < 0;
  for (int64_t j = 0; j < J; ++j) {
    const int32_t p = __ldg(cp + j), U = __ldg(cb + j);
    if ((p | U) < 0) {
      bad = true;
      if (k == 0) {
        choice[j] = -1;
        if (headroom) headroom[j] = 0;
      }
      continue;
    }
    const long long need = (static_cast<long long>(p) + U + S - 1) / S;  // Eq. (feasibility)
    const bool feas = has && B >= need;
    const bool any = __syncthreads_or(feas) != 0;
    // the largest wins: -Q among the decoders that fit, else the budget
    const bool in = any ? feas : has;
    const long long v = !in ? LLONG_MIN : any ? -static_cast<long long>(q) : B;
    long long m = v;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(kAll, m, off));
    if (lane == 0) s_v[warp] = m;
    __syncthreads();
    m = lane < nw ? s_v[lane] : LLONG_MIN;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_xor_sync(kAll, m, off));
    const unsigned mine = __reduce_min_sync(kAll, in && v == m ? static_cast<unsigned>(k) : ~0u);
    if (lane == 0) s_k[warp] = mine;
    __syncthreads();
    const unsigned kk = __reduce_min_sync(kAll, lane < nw ? s_k[lane] : ~0u);
    if (static_cast<unsigned>(k) == kk) {
      choice[j] = k;
      if (headroom) headroom[j] = B - need;
      B -= need;
      if (q == 0x7fffffff)
        bad = true;
      else
        q += 1;
    }
  }
  if (bad) flag_error(status, MAPS_E_RANGE);
  if (has) Q[k] = q;
}

using Alg1Seq = void (*)(int, int, const long long *, const int32_t *, int32_t *, int64_t, const int32_t *,
                         const int32_t *, int32_t *, int64_t *, int32_t *);
Alg1Seq alg1_sequential_for(int D) {
  return D <= 32    ? alg1_sequential_kernel<1>
         : D <= 64  ? alg1_sequential_kernel<2>
         : D <= 128 ? alg1_sequential_kernel<4>
         : D <= 256 ? alg1_sequential_kernel<8>
         : D <= 512 ? alg1_sequential_kernel<16>
                    : alg1_sequential_kernel<32>;
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct SnapGeom {
  int box_rows, boxes, Drows, W2, T2, tile_stride, comp_off, region;
  bool alias;
  size_t smem;
};

SnapGeom snap_geom(int D, int H) {
  SnapGeom g;
  g.box_rows = D < kBoxRows ? D : kBoxRows;
  g.boxes = (D + g.box_rows - 1) / g.box_rows;
  g.Drows = g.boxes * g.box_rows;
  int w = 256;
  while (w > 16 && static_cast<long long>(w) * g.Drows > 8192) w >>= 1;
  g.W2 = w;
  g.T2 = static_cast<int>((static_cast<long long>(H) + w - 1) / w);
  g.tile_stride = (g.Drows * w + 255) / 256 * 256;  // 1 KB-aligned buffer
  // with 32-column tiles and at most one row per thread, comp (the prefix
  // maxima, padded rows) overwrites the tile once every row is in registers
  const int comp_words = (D + 1) * w;
  g.alias = w == 32 && D <= kMainThreads;
  g.comp_off = g.alias ? 0 : g.tile_stride;
  g.region = g.alias ? std::max(g.tile_stride, comp_words) : g.tile_stride + comp_words;
  size_t b = static_cast<size_t>(g.region) * 4;       // K tile and comp
  b += 4 * static_cast<size_t>(D) * 4;                // capq, sig, rank, carry
  b += 2 * static_cast<size_t>(w) * 4;                // slot, argA
  b += 16;                                            // alignment slack
  b += static_cast<size_t>(w) * 8;                    // maxA
  b += 8;                                             // barrier
  b += static_cast<size_t>(kMainThreads) * (8 + 4 + 4);  // per-segment partials [8][32]
  b += 2 * static_cast<size_t>(w) * 4;                    // columns needing PMq, their list
  g.smem = b;
  return g;
}

struct SnapWs {
  uint32_t *zero;  // tcount[T2], tcursor[T2], nunits, ticket (zeroed per call)
  size_t zero_words;
  uint32_t *toff;
  Unit *units;
  int32_t *ord, *sp, *su;
  int32_t *sig, *rank_of, *capq;
  uint32_t *carry;  // [D][T2]
  uint32_t *kmax;   // [D][ceil(H/16)], used when the caller passes none
  int64_t max_units;
};

SnapWs carve_snap(Carve &c, int D, int H, int T2, int64_t J) {
  SnapWs w;
  w.zero_words = 2 * static_cast<size_t>(T2) + 2;  // tcount, tcursor, nunits, ticket
  w.zero = c.take<uint32_t>(w.zero_words);
  w.toff = c.take<uint32_t>(static_cast<size_t>(T2) + 1);
  w.max_units = static_cast<int64_t>(T2) + (J + kUnitCands - 1) / kUnitCands;
  w.units = c.take<Unit>(static_cast<size_t>(w.max_units) + 1);
  const size_t nj = static_cast<size_t>(J > 0 ? J : 1);
  w.ord = c.take<int32_t>(nj);
  w.sp = c.take<int32_t>(nj);
  w.su = c.take<int32_t>(nj);
  w.sig = c.take<int32_t>(static_cast<size_t>(D));
  w.rank_of = c.take<int32_t>(static_cast<size_t>(D));
  w.capq = c.take<int32_t>(static_cast<size_t>(D));
  w.carry = c.take<uint32_t>(static_cast<size_t>(T2) * D);
  w.kmax = c.take<uint32_t>(static_cast<size_t>(D) * ((static_cast<size_t>(H) + kSumBlock - 1) / kSumBlock));
  return w;
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

constexpr int kMaxH = 1 << 28;
constexpr size_t kStaticSmem = 2048;  // left to the kernels' static arrays (1 KB at most)

// Events recorded around the scoring kernel (maps_set_dispatch_events).
thread_local cudaEvent_t g_score_ev[2] = {nullptr, nullptr};

template <int W2>
int run_snapshot(int64_t grid, size_t smem, cudaStream_t s, const CUtensorMap &tmap, const SnapArgs &a) {
  MAPS_TRY(allow_smem(dispatch_snapshot_kernel<W2>, smem_beside(kStaticSmem)));
  if (g_score_ev[0]) MAPS_TRY(cuda_ok(cudaEventRecord(g_score_ev[0], s)));
  launch_pdl(dispatch_snapshot_kernel<W2>, static_cast<unsigned>(grid), kMainThreads, smem, s, tmap, a);
  MAPS_TRY(launch_ok());
  if (g_score_ev[1]) MAPS_TRY(cuda_ok(cudaEventRecord(g_score_ev[1], s)));
  return MAPS_OK;
}

int launch_snapshot(int D, int H, const int32_t *K, const uint32_t *kmax, const int32_t *cap,
                    const int32_t *Q, int64_t J, const int32_t *cp, const int32_t *cb,
                    int32_t *choice, int64_t *headroom, void *ws, cudaStream_t s) {
  const SnapGeom g = snap_geom(D, H);
  if (g.smem + 1024 > static_cast<size_t>(max_smem_optin())) return MAPS_E_INVALID;
  Carve cv(ws);
  const SnapWs w = carve_snap(cv, D, H, g.T2, J);
  if (w.max_units > 0x7fffffffLL) return MAPS_E_INVALID;
  int32_t *status = status_word(ws);
  uint32_t *tcount = w.zero, *tcursor = w.zero + g.T2;
  uint32_t *nunits = w.zero + 2 * static_cast<size_t>(g.T2);
  uint32_t *ticket = nunits + 1;  // bin_count blocks finished
  const int sms = sm_count();
  const bool check_kmax = kmax != nullptr;
  const int64_t nb = (static_cast<int64_t>(H) + kSumBlock - 1) / kSumBlock;
  const bool direct = direct_fits(D, H, J);
  if (!direct) MAPS_TRY(cuda_ok(cudaMemsetAsync(w.zero, 0, w.zero_words * 4, s)));
  if (kmax == nullptr) {
    const int gk = static_cast<int>(std::min<int64_t>((nb * D + 255) / 256, 8LL * sms));
    launch_pdl(kmax_from_K_kernel, gk, 256, 0, s, D, H, K, w.kmax, status);
    kmax = w.kmax;
  }
  if (direct) {
    const int share = direct_share(D);
    const int64_t blocks = (J * share + kDirectWarps - 1) / kDirectWarps;
    // the reading of K takes blocks of its own where the candidates have few
    const int64_t reading = static_cast<int64_t>(D) * H / (32 * kDirectWarps * 16);
    const int grid = static_cast<int>(
        std::min<int64_t>(std::max(blocks, std::min<int64_t>(reading, 2LL * sms)), 8LL * sms));
    if (g_score_ev[0]) MAPS_TRY(cuda_ok(cudaEventRecord(g_score_ev[0], s)));
    auto launch = [&](auto kern) {
      launch_pdl(kern, grid, 32 * kDirectWarps, 0, s, D, H, K, kmax, check_kmax ? 1 : 0, cap, Q, J, cp, cb,
                 choice, headroom, status, share);
    };
    if (nb % 4 == 0 && aligned(kmax, 16))
      launch(dispatch_direct_kernel<true>);
    else
      launch(dispatch_direct_kernel<false>);
    MAPS_TRY(launch_ok());
    if (g_score_ev[1]) MAPS_TRY(cuda_ok(cudaEventRecord(g_score_ev[1], s)));
    return MAPS_OK;
  }
  // carries of D decoders, and candidate counts in blocks of 256 candidates
  const int gc = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((J + 255) / 256, 4LL * sms)));
  launch_pdl(dispatch_prep_kernel, D + gc, 256, 0, s, D, D, H, g.W2, g.T2, K, check_kmax, kmax,
             w.carry, Q, cap,
             w.sig, w.rank_of, w.capq, J, cp, cb, tcount, choice, headroom, status, ticket, w.toff,
             w.units, nunits);
  const int gb = static_cast<int>(std::min<int64_t>((J + 255) / 256, 4LL * sms));
  launch_pdl(bin_scatter_kernel, gb, 256, 0, s, J, H, g.W2, g.T2, cp, cb, w.toff, tcursor, w.ord,
             w.sp, w.su);
  MAPS_TRY(launch_ok());

  CUtensorMap tmap;
  std::memset(&tmap, 0, sizeof(tmap));
  bool use_tma = (H % 4 == 0) && aligned(K, 16);
  PFN_cuTensorMapEncodeTiled_v12000 enc = use_tma ? tensor_map_encoder() : nullptr;
  if (enc == nullptr) use_tma = false;
  if (use_tma) {
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(H), static_cast<cuuint64_t>(D)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(H) * 4};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(g.W2), static_cast<cuuint32_t>(g.box_rows)};
    cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_INT32, 2, const_cast<int32_t *>(K), dims,
                           strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           g.W2 == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) use_tma = false;
  }
  SnapArgs a;
  a.D = D;
  a.H = H;
  a.W2 = g.W2;
  a.T2 = g.T2;
  a.Drows = use_tma ? g.Drows : D;
  a.boxes = g.boxes;
  a.box_rows = g.box_rows;
  a.tile_stride = g.tile_stride;
  a.comp_off = g.comp_off;
  a.region = g.region;
  a.alias = g.alias;
  a.use_tma = use_tma;
  a.K = K;
  a.sig = w.sig;
  a.rank_of = w.rank_of;
  a.capq = w.capq;
  a.carry = w.carry;
  a.units = w.units;
  a.nunits = nunits;
  a.ord = w.ord;
  a.sp = w.sp;
  a.su = w.su;
  a.choice = choice;
  a.headroom = headroom;
  a.status = status;
  const int64_t grid = std::max<int64_t>(1, w.max_units);  // units past *nunits return at once
  switch (g.W2) {
    case 16: return run_snapshot<16>(grid, g.smem, s, tmap, a);
    case 32: return run_snapshot<32>(grid, g.smem, s, tmap, a);
    case 64: return run_snapshot<64>(grid, g.smem, s, tmap, a);
    case 128: return run_snapshot<128>(grid, g.smem, s, tmap, a);
    default: return run_snapshot<256>(grid, g.smem, s, tmap, a);
  }
}

}  // namespace
}  // namespace maps

namespace maps {
namespace {
struct SeqWs {
  uint32_t *km;  // [D][ceil(H/16)]
  uint32_t *cm;  // [D][ceil(H/128)]
};
SeqWs carve_seq(Carve &c, int D, int H) {
  SeqWs w;
  w.km = c.take<uint32_t>(static_cast<size_t>(D) * ((static_cast<size_t>(H) + kSumBlock - 1) / kSumBlock));
  w.cm = c.take<uint32_t>(static_cast<size_t>(D) * ((static_cast<size_t>(H) + kSeqChunk - 1) / kSeqChunk));
  return w;
}
}  // namespace

int dispatch_sequential(int D, int H, int32_t *K, const int32_t *cap, int32_t *Q, int64_t J,
                        const int32_t *cp, const int32_t *cb, int32_t *choice, int64_t *headroom,
                        bool mc, void *ws, cudaStream_t s) {
  // a private summary of K (also validating K >= 0); updated in place
  int32_t *status = status_word(ws);
  Carve cv(ws);
  const SeqWs w = carve_seq(cv, D, H);
  const int64_t chunks = (static_cast<int64_t>(H) + kSeqChunk - 1) / kSeqChunk;
  const int gk = static_cast<int>(std::min<int64_t>((8 * chunks * D + 255) / 256, 8LL * sm_count()));
  launch_pdl(seq_summary_kernel, gk, 256, 0, s, D, H, K, w.km, w.cm, status);
  SeqArgs a;
  a.D = D;
  a.H = H;
  a.mc = mc ? 1 : 0;
  a.K = K;
  a.km = w.km;
  a.cm = w.cm;
  a.cap = cap;
  a.Q = Q;
  a.J = J;
  a.cp = cp;
  a.cb = cb;
  a.choice = choice;
  a.headroom = headroom;
  a.status = status;
  a.kb = 0;
  while ((1 << a.kb) < D) ++a.kb;
  a.ncol = std::min((D + 7) / 8, kColWarps);
  // shared memory per row: a thirty-second for chunk maxima, the rest resident
  // steps (1 + 1/4 + 1/16 words each)
  const int64_t fixed = kSeqWords * seq_dw(D) + kSeqPad;
  const size_t limit = smem_beside(kStaticSmem);
  const int64_t words = (static_cast<int64_t>(limit) / 4 - fixed) / D;
  // One or two candidates are not worth the rows' way to shared memory and back.  24
  // decoders, H 4,800, candidates of a few hundred steps, without it and with: one
  // 7.9 against 10.7 us, two 8.8 against 12.8; of three it pays.
  const bool few = J <= 2;
  a.P2 = few ? 0 : static_cast<int>(std::min<int64_t>(chunks, words / 32));
  a.P0 = 0;
  while (!few && a.P0 < chunks * kSeqChunk && seq_row_words(a.P0 + kSeqChunk, a.P2) <= words) a.P0 += kSeqChunk;
  const size_t smem = 4 * (static_cast<size_t>(D) * seq_row_words(a.P0, a.P2) + fixed);
  auto launch = [&](void (*kern)(SeqArgs)) {
    MAPS_TRY(allow_smem(kern, limit));
    launch_pdl(kern, 1, 1024, smem, s, a);
    return launch_ok();
  };
  return D <= 32   ? launch(dispatch_sequential_kernel<1>)
         : D <= 64 ? launch(dispatch_sequential_kernel<2>)
                   : launch(dispatch_sequential_kernel<0>);
}
}  // namespace maps

extern "C" {

int maps_set_dispatch_events(void *before, void *after) {
  maps::g_score_ev[0] = static_cast<cudaEvent_t>(before);
  maps::g_score_ev[1] = static_cast<cudaEvent_t>(after);
  return MAPS_OK;
}

size_t maps_dispatch_workspace_size(int32_t mode, int32_t D, int32_t H, int64_t J) {
  using namespace maps;
  Carve c(nullptr);
  if (mode == MAPS_MODE_SNAPSHOT && D >= 1 && H >= 1 && H <= kMaxH) {
    const SnapGeom g = snap_geom(D, H);
    carve_snap(c, D, H, g.T2, J);
  } else if (mode == MAPS_MODE_SEQUENTIAL && D >= 1 && H >= 1 && H <= kMaxH) {
    carve_seq(c, D, H);
  } else if ((mode == MAPS_MODE_ALG1_SNAPSHOT || mode == MAPS_MODE_ALG1_SEQUENTIAL) && D >= 1) {
    c.take<long long>(static_cast<size_t>(D));
  }
  return c.bytes();
}

int maps_dispatch(int32_t mode, int32_t D, int32_t H, int32_t S, int32_t *K, const uint32_t *kmax,
                  const int32_t *cap, int32_t *Q, const int64_t *res_off, int64_t R, const int32_t *prompt,
                  const int32_t *gen, const int32_t *bound, int64_t J, const int32_t *cand_prompt,
                  const int32_t *cand_bound, int32_t *choice_out, int64_t *headroom_out, void *ws,
                  size_t ws_bytes, void *stream) {
  using namespace maps;
  if (mode < MAPS_MODE_SNAPSHOT || mode > MAPS_MODE_ALG1_SEQUENTIAL) return MAPS_E_INVALID;
  if (D < 1 || D > kMaxD || J < 0 || J > 0x7fffffffLL || cap == nullptr || Q == nullptr)
    return MAPS_E_INVALID;
  if (J > 0 && (cand_prompt == nullptr || cand_bound == nullptr || choice_out == nullptr))
    return MAPS_E_INVALID;
  const bool horizon = mode == MAPS_MODE_SNAPSHOT || mode == MAPS_MODE_SEQUENTIAL;
  if (horizon && (H < 1 || H > kMaxH || K == nullptr)) return MAPS_E_INVALID;
  if (!horizon && (S < 1 || res_off == nullptr || R < 0 ||
                   (R > 0 && (prompt == nullptr || gen == nullptr || bound == nullptr))))
    return MAPS_E_INVALID;
  MAPS_TRY(check_ws(ws, ws_bytes, maps_dispatch_workspace_size(mode, D, H, J)));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int32_t *status = status_word(ws);
  if (J == 0) return MAPS_OK;
  switch (mode) {
    case MAPS_MODE_SNAPSHOT:
      return launch_snapshot(D, H, K, kmax, cap, Q, J, cand_prompt, cand_bound, choice_out,
                             headroom_out, ws, s);
    case MAPS_MODE_SEQUENTIAL:
      return dispatch_sequential(D, H, K, cap, Q, J, cand_prompt, cand_bound, choice_out,
                                 headroom_out, false, ws, s);
    default: {
      Carve cv(ws);
      long long *B_eff = cv.take<long long>(static_cast<size_t>(D));
      launch_pdl(alg1_budget_kernel, D, 256, 0, s, D, S, res_off, R, prompt, gen, bound, cap, B_eff, status);
      if (mode == MAPS_MODE_ALG1_SNAPSHOT) {
        const int grid = static_cast<int>(std::min<int64_t>((J + 255) / 256, 4LL * sm_count()));
        launch_pdl(alg1_snapshot_kernel, grid, 256, 0, s, D, S, B_eff, cap, Q, J, cand_prompt, cand_bound,
                                                  choice_out, headroom_out, status);
      } else if (J <= kFewCands && D > kFewD) {
        launch_pdl(alg1_few_kernel, 1, (D + 31) / 32 * 32, 0, s, D, S, B_eff, cap, Q, J, cand_prompt,
                   cand_bound, choice_out, headroom_out, status);
      } else {
        launch_pdl(alg1_sequential_for(D), 1, 32, 0, s, D, S, B_eff, cap, Q, J, cand_prompt, cand_bound,
                   choice_out, headroom_out, status);
      }
      return launch_ok();
    }
  }
}

}  // extern "C"
