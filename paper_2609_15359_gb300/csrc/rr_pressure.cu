// rr_pressure.cu -- the round-robin KV-pressure simulation of App. A and its
// high-pressure (HP) interval metrics, for many workload realisations at once.
//
// Model (App. A): requests arrive in order; round robin sends request i to
// decoder i mod N (App. A, routing equation); a request holds
// M = L_p + L_out KV tokens while admitted (Eq. kv_demand); a decoder admits
// the head of its FIFO queue while K + M(head) <= C (Eq. admission); service
// is processor sharing at one token per t_tok, taken at token granularity: a
// round gives each of the n admitted requests one token and lasts n * t_tok,
// completions and admissions happen at round boundaries (completions first),
// and an idle decoder admits a request when it arrives.  A decoder is under
// high pressure while K * 1e6 >= theta_ppm * C (Definition of the HP
// interval).  All times are integer microseconds.
//
// Under round robin the decoders never interact, so every (realisation,
// decoder) stream is simulated by one warp on its own.  The warp does not
// step round by round: between two events every admitted request gains the
// same number of tokens, so it jumps straight to the next one -- the first
// completion (the smallest finishing round among the admitted requests), or,
// when the queue is empty, the round boundary at or after the next arrival.
// A second, small kernel turns each realisation's last completion into its
// simulated span T_sim.
//
// A stream is one chain of about two events a request, so the cost is the
// instructions of an event (five to six cycles each for a lone warp).  The
// admitted requests (stream position, finishing round, footprint) sit in the
// warp's registers, two or eight a lane in any slot, free where the finishing
// round is ~0: the next completion is one 32-bit warp minimum, a completion clears
// its slots and an admission fills the first free one.  The head of the queue
// is held in every lane, the next 64 requests one per lane; the waiting
// statistics are gathered at the admissions.  Every load is a window ahead of
// its use, the round boundary comes from a multiplication by the reciprocal of
// a round and a remainder, tokens and loop counts are 32-bit.  64 draws x 6
// utilisations of 10,000 requests on 4 decoders (1,536 streams): 4.10 -> 1.70
// ms (1.91 with a division an event, waits for the windows' loads and 64-bit
// counts); before, the set sat in shared memory and was compacted at every
// completion, with 64-bit shuffle reductions and a 64-bit division an event, and
// the waiting statistics took a second pass with a binary search a request.
// (Four slots a lane for every stream, 64-bit positions: 2.16 ms.  The free
// lanes kept as a mask, the next head shuffled ahead of its use, or a lone
// completion's footprint by shuffle instead of the sum: 0 to 5% slower each.)
// A stream that comes to run more than 64 (then 256) requests at once starts
// over on the next variant, the last one with its running set in shared memory.
#include "maps_internal.cuh"

namespace maps {
namespace {

constexpr int kRRWarps = 2;      // streams per CTA
constexpr int kRunCap = 1536;    // requests one decoder may run at once
constexpr int kStats = 6;        // T_hp, B_hp, C_hp, completed, longest queue, total wait

struct RRStream {
  int32_t pos[kRunCap];  // stream position of each admitted request
  int32_t fin[kRunCap];  // the round at whose end it completes
  int32_t m[kRunCap];    // its footprint
};

__device__ __forceinline__ int64_t warp_min64(int64_t v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const int64_t y = __shfl_xor_sync(0xffffffffu, v, off);
    v = y < v ? y : v;
  }
  return v;
}
__device__ __forceinline__ int64_t warp_sum64(int64_t v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// One stream's simulation: its inputs, and the results of a run.
struct RRSim {
  // request s of the stream is index d + s N of its realisation
  const int64_t *A;
  const int32_t *P, *O;
  int64_t *adm, *dn;
  int64_t n_d, C, tok, K_hp;  // K >= K_hp: high pressure
  int d, N;
  // results
  int64_t T_hp, B_hp, C_hp, completed, t_last, wait, qmax;
  bool fail;

  // high-pressure state after every change at t
  __device__ __forceinline__ void pressure(bool now, int64_t t, bool &in_hp, int64_t &t_s) {
    if (now && !in_hp) {
      in_hp = true;
      t_s = t;
    } else if (!now && in_hp) {
      in_hp = false;
      const int64_t len = t - t_s;
      T_hp += len;
      B_hp = len > B_hp ? len : B_hp;
      C_hp += 1;
    }
  }
  template <int kSlots>
  __device__ bool run_registers();
  __device__ void run_general(RRStream &rs);
};

// The running set in registers, kSlots requests a lane; false when it does not
// fit (start over).  Stream positions fit 31 bits here.
template <int kSlots>
__device__ bool RRSim::run_registers() {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int64_t kNever = INT64_MAX;
  const int lane = threadIdx.x & 31;
  uint32_t fin[kSlots];
  int32_t m[kSlots], pos[kSlots];
#pragma unroll
  for (int i = 0; i < kSlots; ++i) {
    fin[i] = ~0u;
    m[i] = pos[i] = 0;
  }
  // lane l: requests wb + l and wb + 32 + l (the second in flight); past the
  // last one the arrival is kNever, so it is neither admitted nor waited for
  const int n = static_cast<int>(n_d);
  const int32_t tok_us = static_cast<int32_t>(tok), stride = 8 * N;
  const uint32_t cap = static_cast<uint32_t>(C), hp = static_cast<uint32_t>(K_hp);
  const int64_t *const Ad = A + d;
  int64_t wa = kNever, na = kNever;
  int32_t wp = 0, wo = 0, np = 0, no = 0;
  auto load = [&](int s, int64_t &a, int32_t &p, int32_t &o) {
    a = kNever;
    if (s < n) {
      const int64_t i = static_cast<int64_t>(s) * N;
      a = Ad[i];
      o = O[d + i];
      p = P[d + i];
    }
  };
  int wi = 0;  // the head's lane
  load(lane, wa, wp, wo);
  load(32 + lane, na, np, no);
  // arrivals counted for the longest queue: those before index ab all arrived
  // before the last admission; lane l holds arrivals ab + l and ab + 32 + l
  auto arrival = [&](int s) { return s < n ? Ad[static_cast<int64_t>(s) * N] : kNever; };
  int ab = 0;
  int64_t aa = arrival(lane), ab2 = arrival(32 + lane);
  int64_t t = n > 0 ? Ad[0] : 0, t_s = 0;
  char *adm_h = reinterpret_cast<char *>(adm + d);  // the head's admission time
  char *const dn_d = reinterpret_cast<char *>(dn + d);
  uint32_t R = 0, K = 0;
  uint32_t f = ~0u;  // the smallest finishing round
  int qh = 0, n_run = 0, qm = 0;
  bool in_hp = false;
  int64_t ha = __shfl_sync(kAll, wa, 0);
  int32_t ho = __shfl_sync(kAll, wo, 0);
  uint32_t hm = static_cast<uint32_t>(__shfl_sync(kAll, wp, 0) + ho);
  // 1 / (lane + 1) steps of one token, for running sets up to 32
  const float inv = 1.0f / (static_cast<float>(lane + 1) * static_cast<float>(tok_us));
  // every iteration admits, completes, or reaches an arrival's round boundary
  for (uint32_t left = 4u * static_cast<uint32_t>(n) + 16u; left > 0; --left) {
    // admissions at t: the FIFO head while it has arrived and fits (K and a
    // footprint are at most C < 2^31)
    while (ha <= t && K + hm <= cap) {
      if (R > 0x7fffffffu - static_cast<uint32_t>(ho)) {
        fail = true;
        return true;
      }
      const uint32_t fh = R + static_cast<uint32_t>(ho);
      bool placed = false;
#pragma unroll
      for (int i = 0; i < kSlots; ++i) {
        if (placed) continue;
        const unsigned free_lanes = __ballot_sync(kAll, fin[i] == ~0u);
        if (free_lanes == 0) continue;
        placed = true;
        const bool me = lane == __ffs(free_lanes) - 1;
        fin[i] = me ? fh : fin[i];
        m[i] = me ? static_cast<int32_t>(hm) : m[i];
        pos[i] = me ? qh : pos[i];
      }
      if (!placed) return false;
      f = min(f, fh);
      if (lane == 0) *reinterpret_cast<int64_t *>(adm_h) = t;
      adm_h += stride;
      // the requests that arrived before t and are not admitted before this one
      wait += t - ha;
      unsigned before;
      while ((before = __ballot_sync(kAll, aa < t)) == kAll) {
        ab += 32;
        aa = ab2;
        ab2 = arrival(ab + 32 + lane);
      }
      qm = max(qm, ab + __popc(before) - qh);
      ++n_run;
      K += hm;
      ++qh;
      if (++wi == 32) {
        wi = 0;
        wa = na, wp = np, wo = no;
        load(qh + 32 + lane, na, np, no);
      }
      ha = __shfl_sync(kAll, wa, wi);
      ho = __shfl_sync(kAll, wo, wi);
      hm = static_cast<uint32_t>(__shfl_sync(kAll, wp, wi) + ho);
    }
    if ((K >= hp) != in_hp) pressure(!in_hp, t, in_hp, t_s);
    if (n_run == 0) {
      if (qh >= n) break;
      t = ha;  // idle until the head arrives (it fits an empty decoder)
      continue;
    }
    // next event: the first completion, or the boundary where the head arrives
    const int64_t step = static_cast<int64_t>(n_run) * tok_us;
    const int64_t tc = static_cast<int64_t>(f - R) * step, gap = ha - t;
    if (gap > 0 && gap < tc) {
      // rounds to the boundary, ceil(gap / step), at most f - R
      uint32_t k;
      if (((gap | step) >> 31) == 0) {
        const uint32_t g = static_cast<uint32_t>(gap), st = static_cast<uint32_t>(step);
        const float e = static_cast<float>(g) * __shfl_sync(kAll, inv, n_run - 1);
        if (n_run <= 32 && e < 1e6f) {
          // within one of the quotient: the factors' relative errors add up to
          // less than 2^-21
          k = static_cast<uint32_t>(e);
          const int32_t rest = static_cast<int32_t>(g - k * st);
          k += (rest > 0 ? 1 : 0) + (rest > static_cast<int32_t>(st) ? 1 : 0) -
               (rest <= -static_cast<int32_t>(st) ? 1 : 0);
        } else {
          k = (g + st - 1u) / st;
        }
      } else {
        k = static_cast<uint32_t>((gap + step - 1) / step);
      }
      t += k * step;
      R += k;
    } else {
      t += tc;
      R = f;
    }
    if (R == f) {  // completions
      uint32_t freed = 0, gone = 0;
      f = ~0u;
#pragma unroll
      for (int i = 0; i < kSlots; ++i) {
        const bool now = fin[i] == R;
        if (now) *reinterpret_cast<int64_t *>(dn_d + static_cast<int64_t>(pos[i]) * stride) = t;
        freed += now ? static_cast<uint32_t>(m[i]) : 0u;
        gone += now ? 1u : 0u;
        fin[i] = now ? ~0u : fin[i];
        f = min(f, fin[i]);
      }
      f = __reduce_min_sync(kAll, f);
      K -= __reduce_add_sync(kAll, freed);
      n_run -= static_cast<int>(__reduce_add_sync(kAll, gone));
      t_last = t;
    }
  }
  completed = qh - n_run;
  qmax = qm;
  if (n_run != 0 || qh < n) fail = true;
  return true;
}

// The running set in shared memory, at most kRunCap requests.
__device__ void RRSim::run_general(RRStream &rs) {
  const int lane = threadIdx.x & 31;
  // window of the next 32 requests, lane j = stream position wb + j
  int64_t wb = 0, wa = 0;
  int32_t wm = 0, wo = 0;
  auto load_window = [&](int64_t base) {
    wb = base;
    const int64_t s = base + lane;
    if (s < n_d) {
      const int64_t i = d + s * N;
      wa = A[i];
      wo = O[i];
      wm = P[i] + wo;
    }
  };
  load_window(0);

  int64_t t = n_d > 0 ? A[d] : 0, R = 0, K = 0, qh = 0;
  int n_run = 0;
  bool in_hp = false;
  int64_t t_s = 0;
  // every iteration admits, completes, or reaches an arrival's round boundary
  const int64_t max_iter = 4 * n_d + 16;
  for (int64_t iter = 0; iter < max_iter; ++iter) {
    // admissions at t: the FIFO head while it has arrived and fits
    int64_t ha = 0;
    for (;;) {
      if (qh >= n_d) break;
      if (qh - wb >= 32) load_window(qh);
      const int src = static_cast<int>(qh - wb);
      ha = __shfl_sync(0xffffffffu, wa, src);
      const int32_t hm = __shfl_sync(0xffffffffu, wm, src);
      const int32_t ho = __shfl_sync(0xffffffffu, wo, src);
      if (ha > t || K + hm > C) break;
      if (n_run >= kRunCap || R + ho > 0x7fffffffLL) {
        fail = true;
        break;
      }
      if (lane == 0) {
        rs.pos[n_run] = static_cast<int32_t>(qh);
        rs.fin[n_run] = static_cast<int32_t>(R + ho);
        rs.m[n_run] = hm;
        adm[d + qh * N] = t;
      }
      ++n_run;
      K += hm;
      ++qh;
    }
    if (fail) break;
    pressure(K >= K_hp, t, in_hp, t_s);
    if (n_run == 0) {
      if (qh >= n_d) break;
      t = ha;  // idle until the head arrives (it fits an empty decoder)
      continue;
    }
    __syncwarp();
    // next event: the first completion, or the boundary where the head arrives
    int64_t f = 0x7fffffffffffffffLL;
    for (int j = lane; j < n_run; j += 32) f = rs.fin[j] < f ? rs.fin[j] : f;
    const int64_t f_min = warp_min64(f);
    int64_t k = f_min - R;
    const int64_t step = static_cast<int64_t>(n_run) * tok;
    if (qh < n_d && ha > t) {
      const int64_t ka = (ha - t + step - 1) / step;
      k = ka < k ? ka : k;
    }
    t += k * step;
    R += k;
    if (R == f_min) {
      // completions: record them and compact the rest in place (a chunk is
      // read whole before it is written, and writes never pass the reads)
      int wpos = 0, gone = 0;
      int64_t freed = 0;
      for (int base = 0; base < n_run; base += 32) {
        const int j = base + lane;
        const bool live = j < n_run;
        const int32_t pj = live ? rs.pos[j] : 0, fj = live ? rs.fin[j] : 0, mj = live ? rs.m[j] : 0;
        const bool fin_now = live && fj == R;
        if (fin_now) {
          dn[d + static_cast<int64_t>(pj) * N] = t;
          freed += mj;
        }
        const unsigned keep = __ballot_sync(0xffffffffu, live && !fin_now);
        __syncwarp();
        if (live && !fin_now) {
          const int to = wpos + __popc(keep & ((1u << lane) - 1u));
          rs.pos[to] = pj;
          rs.fin[to] = fj;
          rs.m[to] = mj;
        }
        __syncwarp();
        wpos += __popc(keep);
        gone += __popc(__ballot_sync(0xffffffffu, fin_now));
      }
      n_run = wpos;
      K -= warp_sum64(freed);
      completed += gone;
      t_last = t;
    }
  }
  if (n_run != 0 || qh < n_d) fail = true;  // no progress
  __syncwarp();

  // waiting statistics from the admission times (non-decreasing along the
  // stream: FIFO): the total wait, and at each arrival the requests that had
  // arrived and were not yet admitted
  wait = qmax = 0;
  for (int64_t s = lane; s < n_d; s += 32) {
    const int64_t i = d + s * N;
    const int64_t ai = A[i];
    wait += adm[i] - ai;
    // first position j <= s with admit_j > a_i
    int64_t lo = 0, hi = s + 1;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (adm[d + mid * N] > ai)
        hi = mid;
      else
        lo = mid + 1;
    }
    const int64_t q = s + 1 - lo;
    qmax = q > qmax ? q : qmax;
  }
  wait = warp_sum64(wait);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const int64_t y = __shfl_xor_sync(0xffffffffu, qmax, off);
    qmax = y > qmax ? y : qmax;
  }
}

__global__ void __launch_bounds__(32 * kRRWarps)
rr_stream_kernel(int64_t n_real, int64_t n, int N, int64_t C, int64_t tok, uint32_t theta_ppm,
                 const int64_t *__restrict__ arrival, const int32_t *__restrict__ prompt,
                 const int32_t *__restrict__ out_len, int64_t *__restrict__ admit,
                 int64_t *__restrict__ done, int64_t *__restrict__ stats,
                 int64_t *__restrict__ last_done, int32_t *status) {
  pdl_prologue();
  __shared__ RRStream sm[kRRWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t stream = static_cast<int64_t>(blockIdx.x) * kRRWarps + warp;
  if (stream >= n_real * N) return;
  const int64_t r = stream / N;
  const int d = static_cast<int>(stream - r * N);
  const int64_t *A = arrival + r * n;
  const int32_t *P = prompt + r * n, *O = out_len + r * n;
  int64_t *adm = admit + r * n, *dn = done + r * n;
  int64_t *st = stats + stream * kStats;
  const int64_t n_d = d < n ? (n - 1 - d) / N + 1 : 0;  // requests d, d + N, ...

  // the stream's requests in the domain (a footprint above C would block its
  // queue for ever), and arrival in order
  bool bad = false;
  int64_t foot = 0;
#pragma unroll 4
  for (int64_t s = lane; s < n_d; s += 32) {
    const int64_t i = d + s * N;
    const int32_t p = P[i], o = O[i];
    if (p < 0 || o < 1 || static_cast<int64_t>(p) + o > C || A[i] < 0 || (i > 0 && A[i] < A[i - 1]))
      bad = true;
    foot += static_cast<int64_t>(p) + o;
  }
  foot = warp_sum64(foot);
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) {
      flag_error(status, MAPS_E_RANGE);
      for (int q = 0; q < kStats; ++q) st[q] = 0;
      last_done[stream] = 0;
    }
    return;
  }

  RRSim sim;
  sim.A = A, sim.P = P, sim.O = O, sim.adm = adm, sim.dn = dn;
  sim.n_d = n_d, sim.C = C, sim.tok = tok, sim.d = d, sim.N = N;
  // K * 10^6 >= theta_ppm * C
  sim.K_hp = (static_cast<int64_t>(theta_ppm) * C + 999999) / 1000000;
  auto clear = [&] {
    sim.T_hp = sim.B_hp = sim.C_hp = sim.completed = sim.t_last = sim.wait = sim.qmax = 0;
    sim.fail = false;
  };
  clear();
  // the variant by the footprints a capacity holds on average, with room for
  // the spread; a set that turns out larger moves on to the next.  192
  // realisations of 10,000 requests, two a lane against eight a lane against shared
  // memory: at the usual loads, capacities of 24 footprints 1.51, 1.71 and 3.81 ms,
  // of 64 1.55, 1.76 and 3.93, of 90 (two a lane starts over) 3.19, 1.77 and 3.96,
  // of 200 3.23, 1.81 and 4.04.  Overloaded, when the set fills the capacity: 43
  // 1.00, 1.17 and 2.54, 56 1.01, 1.18 and 2.70, 64 (starting over) 1.24, 1.19 and
  // 2.70, 220 eight a lane 1.31 against 3.15, 250 (starting over) 3.09 against 3.22.
  // So the sets of this workload stay within a variant's room to some 0.9 of it;
  // the lines leave a third and a fifth for footprints that spread more.
  const int64_t about = C * n_d / (foot > 0 ? foot : 1);
  const bool small = n_d <= 0x3ffffff0 && N < (1 << 28);  // what their 32-bit counts hold
  bool ran = small && about <= 44 && sim.run_registers<2>();
  if (!ran && small && about <= 200) {
    clear();
    ran = sim.run_registers<8>();
  }
  if (!ran) {
    clear();
    sim.run_general(sm[warp]);
  }
  if (lane == 0) {
    if (sim.fail) flag_error(status, MAPS_E_RANGE);  // capacity of the running set, or no progress
    st[0] = sim.T_hp;
    st[1] = sim.B_hp;
    st[2] = sim.C_hp;
    st[3] = sim.completed;
    st[4] = sim.qmax;
    st[5] = sim.wait;
    last_done[stream] = sim.t_last;
  }
}

// T_sim of every realisation: its last completion minus its first arrival.
__global__ void __launch_bounds__(256)
rr_span_kernel(int64_t n_real, int64_t n, int N, const int64_t *__restrict__ arrival,
               const int64_t *__restrict__ last_done, int64_t *__restrict__ t_sim) {
  pdl_prologue();
  const int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= n_real) return;
  int64_t m = 0;
  for (int d = 0; d < N; ++d) m = last_done[r * N + d] > m ? last_done[r * N + d] : m;
  t_sim[r] = m - arrival[r * n];
}

}  // namespace
}  // namespace maps

extern "C" {

size_t maps_rr_pressure_workspace_size(const maps_rr_cfg *cfg, int64_t n_real) {
  using namespace maps;
  Carve c(nullptr);
  if (cfg != nullptr && n_real > 0 && cfg->N > 0) c.take<int64_t>(static_cast<size_t>(n_real) * cfg->N);
  return c.bytes();
}

int maps_rr_pressure(const maps_rr_cfg *cfg, int64_t n_real, const int64_t *arrival_us,
                     const int32_t *prompt, const int32_t *out_len, int64_t *admit_us,
                     int64_t *done_us, int64_t *stats_out, int64_t *t_sim_out, void *ws,
                     size_t ws_bytes, void *stream) {
  using namespace maps;
  if (cfg == nullptr || n_real < 1 || cfg->n_req < 1 || cfg->N < 1 || cfg->C < 1 ||
      cfg->t_tok_us < 1 || cfg->theta_ppm == 0 || cfg->theta_ppm > 1000000u)
    return MAPS_E_INVALID;
  if (n_real > (int64_t(1) << 40) / cfg->n_req || n_real * cfg->N > 0x7fffffffLL * kRRWarps)
    return MAPS_E_INVALID;
  if (arrival_us == nullptr || prompt == nullptr || out_len == nullptr || admit_us == nullptr ||
      done_us == nullptr || stats_out == nullptr || t_sim_out == nullptr)
    return MAPS_E_INVALID;
  MAPS_TRY(check_ws(ws, ws_bytes, maps_rr_pressure_workspace_size(cfg, n_real)));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int32_t *status = status_word(ws);
  Carve c(ws);
  int64_t *last = c.take<int64_t>(static_cast<size_t>(n_real) * cfg->N);
  const int64_t streams = n_real * cfg->N;
  launch_pdl(rr_stream_kernel, static_cast<unsigned>((streams + kRRWarps - 1) / kRRWarps),
             32 * kRRWarps, 0, s, n_real, cfg->n_req, cfg->N, static_cast<int64_t>(cfg->C),
             static_cast<int64_t>(cfg->t_tok_us), cfg->theta_ppm, arrival_us, prompt, out_len,
             admit_us, done_us, stats_out, last, status);
  launch_pdl(rr_span_kernel, static_cast<unsigned>((n_real + 255) / 256), 256, 0, s, n_real,
             cfg->n_req, cfg->N, arrival_us, last, t_sim_out);
  return launch_ok();
}

}  // extern "C"
