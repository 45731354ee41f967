// stream.cu -- the streaming scheduler loop (Sec. 3.2 sliding calibration
// window, Sec. 3.3 dispatch and local order, Algorithm 1's round-robin
// fallback, App. A Eq. admission) with all state resident on the device.
//
// Per batch of arrivals, in the paper's order:
//   1. advance every running request by the steps since the last batch; a
//      request completes on reaching its true length      (stream_advance)
//   2. completions enter the calibration window in (completion step, id)
//      order: maps_order_local sorts them, stream_window writes the ring
//   3. calibrate on the window and bound every request in the system and the
//      batch (maps_calibrate); an unbounded quantile sends the batch round
//      robin                                                (stream_rr)
//   4. group running and waiting requests by decoder      (stream_csr)
//   5. dispatch the batch SEQUENTIALly with Q = the waiting counts: a walk
//      over each decoder's sorted end steps in shared memory (stream_dispatch),
//      or, where those lists do not fit, maps_project_occupancy and
//      maps_dispatch
//   6. the batch joins its decoders' waiting queues        (stream_enqueue)
//   7. local order of every waiting queue (stream_waitlist, maps_order_local)
//   8. admission in queue order while used + p + U <= capacity, the first
//      misfit blocking its queue                            (stream_admit)
// Policy variants replace step 5 (max-headroom, round-robin or least-requests
// dispatch: stream_dispatch with mc, stream_rr, stream_lr), the order of step 7
// (FCFS: every entry promoted, so arrival order alone) and what a running
// request counts for in step 8 (occupancy, staged or held reservation).
// Fidelity modes: per-step admission with preemption replaces step 1 by a
// step-by-step simulation of each decoder (stream_interval); deferral splits
// the arrived requests at each dispatch step into those with a bound, those
// timed out to round robin and those that keep waiting (stream_select).
// Batches that fit one block run inside one kernel, up to 256 a launch
// (stream_loop_kernel).  The others are launched step by step by the host, which
// reads the 56 bytes of loop state once a batch (the request, completion and waiting
// counts, and the deferral's list lengths, that size the calls).
#include <algorithm>
#include <climits>

#include "maps_internal.cuh"

namespace maps {
namespace {

constexpr int kSt = 1024;  // threads of the one-block kernels
constexpr int kStWarps = kSt / 32;
constexpr int kStreamMaxD = 1024;
enum : uint8_t { kNotYet = 0, kWaiting = 1, kRunning = 2, kDone = 3 };

struct StreamState {
  long long prev_s;  // dispatch step of the previous batch
  int32_t nact;      // requests in the system (waiting or running)
  int32_t ndone;     // completions found by the last advance
  int32_t nwait;     // waiting requests after the last advance
  int32_t npend;     // deferral: arrived requests not yet dispatched
  int32_t nc;        // deferral: requests for the dispatch policy at this step
  int32_t nto;       // deferral: requests timed out to round robin at this step
  int32_t adm_i;     // per-step mode: admissions between the dispatch steps
  int32_t lists;     // the last dispatch: 1 walked sorted lists of up to 32 decoders, 2 left that to the host
  long long next_b;      // the one-block loop: the batch it stopped before
  long long total_done;  // completions by then
};

// Exclusive position of a 0/1 flag across the block (kSt threads) and the
// block's total.  Every thread must call it.
__device__ __forceinline__ int block_flag_scan(bool f, int *s_w, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(0xffffffffu, f);
  if (lane == 0) s_w[warp] = __popc(m);
  __syncthreads();
  int base = 0, tot = 0;
#pragma unroll 8
  for (int w = 0; w < kStWarps; ++w) {
    const int c = s_w[w];
    base += w < warp ? c : 0;
    tot += c;
  }
  __syncthreads();
  total = tot;
  return base + __popc(m & ((1u << lane) - 1u));
}

__global__ void stream_validate_kernel(int64_t N, const int64_t *arrival, const int32_t *prompt,
                                       const int32_t *true_len, const int32_t *pred,
                                       const int32_t *pred_delay, int32_t *status) {
  pdl_prologue();
  bool bad = false;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < N; i += stride)
    if (prompt[i] < 0 || true_len[i] < 1 || pred[i] < 0 || (i > 0 && arrival[i] < arrival[i - 1]) ||
        (pred_delay != nullptr && pred_delay[i] < 0))
      bad = true;
  if (bad) flag_error(status, MAPS_E_RANGE);
}

__global__ void stream_init_kernel(int64_t first_hi, int D, int32_t cap, const int64_t *arrival,
                                   int32_t *capv, StreamState *S) {
  pdl_prologue();
  for (int k = threadIdx.x; k < D; k += blockDim.x) capv[k] = cap;
  if (threadIdx.x == 0) {
    S->prev_s = arrival[first_hi - 1];
    S->nact = 0;
    S->ndone = 0;
    S->nwait = 0;
    S->npend = 0;
    S->nc = 0;
    S->nto = 0;
    S->adm_i = 0;
    S->lists = 0;
    S->next_b = 0;
    S->total_done = 0;
  }
}

// 1. Advance by delta = s - prev_s steps; keep the survivors in id order.
//    occupancy = p + g of the running requests (the over-capacity count);
//    used = what admission counts for them: p + g, p + max(U*, g) (staged)
//    or 2p + max(U*, g) (held), U* the bound reserved at admission.
__device__ void
advance_block(int64_t hi, int D, int32_t cap, int acct, int per_step, const int64_t *arrival,
              const int32_t *prompt, const int32_t *true_len, const int32_t *res_u,
              uint8_t *st, int32_t *g, const int32_t *dec, const int32_t *act_in,
              int32_t *act_out, int32_t *done_id, int32_t *done_rem, long long *used,
              StreamState *S, int64_t *stats_b, int64_t *dst) {
  __shared__ unsigned long long s_occ[kStreamMaxD], s_used[kStreamMaxD];
  __shared__ int s_w[kStWarps];
  __shared__ int s_nwait;
  const int tid = threadIdx.x;
  for (int k = tid; k < D; k += kSt) s_occ[k] = s_used[k] = 0;
  if (tid == 0) s_nwait = 0;
  const long long s = arrival[hi - 1];
  const long long delta = s - S->prev_s;  // 0 after the per-step interval
  const int nact = S->nact;
  // per-step mode: the interval kernel's completions come first
  int nkeep = 0, ndone = per_step ? S->ndone : 0, nwait = 0;
  __syncthreads();
  for (int c0 = 0; c0 < nact; c0 += kSt) {
    const int x = c0 + tid;
    int id = -1, rem32 = 0;
    bool done = false, gone = false;
    if (x < nact) {
      id = act_in[x];
      const uint8_t sv = st[id];
      gone = sv == kDone;  // completed in the per-step interval
      if (sv == kRunning) {
        const long long rem = static_cast<long long>(true_len[id]) - g[id];  // >= 1
        if (rem <= delta) {
          done = true;
          rem32 = static_cast<int>(rem);
          st[id] = kDone;
        } else {
          const int gn = g[id] + static_cast<int>(delta);  // < true_len
          g[id] = gn;
          const long long p = prompt[id];
          atomicAdd(&s_occ[dec[id]], static_cast<unsigned long long>(p + gn));
          if (acct != MAPS_STREAM_OCCUPANCY) {
            const long long out = max(static_cast<long long>(res_u[id]), static_cast<long long>(gn));
            atomicAdd(&s_used[dec[id]], static_cast<unsigned long long>(
                                            (acct == MAPS_STREAM_HELD ? 2 * p : p) + out));
          }
        }
      } else if (sv == kWaiting) {
        ++nwait;
      }
    }
    int tk, td;
    const int pk = block_flag_scan(id >= 0 && !done && !gone, s_w, tk);
    const int pd = block_flag_scan(done, s_w, td);
    if (id >= 0 && !done && !gone) act_out[nkeep + pk] = id;
    if (done) {
      done_id[ndone + pd] = id;
      done_rem[ndone + pd] = rem32;
    }
    nkeep += tk;
    ndone += td;
  }
  if (nwait) atomicAdd(&s_nwait, nwait);
  const bool ov = tid < D && static_cast<long long>(s_occ[tid]) > cap;  // D <= kSt
  if (tid < D) {
    used[tid] = static_cast<long long>(acct == MAPS_STREAM_OCCUPANCY ? s_occ[tid] : s_used[tid]);
    if (dst != nullptr && ov) dst[4 * tid + 1] += 1;
  }
  const int over = __syncthreads_count(ov);
  if (tid == 0) {
    S->prev_s = s;
    S->nact = nkeep;
    S->ndone = ndone;
    S->nwait = s_nwait;
    stats_b[0] = ndone;
    stats_b[3] = over;
  }
}
__global__ void __launch_bounds__(kSt, 1)
stream_advance_kernel(int64_t hi, int D, int32_t cap, int acct, int per_step, const int64_t *arrival,
                      const int32_t *prompt, const int32_t *true_len, const int32_t *res_u,
                      uint8_t *st, int32_t *g, const int32_t *dec, const int32_t *act_in,
                      int32_t *act_out, int32_t *done_id, int32_t *done_rem, long long *used,
                      StreamState *S, int64_t *stats_b, int64_t *dst) {
  pdl_prologue();
  advance_block(hi, D, cap, acct, per_step, arrival, prompt, true_len, res_u, st, g, dec, act_in,
                act_out, done_id, done_rem, used, S, stats_b, dst);
}

// 1'. Per-step mode: the steps prev_s + 1 .. s, one warp per decoder
//     (decoders do not interact between dispatch steps).  Each decoder holds
//     its running requests (in rbuf, unordered; the admission order is aseq)
//     and the requests it preempted since the last dispatch step (sbuf, a
//     stack, the latest on top); its waiting queue is the order computed at
//     the last dispatch step past the requests admitted then.  A step: while
//     the running requests would pass the capacity by taking one token each,
//     the most recently admitted one (never the last) is preempted, losing
//     its tokens; each takes a token, and those reaching their true length
//     complete; then, except on the dispatch step s, the stack top or the
//     queue head is admitted while used + p + U <= capacity.  Between events
//     nothing but the growth happens: no admission can succeed (used only
//     grows and nothing is freed since the head last failed), so the warp
//     jumps to the next step with a completion or a preemption, or to s.
//     Every iteration advances the step, so the loop ends.
// A decoder's simulation between dispatch steps as one warp holds it.
struct IntervalRun {
  long long t, s;              // the current step, the dispatch step
  long long qh, qe;            // the queue: its head and end in the order
  long long seq, integ;        // next admission number; waiting steps summed
  int n, ns, npre, nadm;       // running, preempted since the last dispatch step; counts
};

// The running set in registers, kS requests a lane in any slot, from t until s
// or until an admission finds no free slot; then the set goes back to rbuf (and
// g), where the general loop takes it up.  The tokens held are one running sum,
// and the queue's head is kept, so an event reads no memory unless a request
// moves: a lane's slots, one warp minimum and the uniform arithmetic (the steps
// to a preemption are divided out only when one comes before the completion).
template <int kS>
__device__ void interval_registers(IntervalRun &v, int32_t cap, int acct, const int32_t *prompt,
                                   const int32_t *true_len, const int32_t *U, int32_t *res_u, uint8_t *st,
                                   int32_t *g, const int32_t *wid, const int32_t *wperm, long long *aseq,
                                   int32_t *rbuf, int32_t *sbuf, int32_t *done_id, int32_t *done_rem,
                                   long long s0, int *s_done) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int id[kS], gi[kS], L[kS], pr[kS], ru[kS];  // id < 0: a free slot
  long long as[kS];
  long long tok = 0;
#pragma unroll
  for (int i = 0; i < kS; ++i) {
    const int x = 32 * i + lane;
    id[i] = x < v.n ? rbuf[x] : -1;
  }
#pragma unroll
  for (int i = 0; i < kS; ++i) {
    const bool ok = id[i] >= 0;
    gi[i] = ok ? g[id[i]] : 0;
    L[i] = ok ? true_len[id[i]] : 0;
    pr[i] = ok ? prompt[id[i]] : 0;
    ru[i] = ok ? res_u[id[i]] : 0;
    as[i] = ok ? aseq[id[i]] : -1;
    tok += static_cast<long long>(pr[i]) + gi[i];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) tok += __shfl_xor_sync(kAll, tok, off);
  // the stack's top, else the queue's head (hc < 0: nobody waits)
  int hc = -1, hp = 0, hu = 0;
  auto head = [&] {
    hc = v.ns > 0 ? sbuf[v.ns - 1] : v.qh < v.qe ? wid[wperm[v.qh]] : -1;
    hp = hc >= 0 ? prompt[hc] : 0;
    hu = hc >= 0 ? U[hc] : 0;
  };
  head();
  bool full = false;
  while (v.t < v.s && !full) {
    const int n = v.n;
    long long je = LLONG_MAX;  // steps to the next completion or preemption
    if (n > 0) {
      uint32_t m = ~0u;
#pragma unroll
      for (int i = 0; i < kS; ++i) m = id[i] >= 0 ? min(m, static_cast<uint32_t>(L[i] - gi[i])) : m;
      je = __reduce_min_sync(kAll, m);
      if (n > 1 && tok + n * je > cap) je = tok + n > cap ? 1 : (cap - tok) / n + 1;
    }
    const long long te = je >= v.s - v.t ? v.s : v.t + je;
    const int quiet = static_cast<int>(te - v.t - 1);  // steps of growth alone
    if (quiet > 0) {
#pragma unroll
      for (int i = 0; i < kS; ++i) gi[i] += id[i] >= 0 ? quiet : 0;
    }
    v.integ += (v.ns + (v.qe - v.qh)) * (te - v.t - 1);
    tok += n * (te - v.t - 1);
    v.t = te;
    // preempt the latest admitted while the next tokens do not fit
    bool moved = false;
    while (v.n > 1 && tok + v.n > cap) {
      long long best = -1;
      int bi = 0;
#pragma unroll
      for (int i = 0; i < kS; ++i)
        if (id[i] >= 0 && as[i] > best) {
          best = as[i];
          bi = 32 * i + lane;
        }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const long long ob = __shfl_xor_sync(kAll, best, off);
        const int oi = __shfl_xor_sync(kAll, bi, off);
        if (ob > best) {
          best = ob;
          bi = oi;
        }
      }
      int held = 0;  // the victim's tokens, from its lane
#pragma unroll
      for (int i = 0; i < kS; ++i)
        if (bi == 32 * i + lane) {
          held = pr[i] + gi[i];
          sbuf[v.ns] = id[i];
          st[id[i]] = kWaiting;
          g[id[i]] = 0;
          id[i] = -1;
        }
      tok -= __shfl_sync(kAll, held, bi & 31);
      v.n -= 1;
      v.ns += 1;
      v.npre += 1;
      moved = true;
      __syncwarp();
    }
    // one token each; completions free their slots
    tok += v.n;
    int gone = 0;
    long long freed = 0;
#pragma unroll
    for (int i = 0; i < kS; ++i) {
      const bool run = id[i] >= 0;
      gi[i] += run ? 1 : 0;
      const bool fin = run && gi[i] == L[i];
      const unsigned fm = __ballot_sync(kAll, fin);
      if (fm == 0) continue;
      gone += __popc(fm);
      if (fin) {
        st[id[i]] = kDone;
        const int o = atomicAdd(s_done, 1);
        done_id[o] = id[i];
        done_rem[o] = static_cast<int>(v.t - s0);
        freed += static_cast<long long>(pr[i]) + gi[i];
        id[i] = -1;
      }
    }
    if (gone > 0) {
      v.n -= gone;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) freed += __shfl_xor_sync(kAll, freed, off);
      tok -= freed;
    }
    if (v.t == v.s) break;
    if (moved) head();
    // admission in queue order (the stack first)
    if (hc >= 0) {
      long long used = tok;
      if (acct != MAPS_STREAM_OCCUPANCY) {
        used = 0;
#pragma unroll
        for (int i = 0; i < kS; ++i)
          if (id[i] >= 0)
            used += (acct == MAPS_STREAM_STAGED ? 1ll : 2ll) * pr[i] + max(ru[i], gi[i]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) used += __shfl_xor_sync(kAll, used, off);
      }
      while (hc >= 0 && used + hp + hu <= cap) {
        bool placed = false;
#pragma unroll
        for (int i = 0; i < kS; ++i) {
          if (placed) continue;
          const unsigned fl = __ballot_sync(kAll, id[i] < 0);
          if (fl == 0) continue;
          placed = true;
          if (lane == __ffs(fl) - 1) {
            id[i] = hc;
            gi[i] = 0;
            L[i] = true_len[hc];
            pr[i] = hp;
            ru[i] = hu;
            as[i] = v.seq;
            st[hc] = kRunning;
            res_u[hc] = hu;
            aseq[hc] = v.seq;
          }
        }
        if (!placed) {
          full = true;  // this admission is the general loop's
          break;
        }
        if (v.ns > 0)
          v.ns -= 1;
        else
          v.qh += 1;
        v.n += 1;
        v.seq += 1;
        v.nadm += 1;
        tok += hp;
        used += acct == MAPS_STREAM_OCCUPANCY ? static_cast<long long>(hp)
                : acct == MAPS_STREAM_STAGED  ? static_cast<long long>(hp) + hu
                                              : 2ll * hp + hu;
        head();
      }
    }
    if (!full) v.integ += v.ns + (v.qe - v.qh);  // waiting through step t
  }
  // the running set and its tokens
  int base = 0;
#pragma unroll
  for (int i = 0; i < kS; ++i) {
    const unsigned rm = __ballot_sync(kAll, id[i] >= 0);
    if (id[i] >= 0) {
      g[id[i]] = gi[i];
      rbuf[base + __popc(rm & ((1u << lane) - 1u))] = id[i];
    }
    base += __popc(rm);
  }
  __syncwarp();
}

__device__ void
interval_block(int32_t *scratch, int64_t hi, int D, int32_t cap, int acct, const int64_t *arrival,
               const int32_t *prompt, const int32_t *true_len, const int32_t *U,
               int32_t *res_u, uint8_t *st, int32_t *g, const int32_t *dec,
               const int32_t *act, const int32_t *wid, const int32_t *wperm,
               const int64_t *wseg, const int64_t *qhead, long long *aseq,
               long long *dseq, int32_t *rbuf, int32_t *sbuf, int32_t *done_id,
               int32_t *done_rem, StreamState *S, int64_t *dst) {
  int32_t *s_cnt = scratch, *s_run = scratch + kStreamMaxD, *s_cur = scratch + 2 * kStreamMaxD;
  __shared__ int s_w[kStWarps];
  __shared__ int s_done, s_adm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long s = arrival[hi - 1];
  const long long s0 = S->prev_s;
  const int nact = S->nact;
  for (int k = tid; k < D; k += kSt) s_cnt[k] = s_run[k] = 0;
  if (tid == 0) s_done = s_adm = 0;
  __syncthreads();
  // each decoder's region: room for all its requests in the system
  for (int x = tid; x < nact; x += kSt) {
    const int id = act[x];
    atomicAdd(&s_cnt[dec[id]], 1);
    if (st[id] == kRunning) atomicAdd(&s_run[dec[id]], 1);
  }
  __syncthreads();
  {
    const int c = tid < D ? s_cnt[tid] : 0;  // D <= kSt
    int incl = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += y;
    }
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    int base = 0;
    for (int w = 0; w < warp; ++w) base += s_w[w];
    if (tid < D) {
      s_cnt[tid] = base + incl - c;  // now the region's start
      s_cur[tid] = 0;
    }
  }
  __syncthreads();
  for (int x = tid; x < nact; x += kSt) {
    const int id = act[x];
    if (st[id] == kRunning) {
      const int k = dec[id];
      rbuf[s_cnt[k] + atomicAdd(&s_cur[k], 1)] = id;
    }
  }
  __syncthreads();
  for (int k = warp; k < D; k += kStWarps) {
    const int base = s_cnt[k];
    int n = s_run[k], ns = 0;
    long long qh = qhead[k];
    const long long qe = wseg[k + 1];
    long long seq = dseq[k], integ = 0;
    int npre = 0, nadm = 0;
    long long t = s0;
    bool admit_first = false;  // step t has been taken up to its admission
    if (n <= 64 && s - s0 <= 0x7fffffff) {
      IntervalRun v = {t, s, qh, qe, seq, 0, n, 0, 0, 0};
      interval_registers<2>(v, cap, acct, prompt, true_len, U, res_u, st, g, wid, wperm, aseq, rbuf + base,
                            sbuf + base, done_id, done_rem, s0, &s_done);
      t = v.t, qh = v.qh, seq = v.seq, integ = v.integ;
      n = v.n, ns = v.ns, npre = v.npre, nadm = v.nadm;
      admit_first = t < s;
    }
    while (t < s) {
      if (!admit_first) {
      long long tok = 0;
      int jc = INT_MAX;
      for (int i = lane; i < n; i += 32) {
        const int id = rbuf[base + i];
        const int gi = g[id];
        tok += static_cast<long long>(prompt[id]) + gi;
        jc = min(jc, true_len[id] - gi);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        tok += __shfl_xor_sync(0xffffffffu, tok, off);
        jc = min(jc, __shfl_xor_sync(0xffffffffu, jc, off));
      }
      // steps to the next completion (jc) and to the next preemption (jp)
      long long je = LLONG_MAX;
      if (n > 0) {
        je = jc;
        if (n > 1) je = min(je, tok + n > cap ? 1LL : (cap - tok) / n + 1);
      }
      const long long te = je >= s - t ? s : t + je;
      const long long quiet = te - t - 1;  // steps of growth alone
      if (quiet > 0) {
        for (int i = lane; i < n; i += 32) g[rbuf[base + i]] += static_cast<int>(quiet);
        integ += (static_cast<long long>(ns) + (qe - qh)) * quiet;
        tok += static_cast<long long>(n) * quiet;
      }
      t = te;
      __syncwarp();
      // step t: preempt the latest admitted while the next tokens do not fit
      while (n > 1 && tok + n > cap) {
        long long best = -1;
        int bi = 0;
        for (int i = lane; i < n; i += 32) {
          const long long a = aseq[rbuf[base + i]];
          if (a > best) {
            best = a;
            bi = i;
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          const long long ob = __shfl_xor_sync(0xffffffffu, best, off);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
          if (ob > best) {
            best = ob;
            bi = oi;
          }
        }
        const int v = rbuf[base + bi];
        tok -= static_cast<long long>(prompt[v]) + g[v];
        __syncwarp();
        if (lane == 0) {
          rbuf[base + bi] = rbuf[base + n - 1];
          sbuf[base + ns] = v;
          st[v] = kWaiting;
          g[v] = 0;
        }
        --n;
        ++ns;
        ++npre;
        __syncwarp();
      }
      // one token each; completions leave the running set (in-place compaction)
      int kept = 0;
      for (int r0 = 0; r0 < n; r0 += 32) {
        const int i = r0 + lane;
        const int id = i < n ? rbuf[base + i] : -1;
        bool fin = false;
        if (id >= 0) {
          const int gi = g[id] + 1;
          g[id] = gi;
          fin = gi == true_len[id];
          if (fin) {
            st[id] = kDone;
            const int o = atomicAdd(&s_done, 1);
            done_id[o] = id;
            done_rem[o] = static_cast<int>(t - s0);
          }
        }
        const unsigned km = __ballot_sync(0xffffffffu, id >= 0 && !fin);
        if (id >= 0 && !fin) rbuf[base + kept + __popc(km & ((1u << lane) - 1u))] = id;
        kept += __popc(km);
        __syncwarp();
      }
      n = kept;
      if (t == s) break;
      }
      admit_first = false;
      // admission in queue order (the stack first)
      long long used = 0;
      for (int i = lane; i < n; i += 32) {
        const int id = rbuf[base + i];
        const long long p = prompt[id], gi = g[id];
        const long long out = max(static_cast<long long>(res_u[id]), gi);
        used += acct == MAPS_STREAM_OCCUPANCY ? p + gi
                : acct == MAPS_STREAM_STAGED  ? p + out
                                              : 2 * p + out;
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) used += __shfl_xor_sync(0xffffffffu, used, off);
      if (lane == 0) {
        for (;;) {
          const bool from_stack = ns > 0;
          if (!from_stack && qh >= qe) break;
          const int c = from_stack ? sbuf[base + ns - 1] : wid[wperm[qh]];
          const long long p = prompt[c], uu = U[c];
          if (used + p + uu > cap) break;
          if (from_stack)
            --ns;
          else
            ++qh;
          rbuf[base + n] = c;
          ++n;
          st[c] = kRunning;
          g[c] = 0;
          res_u[c] = static_cast<int32_t>(uu);
          aseq[c] = seq++;
          used += acct == MAPS_STREAM_OCCUPANCY ? p : acct == MAPS_STREAM_STAGED ? p + uu : 2 * p + uu;
          ++nadm;
        }
      }
      n = __shfl_sync(0xffffffffu, n, 0);
      ns = __shfl_sync(0xffffffffu, ns, 0);
      qh = __shfl_sync(0xffffffffu, qh, 0);
      seq = __shfl_sync(0xffffffffu, seq, 0);
      __syncwarp();
      integ += static_cast<long long>(ns) + (qe - qh);  // waiting through step t
    }
    if (lane == 0) {
      dseq[k] = seq;
      if (dst != nullptr) {
        dst[4 * k] += integ;
        dst[4 * k + 2] += nadm;
        dst[4 * k + 3] += npre;
      }
      if (nadm) atomicAdd(&s_adm, nadm);
    }
  }
  __syncthreads();
  if (tid == 0) {
    S->ndone = s_done;
    S->adm_i = s_adm;
    S->prev_s = s;  // the advance that follows moves nobody
  }
}
__global__ void __launch_bounds__(kSt, 1)
stream_interval_kernel(int64_t hi, int D, int32_t cap, int acct, const int64_t *arrival,
                       const int32_t *prompt, const int32_t *true_len, const int32_t *U,
                       int32_t *res_u, uint8_t *st, int32_t *g, const int32_t *dec,
                       const int32_t *act, const int32_t *wid, const int32_t *wperm,
                       const int64_t *wseg, const int64_t *qhead, long long *aseq,
                       long long *dseq, int32_t *rbuf, int32_t *sbuf, int32_t *done_id,
                       int32_t *done_rem, StreamState *S, int64_t *dst) {
  pdl_prologue();
  __shared__ int32_t scratch[3 * kStreamMaxD];
  interval_block(scratch, hi, D, cap, acct, arrival, prompt, true_len, U, res_u, st, g, dec, act, wid,
                 wperm, wseg, qhead, aseq, dseq, rbuf, sbuf, done_id, done_rem, S, dst);
}

// Deferral: the requests arrived but not dispatched, then the batch, in index
// order, split three ways (stable): a bound available by s (the arrival plus
// the prediction delay) -> the dispatch policy; waited beta steps past
// arrival without one, or the last dispatch step -> round robin; otherwise
// they keep waiting for the next dispatch step.
__device__ void
select_block(int64_t lo, int nb, int64_t hi, int32_t beta, int last, const int64_t *arrival,
             const int32_t *pred_delay, const int32_t *pend_in, int32_t *pend_out,
             int32_t *cid, int32_t *tout, StreamState *S) {
  __shared__ int s_w[kStWarps];
  const long long s = arrival[hi - 1];
  const int np = S->npend, n = np + nb;
  int nc = 0, nt = 0, nk = 0;
  for (int c0 = 0; c0 < n; c0 += kSt) {
    const int x = c0 + static_cast<int>(threadIdx.x);
    int id = -1;
    bool av = false, to = false, kp = false;
    if (x < n) {
      id = x < np ? pend_in[x] : static_cast<int>(lo + (x - np));
      av = arrival[id] + pred_delay[id] <= s;
      to = !av && (arrival[id] + beta <= s || last);
      kp = !av && !to;
    }
    int tc, tt, tk;
    const int pc = block_flag_scan(av, s_w, tc);
    const int pt = block_flag_scan(to, s_w, tt);
    const int pk = block_flag_scan(kp, s_w, tk);
    if (av) cid[nc + pc] = id;
    if (to) tout[nt + pt] = id;
    if (kp) pend_out[nk + pk] = id;
    nc += tc;
    nt += tt;
    nk += tk;
  }
  if (threadIdx.x == 0) {
    S->nc = nc;
    S->nto = nt;
    S->npend = nk;
  }
}
__global__ void __launch_bounds__(kSt, 1)
stream_select_kernel(int64_t lo, int nb, int64_t hi, int32_t beta, int last, const int64_t *arrival,
                     const int32_t *pred_delay, const int32_t *pend_in, int32_t *pend_out,
                     int32_t *cid, int32_t *tout, StreamState *S) {
  pdl_prologue();
  select_block(lo, nb, hi, beta, last, arrival, pred_delay, pend_in, pend_out, cid, tout, S);
}

// 2. Completions, sorted by (step, id), enter the ring of the last Wn; the
//    c-th completion ever goes to slot c mod Wn.
__global__ void stream_window_kernel(int ndone, long long c0, int Wn, const int32_t *perm,
                                     const int32_t *done_id, const int32_t *true_len,
                                     const int32_t *pred, int32_t *win_true, int32_t *win_pred) {
  pdl_prologue();
  const int stride = gridDim.x * blockDim.x;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < ndone; x += stride) {
    if (x < ndone - Wn) continue;  // overwritten by a later completion of this batch
    const int id = done_id[perm[x]];
    const int slot = static_cast<int>((c0 + x) % Wn);
    win_true[slot] = true_len[id];
    win_pred[slot] = pred[id];
  }
}

// 3. Predictions of the requests in the system, then of the candidates
//    (the batch lo.., or the listed ids, whose prompts are gathered too).
__global__ void stream_gather_kernel(int nact, int nb, int64_t lo, const int32_t *act,
                                     const int32_t *cid, const int32_t *pred,
                                     const int32_t *prompt, int32_t *qpred, int32_t *cp) {
  pdl_prologue();
  const int stride = gridDim.x * blockDim.x;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nact + nb; x += stride) {
    if (x < nact) {
      qpred[x] = pred[act[x]];
    } else {
      const int id = cid ? cid[x - nact] : static_cast<int>(lo + (x - nact));
      qpred[x] = pred[id];
      if (cid) cp[x - nact] = prompt[id];
    }
  }
}

// 3'. No bound available: U = prediction, the batch goes round robin.  With
//     set_u = 0 only the choices (the round-robin dispatch policy).
//     choice[x] is candidate x's: lo + x, or the listed cid[x].
__global__ void stream_rr_kernel(int n, int nb, int64_t lo, int D, int set_u, const int32_t *qpred,
                                 int32_t *Uq, const int32_t *cid, int32_t *choice) {
  pdl_prologue();
  const int stride = gridDim.x * blockDim.x;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
    if (set_u) Uq[x] = qpred[x];
    if (x < nb) choice[x] = static_cast<int32_t>((cid ? static_cast<int64_t>(cid[x]) : lo + x) % D);
  }
}

// 5'. Least requests (one warp): candidate j goes to the decoder with the
//     fewest requests in the system, counting the batch's earlier choices;
//     ties to the lowest index.  Lane l keeps the counts of decoders l, l + 32,
//     ... in shared memory; per candidate two warp minima give the smallest
//     count and then the lowest decoder holding it.
__device__ void lr_warp(uint32_t *s_c, int D, int nb, const int64_t *res_off, int32_t *choice) {
  const int lane = threadIdx.x;
  for (int k = lane; k < D; k += 32) s_c[k] = static_cast<uint32_t>(res_off[k + 1] - res_off[k]);
  __syncwarp();
  for (int j = 0; j < nb; ++j) {
    uint32_t c = 0xffffffffu, ck = 0xffffffffu;  // this lane's smallest count, its lowest decoder
    for (int k = lane; k < D; k += 32)
      if (s_c[k] < c) {
        c = s_c[k];
        ck = static_cast<uint32_t>(k);
      }
    const uint32_t cmin = __reduce_min_sync(0xffffffffu, c);
    const uint32_t bk = __reduce_min_sync(0xffffffffu, c == cmin ? ck : 0xffffffffu);
    if (lane == 0) {
      choice[j] = static_cast<int32_t>(bk);
      s_c[bk] = cmin + 1;
    }
    __syncwarp();
  }
}
__global__ void stream_lr_kernel(int D, int nb, const int64_t *res_off, int32_t *choice) {
  pdl_prologue();
  __shared__ uint32_t s_c[kStreamMaxD];
  lr_warp(s_c, D, nb, res_off, choice);
}

// 4. Residents by decoder (running with g, waiting with g = 0) and the
//    waiting count per decoder; new bounds of the requests in the system.
//    Under deferral a request whose prediction is not in by s (arrival +
//    delay > s) is bounded by the horizon H.
__device__ void
csr_block(int32_t *scratch, int nact, int D, int rr, const int32_t *q_dev, int32_t *q_out_b,
          const int32_t *act, const uint8_t *st, const int32_t *g, const int32_t *dec,
          const int32_t *prompt, int32_t *Uq, int32_t *U, int64_t *res_off,
          int32_t *rp, int32_t *rg, int32_t *rU, int32_t *Q, const int64_t *arrival,
          const int32_t *pred_delay, int64_t hi, int32_t H) {
  if (pred_delay != nullptr) {  // before anything reads Uq
    const long long s = arrival[hi - 1];
    for (int x = threadIdx.x; x < nact; x += kSt) {
      const int id = act[x];
      if (arrival[id] + pred_delay[id] > s) Uq[x] = H;
    }
    __syncthreads();
  }
  int32_t *s_cnt = scratch, *s_q = scratch + kStreamMaxD, *s_cur = scratch + 2 * kStreamMaxD;
  __shared__ int s_w[kStWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int k = tid; k < D; k += kSt) s_cnt[k] = s_q[k] = 0;
  __syncthreads();
  for (int x = tid; x < nact; x += kSt) {
    const int id = act[x];
    U[id] = Uq[x];
    atomicAdd(&s_cnt[dec[id]], 1);
    if (st[id] == kWaiting) atomicAdd(&s_q[dec[id]], 1);
  }
  __syncthreads();
  const int c = tid < D ? s_cnt[tid] : 0;  // D <= kSt
  int incl = c;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  int base = 0;
  for (int w = 0; w < warp; ++w) base += s_w[w];
  if (tid < D) {
    const int ex = base + incl - c;
    s_cur[tid] = ex;
    res_off[tid] = ex;
    Q[tid] = s_q[tid];
    if (tid == D - 1) res_off[D] = ex + c;
  }
  __syncthreads();
  for (int x = tid; x < nact; x += kSt) {
    const int id = act[x];
    const int pos = atomicAdd(&s_cur[dec[id]], 1);
    rp[pos] = prompt[id];
    rg[pos] = st[id] == kRunning ? g[id] : 0;
    rU[pos] = Uq[x];
  }
  if (tid == 0) *q_out_b = rr ? -1 : q_dev[0];
}
__global__ void __launch_bounds__(kSt, 1)
stream_csr_kernel(int nact, int D, int rr, const int32_t *q_dev, int32_t *q_out_b,
                  const int32_t *act, const uint8_t *st, const int32_t *g, const int32_t *dec,
                  const int32_t *prompt, int32_t *Uq, int32_t *U, int64_t *res_off,
                  int32_t *rp, int32_t *rg, int32_t *rU, int32_t *Q, const int64_t *arrival,
                  const int32_t *pred_delay, int64_t hi, int32_t H) {
  pdl_prologue();
  __shared__ int32_t scratch[3 * kStreamMaxD];
  csr_block(scratch, nact, D, rr, q_dev, q_out_b, act, st, g, dec, prompt, Uq, U, res_off, rp, rg, rU, Q,
            arrival, pred_delay, hi, H);
}

// 5. (shared-memory form) SEQUENTIAL dispatch of the batch without a dense K.
// Decoder k's occupancy is held as its residents' pairs (e, b), sorted by e:
// on a step t the live residents are those with e > t, so
//   K_k(t) + t = S(t) + t (C(t) + 1),  S / C = b-sum / count of e > t,
// which is linear and rising between consecutive end steps.  Its maximum over
// t < u is therefore taken at t = e_i - 1 for some e_i <= u, or at t = u - 1:
// with the pairs sorted ascending and S_i / C_i the sums over pairs i.. n-1,
//   M_k(u) = max( max_{e_i <= u} S_i + (e_i - 1)(C_i + 1),
//                 S' + (u - 1)(C' + 1) ),  S' / C' over the pairs with e > u.
// (A pair tied on e with one before it gives a value no larger than the
// first's, so ties need no merging.)  Beside the sorted pairs each decoder
// keeps the suffix sums of b and the prefix maxima of the first term, so a
// score is a binary search for the pairs with e <= u and two reads.  One warp
// walks the batch: a lane scores a decoder, the warp picks (feasible with the
// smallest Q, else the largest headroom, ties to the lowest index), inserts
// (u, p + 1) into the chosen decoder's list and rebuilds its tables.  At most 32
// decoders take walk_registers below while their lists fit it, and where this
// kernel is launched by itself two warps share the walk over longer ones, one
// picking while the other updates the list chosen before: 511 candidates on 6
// decoders of some 650 pairs 1.76 against 2.56 ms by one warp.  The decisions and
// range errors are those of the dense projection followed by maps_dispatch
// SEQUENTIAL.
// Beside the batch and the unsorted pairs: the pool of sorted pairs (the
// residents of decoder k plus room for nb reservations at base_k = res_off[k] +
// k nb) with the tables.
// The packed decision key, the smallest wins: a feasible decoder (h >= 0)
// ranks by Q, an infeasible one after every feasible one by the deficit -h,
// each then by index: inf << 63 | v << 10 | k.  mc (the max-headroom rule)
// ranks every decoder as the infeasible class does, by -h: v = 2^33 - h is
// positive (h <= cap < 2^31) and, like the deficit, below 2^53 for any M the
// walk forms.
__device__ __forceinline__ unsigned long long dispatch_key(long long h, int q, int k, int mc) {
  const bool feas = h >= 0 && !mc;
  const unsigned long long v = feas ? static_cast<unsigned long long>(q)
                               : mc ? static_cast<unsigned long long>((1ll << 33) - h)
                                    : static_cast<unsigned long long>(-h);
  return (feas ? 0ull : 1ull << 63) | (v << 10) | static_cast<unsigned>(k);
}

// Shared memory of the dispatch: the batch, the residents' unsorted pairs and the
// decoders; and, after them, the sorted lists with their tables, 16 bytes a pair.
__host__ __device__ size_t stream_dispatch_smem(int D, int nact, int nb) {
  return (8 * (static_cast<size_t>(nb) + 1) + 8 * static_cast<size_t>(nact) + 16 * static_cast<size_t>(D) +
          12 * static_cast<size_t>(nb) + 15) / 16 * 16;
}
__host__ __device__ size_t stream_lists_bytes(int D, int nact, int nb) {
  return 16 * (static_cast<size_t>(nact) + static_cast<size_t>(D) * nb);
}
// Where the dispatch of nb candidates keeps its lists: 1 in shared memory, 2 in
// the spare global memory (`spare` bytes), which serves where the register walk
// is all but sure to decide the batch (at most 32 decoders with 64 requests each
// on average), 0: neither, the dense projection dispatches.
__host__ __device__ int stream_lists_place(int D, int nact, int nb, size_t smem, size_t spare) {
  const size_t base = stream_dispatch_smem(D, nact, nb), lists = stream_lists_bytes(D, nact, nb);
  if (base + lists <= smem) return 1;
  return D <= 32 && nact <= 64 * D && base <= smem && lists <= spare ? 2 : 0;
}

// Whether two warps' walk of up to 32 decoders' lists is worth leaving the one-block
// loop for, batch after batch: it saves about 4 ns a candidate and pair of its
// decoder's list, and costs 50 us.  Whole runs, every such batch left against none:
// batches of 334 on 5 decoders of some 100 pairs 1.73 against 2.01 ms, of 348 on 5
// 5.7 against 7.1, of 458 on 5 3.5 against 4.6; but of 81 on 4 of 200 4.8 against
// 2.9, of 38 on 4 4.1 against 3.0.
__host__ __device__ inline bool stream_lists_long(int D, int nact, int nb) {
  return static_cast<int64_t>(nb) * (nact + nb / 2) > static_cast<int64_t>(12000) * D;
}

// Barrier `id` over the first `count` threads (whole warps) of the block.
__device__ __forceinline__ void named_bar(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// A decoder's tables from its sorted pairs (one warp): SS[i] = sum of b over
// pairs i.. n-1, and PM[i] = the largest V over pairs 0..i, with
// V_i = SS[i] + (E[i] - 1)(n - i + 1) (K + t at t = E[i] - 1).  Returns
// whether some K(t) exceeds INT32_MAX (the projection's range error); below
// that every SS, V and PM fits 32 bits.
__device__ bool rebuild_tables(const int32_t *E, const int32_t *Bv, uint32_t *SS, uint32_t *PM,
                               int n) {
  const int lane = threadIdx.x & 31;
  unsigned long long carry = 0;
  bool over = false;
  for (int r = (n - 1) >> 5; r >= 0; --r) {  // suffix sums, last round first
    const int i = r * 32 + lane;
    const unsigned long long b = i < n ? static_cast<unsigned long long>(Bv[i]) : 0ull;
    unsigned long long suf = b;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned long long y = __shfl_down_sync(0xffffffffu, suf, off);
      if (lane + off < 32) suf += y;
    }
    if (i < n) {
      const unsigned long long ss = suf + carry;
      // K at the segment's last step: the pairs i.. n-1 are live there
      over |= ss + static_cast<unsigned long long>(E[i] - 1) * (n - i) > 0x7fffffffull;
      SS[i] = static_cast<uint32_t>(ss);
    }
    carry += __shfl_sync(0xffffffffu, suf, 0);
  }
  __syncwarp();
  uint32_t run = 0;
  for (int r = 0; r <= (n - 1) >> 5; ++r) {  // prefix maxima, first round first
    const int i = r * 32 + lane;
    uint32_t incl = i < n ? SS[i] + static_cast<uint32_t>(E[i] - 1) * static_cast<uint32_t>(n - i + 1) : 0u;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl = max(incl, y);
    }
    incl = max(incl, run);
    if (i < n) PM[i] = incl;
    run = __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  return __any_sync(0xffffffffu, over);
}

// The walk with a warp a decoder (at most 32): warp k keeps decoder k's pairs
// in registers, kS a lane in any order, each with V = K(t) + t at its last live
// step t = e - 1.  Reserving (u, p + 1) adds p + e to V where e <= u, and the
// new pair's own V is P + p + u with P = K(u - 1) + u - 1, known from scoring
// the candidate, so a reservation moves nothing.  M(u) is the larger of the V
// with e < u and P: two warp reductions.  A decision takes one
// barrier: every warp picks from the keys published before it, the winner's
// reserves, and all score the next candidate.  Keys as for maps_dispatch
// SEQUENTIAL: a feasible decoder is min(Q - q0, lim) << 5 | k, an infeasible one
// 1 << 31 | min(M - cap - x0, lim) << 5 | k; at lim the 64-bit keys decide.
// Returns false when a list outgrows 32 kS pairs (nothing is kept then).
// The winner's chain (pick, reserve, score, publish: three warp reductions of
// about 100 cycles among some 60 instructions) and 32 warps' instructions both
// cost, so what can be kept is (a feasible key, the choices of 32 candidates).
// 32 decoders at 16,000 tokens, a candidate: two warps sharing the walk over
// sorted lists in shared memory 0.6 us, this form 0.38.  (Eight candidates
// scored ahead by four lanes each, decoders reserved on meanwhile one by one:
// fewer instructions, but the chain grew, 0.55 us.)
struct WalkShared {
  uint32_t key[2][32];  // of each decoder for a candidate, by its parity
  uint32_t M[32];       // where the 64-bit keys decide: M and the queue length
  int32_t q[32];
  long long x0;
  int q0, wide, over;
};
template <int kS>
__device__ bool walk_registers(int D, int nb, int mc, const int32_t *uE, const int32_t *uB,
                               const int32_t *s_base, const int32_t *s_n, int32_t *s_q,
                               const int32_t *s_cap, const int2 *cand, int32_t *choice,
                               WalkShared &w, bool &bad) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  const bool has = k < D;
  int n = has ? s_n[k] : 0;
  const int lo = has ? s_base[k] - k * nb : 0;  // the decoder's pairs in uE, uB
  const int32_t cap = has ? s_cap[k] : 0;
  int32_t q = has ? s_q[k] : 0;
  uint32_t e[kS], b[kS], V[kS];
  if (threadIdx.x == 0) {
    w.x0 = LLONG_MAX;
    w.q0 = 0x7fffffff;
    w.wide = w.over = 0;
  }
  __syncthreads();
  long long sb = 0;
  if (has) {
    const bool fit = n <= 32 * kS;
    if (!fit && lane == 0) w.over = 1;
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      const int i = 32 * s + lane;
      e[s] = fit && i < n ? static_cast<uint32_t>(uE[lo + i]) : 0u;
      b[s] = fit && i < n ? static_cast<uint32_t>(uB[lo + i]) : 0u;
      sb += b[s];
    }
    // b-sum and count of the pairs live at e - 1
    unsigned long long S[kS];
    uint32_t C[kS];
#pragma unroll
    for (int s = 0; s < kS; ++s) S[s] = C[s] = 0;
    for (int m = 0; fit && m < n; ++m) {
      const uint32_t em = static_cast<uint32_t>(uE[lo + m]), bm = static_cast<uint32_t>(uB[lo + m]);
#pragma unroll
      for (int s = 0; s < kS; ++s)
        if (em >= e[s]) {
          S[s] += bm;
          C[s] += 1;
        }
    }
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      V[s] = 0;
      if (e[s] > 0) {
        const unsigned long long Kt = S[s] + static_cast<unsigned long long>(e[s] - 1) * C[s];
        if (Kt > 0x7fffffffull) bad = true;  // K at e - 1: the projection's range error
        V[s] = static_cast<uint32_t>(Kt) + e[s] - 1;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sb += __shfl_xor_sync(kAll, sb, off);
    if (sb > 0x7fffffffLL) bad = true;  // K at step 0
    if (lane == 0) {
      atomicMin(&w.x0, sb - cap);
      atomicMin(&w.q0, q);
    }
  }
  __syncthreads();
  if (w.over) return false;
  const long long off64 = -(w.x0 + cap);
  const uint32_t off = static_cast<uint32_t>(off64);
  // M < 2^31 + 2^28 while K is within int32: M + off cannot wrap
  if (has && lane == 0 && (off64 > (1ll << 30) || off64 < INT_MIN)) w.wide = 1;
  __syncthreads();
  const int32_t q0 = w.q0;
  const uint32_t lim = w.wide ? 0u : (1u << 26) - 2u;
  const uint32_t lim_key = lim << 5;
  if (k >= D) {
    __syncthreads();  // the one after the walk
    return w.over == 0;
  }
  if (lane >= D) w.key[0][lane] = w.key[1][lane] = ~0u;
  uint32_t P = 0, M = 0;
  const uint32_t kinf = static_cast<uint32_t>(k) + 0x80000000u;
  const int32_t capf = mc ? 0 : cap;  // mc: no decoder is feasible
  // the key while feasible: it changes with the queue length alone
  auto feasible_key = [&] {
    return (min(static_cast<uint32_t>(q - q0), lim) << 5) + static_cast<uint32_t>(k);
  };
  uint32_t fkey = feasible_key();
  // candidate (p, u) scored and its key published in `to`; ~0: invalid, or the end
  auto score = [&](int2 c, uint32_t *to) {
    const uint32_t u = static_cast<uint32_t>(c.y), t = u - 1;
    uint32_t sum = 0, vm = 0;
#pragma unroll
    for (int s = 0; s < kS; ++s) {
      const bool live = e[s] >= u;  // at step t: holds b + t tokens
      sum += live ? b[s] + t : 0u;
      vm = max(vm, live ? 0u : V[s]);
    }
    sum = __reduce_add_sync(kAll, sum);
    vm = __reduce_max_sync(kAll, vm);
    P = sum + t;
    M = max(vm, P);
    // p + 1 + M <= cap: M < cap - p
    const bool feas = static_cast<int32_t>(M) < capf - c.x && static_cast<int32_t>(M) >= 0;
    const uint32_t ikey = (min(M + off, lim) << 5) + kinf;
    if (lane == 0) to[k] = u == 0 ? ~0u : feas ? fkey : ikey;
  };
  uint32_t *now = w.key[0], *next = w.key[1];
  score(cand[0], now);
  named_bar(1, 32 * D);
  const int2 *cp = cand;
  int kept = 0;
  for (int j = 0; j < nb; ++j) {
    const int2 c1 = *++cp;  // there is one past the end
    const uint32_t best = __reduce_min_sync(kAll, now[lane]);
    int kk = static_cast<int>(best & 31u);
    if ((best & 0x7fffffffu) >= lim_key) {  // in every warp alike
      if (best == ~0u) {
        kk = -1;
        bad = true;
      } else {  // the 64-bit keys
        if (lane == 0) {
          w.M[k] = M;
          w.q[k] = q;
        }
        named_bar(1, 32 * D);
        unsigned long long k64 = ~0ull;
        if (lane < D)
          k64 = dispatch_key(static_cast<long long>(s_cap[lane]) -
                                 (static_cast<long long>(cp[-1].x) + 1 + w.M[lane]),
                             w.q[lane], lane, mc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const unsigned long long y = __shfl_xor_sync(kAll, k64, o);
          k64 = y < k64 ? y : k64;
        }
        kk = static_cast<int>(k64 & 1023u);
        named_bar(1, 32 * D);  // M and q have been read
      }
    }
    if (kk == k) {
      const int2 c = cp[-1];
      const uint32_t p = static_cast<uint32_t>(c.x), u = static_cast<uint32_t>(c.y);
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        if (e[s] - 1u < u) V[s] += p + e[s];
        if (n == 32 * s + lane) {
          e[s] = u;
          b[s] = p + 1u;
          V[s] = P + p + u;
        }
      }
      n += 1;  // past 32 kS: a list that did not fit
      // the largest new cell, K + p + t + 1, is M + p + 1
      bad |= q == 0x7fffffff || M + p > 0x7ffffffeu || M + p < M;
      q += q == 0x7fffffff ? 0 : 1;
      fkey = feasible_key();
    }
    score(c1, next);
    if (k == 0) {  // every warp knows the choices: the first one keeps and writes them
      kept = lane == (j & 31) ? kk : kept;
      if ((j & 31) == 31 || j == nb - 1) {
        if ((j & ~31) + lane <= j) choice[(j & ~31) + lane] = kept;
      }
    }
    uint32_t *const t = now;
    now = next;
    next = t;
    named_bar(1, 32 * D);
  }
  if (n > 32 * kS) w.over = 1;
  __syncthreads();
  const bool ok = w.over == 0;
  if (ok && lane == 0) s_q[k] = q;
  return ok;
}

// The sorted lists are in shared memory behind the rest, or (kGlobal) in `lists`.
// kTwo: up to 32 decoders' sorted lists are walked by two warps.  In the one-block
// loop, whose registers that code would take from the register walk (2 to 4% of its
// batches), one warp walks them, where they fit its `smem` bytes and are not long
// (stream_lists_long); else nothing is decided and the host launches the dispatch.
// *walked_lists: 0 no sorted lists (or more decoders), 1 walked here, 2 left.
template <bool kGlobal, bool kTwo>
__device__ void
dispatch_block(unsigned char *sdm, unsigned char *lists, int D, int H, int nb, int mc, const int64_t *res_off,
               const int32_t *rp, const int32_t *rg, const int32_t *rU, const int32_t *capv,
               int32_t *Q, const int32_t *cp, const int32_t *cU, int32_t *choice,
               int32_t *status, int32_t *walked_lists, size_t smem) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nact = static_cast<int>(res_off[D]);
  const int pool = nact + D * nb;
  int2 *cand = reinterpret_cast<int2 *>(sdm);                        // [nb + 1] the register walk's batch
  int32_t *uE = reinterpret_cast<int32_t *>(cand + nb + 1);          // [nact] unsorted
  int32_t *uB = uE + nact;
  int32_t *s_base = uB + nact, *s_n = s_base + D, *s_q = s_n + D, *s_cap = s_q + D;
  int32_t *s_cp = s_cap + D, *s_cu = s_cp + nb;            // [nb] the batch
  int32_t *s_ch = s_cu + nb;                               // [nb] choices (fast path)
  int32_t *E = reinterpret_cast<int32_t *>(                // [pool] sorted end steps
      kGlobal ? lists : sdm + stream_dispatch_smem(D, nact, nb));
  int32_t *Bv = E + pool;                                  // [pool] their b
  uint32_t *SS = reinterpret_cast<uint32_t *>(Bv + pool);  // [pool] suffix sums of b
  uint32_t *PM = SS + pool;                                // [pool] prefix maxima of V
  __shared__ int s_bad, s_fast;
  if (tid == 0) {
    s_bad = 0;
    s_fast = 0;
  }
  __syncthreads();
  for (int k = tid; k < D; k += kSt) {
    const int lo = static_cast<int>(res_off[k]);
    s_base[k] = lo + k * nb;
    s_n[k] = static_cast<int>(res_off[k + 1]) - lo;
    s_q[k] = Q[k];
    s_cap[k] = capv[k];
    if ((s_q[k] | s_cap[k]) < 0) s_bad = 1;
  }
  for (int j = tid; j < nb; j += kSt) {
    s_cp[j] = cp[j];
    s_cu[j] = cU[j];
  }
  for (int x = tid; x < nact; x += kSt) {  // the residents' pairs, as the projection forms them
    const int32_t p = rp[x], g = rg[x], U = rU[x];
    int32_t e = 1, b = 0;
    if ((p | g | U) < 0) {
      s_bad = 1;
    } else {
      const long long bb = static_cast<long long>(p) + g + 1;
      if (bb > 0x7fffffffLL) s_bad = 1;
      b = static_cast<int32_t>(bb > 0x7fffffffLL ? 0x7fffffffLL : bb);
      e = U - g;
      e = e < 1 ? 1 : (e > H ? H : e);
    }
    uE[x] = e;
    uB[x] = b;
  }
  __syncthreads();
  // With the Q-first rule, a decoder whose peak is provably within its capacity is
  // decided by (Q, index) alone.
  const bool quick = mc == 0;
  // Fast path (at most 32 decoders, Q-first rule): the
  // choices by (Q, index) alone, taken when every decoder is shown feasible at
  // every step, before any list is sorted.  For t < u,
  // K(t) + t = S(t) + t (C(t) + 1) with S <= the decoder's b-sum and C <= n
  // while t < e_max, and K(t) + t = t after e_max, so decoder k's peak for a
  // candidate of horizon u, after the batch's earlier reservations on k, is
  // at most
  //   max(b-sum + (min(u, e_max) - 1)(n + 1), u - 1)
  //   + the sum of p + u over those reservations
  // (each adds p + t + 1 for t < u).  While p + 1 + that bound <= cap for
  // every decoder, every decoder is feasible, so the rule picks the smallest
  // (Q, index), which is the choice taken: the decisions are the walk's, and
  // the lists need no sorting.  If some decoder might not fit at some step
  // the walk decides the whole batch (Q is written only on success).
  // The picks of the Q-first rule have a closed form: taking the smallest
  // (Q, index) and raising that Q by one, level by level, at level L every
  // decoder with Q <= L takes one candidate, in index order.  So candidate j
  // goes to level L, the smallest with cum(L) > j where
  // cum(L) = sum over k of max(0, L - Q_k + 1), and there to the
  // (j - cum(L - 1))-th decoder with Q <= L.  A scan over the levels gives
  // cum and the decoders of each (a thread a level), and each candidate's pick
  // is then found on its own (summing cum over the decoders at every probe
  // of that search took 3.82 ms for 30,000 requests on 32 decoders, the
  // table 3.6).  Then one warp per decoder sums the reservations before each
  // candidate (a scan) and checks the bound.
  if (quick && D <= 32) {
    __shared__ long long f_sb[32];
    __shared__ int f_em[32], f_cnt[32], f_inv, f_miss;
    if (tid == 0) {
      f_inv = 0;
      f_miss = 0;
    }
    __syncthreads();
    if (warp < D) {  // decoder `warp`: its residents' b-sum and largest end step
      const int k = warp, n = s_n[k], lo = s_base[k] - k * nb;
      long long sb = 0;
      int em = 1;
      for (int i = lane; i < n; i += 32) {
        sb += uB[lo + i];
        em = max(em, uE[lo + i]);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        sb += __shfl_xor_sync(0xffffffffu, sb, off);
        em = max(em, __shfl_xor_sync(0xffffffffu, em, off));
      }
      if (lane == 0) {
        f_sb[k] = sb;
        f_em[k] = em;
        f_cnt[k] = 0;
        // checked once: every Q stays within 21 bits (a Q grows by at most
        // nb), and no K of the residents reaches INT32_MAX (so the tables'
        // range checks could not fire); otherwise the walk handles the batch
        if (static_cast<long long>(s_q[k]) + nb >= (1 << 21) ||
            sb + static_cast<long long>(em - 1) * (n + 1) > 0x7fffffffLL)
          f_inv = 1;
      }
    }
    for (int j = tid; j < nb; j += kSt)
      if ((s_cp[j] | s_cu[j]) < 0) f_inv = 1;  // every candidate valid
    __syncthreads();
    if (!f_inv) {
      int qmin = 0x7fffffff;
      for (int k = 0; k < D; ++k) qmin = min(qmin, s_q[k]);
      // per level qmin + l, l < nb (the decoder at qmin alone takes nb picks by
      // the last): the picks made by its end, and the decoders taking one
      int2 *lev = cand;
      __shared__ int f_w[kStWarps];
      int before = 0;  // picks of the levels before this round's
      for (int l0 = 0; l0 < nb; l0 += kSt) {
        const int l = l0 + tid;
        uint32_t mask = 0;
        if (l < nb)
          for (int k = 0; k < D; ++k) mask |= (s_q[k] - qmin <= l ? 1u : 0u) << k;
        int c = __popc(mask);
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, c, off);
          if (lane >= off) c += y;
        }
        if (lane == 31) f_w[warp] = c;
        __syncthreads();
        const int ws = f_w[lane];
        c += before + static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(lane < warp ? ws : 0)));
        before += static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(ws)));
        if (l < nb) lev[l] = make_int2(c, static_cast<int>(mask));
        __syncthreads();
      }
      for (int j = tid; j < nb; j += kSt) {
        int lo = 0, hi = nb - 1;  // the first level whose end is past pick j
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (lev[mid].x > j)
            hi = mid;
          else
            lo = mid + 1;
        }
        int r = j - (lo > 0 ? lev[lo - 1].x : 0);  // its place among the level's decoders
        uint32_t mask = static_cast<uint32_t>(lev[lo].y);
        const bool ok = r >= 0 && r < __popc(mask);
        if (!ok) f_miss = 1;  // cannot happen; the walk would decide the batch
        int k = 0;  // the r-th set bit
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) {
          const int c = __popc(mask & ((1u << h) - 1u));
          if (r >= c) {
            r -= c;
            k += h;
            mask >>= h;
          }
        }
        s_ch[j] = ok ? k : 0;
      }
    }
    __syncthreads();
    if (!f_inv && warp < D) {
      const int k = warp, n = s_n[k], em = f_em[k];
      const long long sb = f_sb[k], cap = s_cap[k];
      long long carry = 0;  // p + u of this decoder's reservations so far
      int cnt = 0;
      bool miss = false;
      for (int j0 = 0; j0 < nb; j0 += 32) {
        const int j = j0 + lane;
        const bool ok = j < nb;
        const int32_t p = ok ? s_cp[j] : 0, U = ok ? s_cu[j] : 1;
        const int u = U < 1 ? 1 : (U > H ? H : U);
        const bool mine = ok && s_ch[j] == k;
        const long long w = mine ? static_cast<long long>(p) + u : 0;
        long long incl = w;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const long long y = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += y;
        }
        const long long add = carry + incl - w;  // the reservations before candidate j
        const long long b0 = max(sb + static_cast<long long>(min(u, em) - 1) * (n + 1),
                                 static_cast<long long>(u - 1));
        miss |= ok && static_cast<long long>(p) + 1 + b0 + add > cap;
        carry += __shfl_sync(0xffffffffu, incl, 31);
        cnt += __popc(__ballot_sync(0xffffffffu, mine));
      }
      if (__any_sync(0xffffffffu, miss) && lane == 0) f_miss = 1;
      if (lane == 0) f_cnt[k] = cnt;
    }
    __syncthreads();
    const bool fits = !f_inv && !f_miss;
    if (fits) {
      for (int j = tid; j < nb; j += kSt) choice[j] = s_ch[j];
      for (int k = tid; k < D; k += kSt) s_q[k] += f_cnt[k];
    }
    if (tid == 0) s_fast = fits ? 1 : 0;
  }
  __syncthreads();

  // At most 32 decoders: a warp each, with the lists in registers; a list that
  // outgrows a variant moves on to the next, the last one below.
  __shared__ WalkShared walk;
  bool walked = s_fast != 0;
  if (!walked && D <= 32) {
    int nmax = 0;
    for (int k = 0; k < D; ++k) nmax = max(nmax, s_n[k]);
    const int about = nmax + 2 * nb / D;
    // (p, u) of the batch, u = 0 marking an invalid candidate and the end
    for (int j = tid; j <= nb; j += kSt) {
      const int32_t p = j < nb ? s_cp[j] : -1, U = j < nb ? s_cu[j] : -1;
      cand[j] = (p | U) < 0 ? make_int2(0, 0) : make_int2(p, U < 1 ? 1 : (U > H ? H : U));
    }
    bool wbad = false;
    auto go = [&](auto walk_fn) {
      wbad = false;
      walked = walk_fn(D, nb, mc, uE, uB, s_base, s_n, s_q, s_cap, cand, choice, walk, wbad);
      __syncthreads();
    };
    if (about <= 32) go(walk_registers<1>);
    if (!walked && about <= 64) go(walk_registers<2>);
    if (!walked && about <= 128) go(walk_registers<4>);
    if (walked && wbad) s_bad = 1;
    __syncthreads();
  }

  if (!kTwo && !walked && D <= 32 &&
      (stream_lists_long(D, nact, nb) ||
       stream_dispatch_smem(D, nact, nb) + stream_lists_bytes(D, nact, nb) > smem)) {
    if (tid == 0) *walked_lists = 2;
    return;
  }
  if (!walked) {
    // sort each decoder's pairs by e (rank among the decoder's pairs, ties by
    // position), and check sum b <= INT32_MAX (K at step 0)
    for (int k = warp; k < D; k += kSt / 32) {
      const int lo = s_base[k] - k * nb, n = s_n[k], base = s_base[k];
      long long sb = 0;
      for (int i = lane; i < n; i += 32) {
        const int ei = uE[lo + i];
        int r = 0;
        for (int j2 = 0; j2 < n; ++j2) {
          const int ej = uE[lo + j2];
          r += ej < ei || (ej == ei && j2 < i);
        }
        E[base + r] = ei;
        Bv[base + r] = uB[lo + i];
        sb += uB[lo + i];
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sb += __shfl_xor_sync(0xffffffffu, sb, off);
      if (lane == 0 && sb > 0x7fffffffLL) s_bad = 1;
      __syncwarp();  // the sorted pairs are written
      if (rebuild_tables(E + base, Bv + base, SS + base, PM + base, n) && lane == 0) s_bad = 1;
    }
    __syncthreads();
  }
  if (tid == 0 && s_bad) flag_error(status, MAPS_E_RANGE);

  // The walk: one warp, no block barrier.  Lane l scores decoders l, l + 32,
  // ...: a binary search over the decoder's sorted ends gives c (the pairs with
  // e <= u), then M = max(PM[c - 1], SS[c] + (u - 1)(n - c + 1)); a packed key
  // picks (feasible first, then Q or the largest headroom, then the lowest
  // index); the warp inserts the footprint and rebuilds that decoder's tables.
  if (walked) {
    // decided above
  } else if (kTwo && D <= 32) {
    // Two warps, one decoder per lane.  Warp 0 holds each decoder's list
    // length, base, Q and capacity in registers, scores the candidates, picks
    // and books each decision and hands it to warp 1 through shared memory
    // (named barrier 1); warp 1 inserts the reservation into the chosen
    // decoder's list and scores that decoder again for the next candidate
    // (named barrier 2).  Meanwhile warp 0 scores the next candidate on the
    // lists as they stand: a reservation only raises the chosen decoder's Q
    // and occupancy, so every other decoder's key is already final and the
    // chosen one's is replaced by warp 1's.  Keys: inf << 63 | v << 10 | k,
    // the smallest wins.
    __shared__ int h_bk, h_pos, h_n, h_base, h_q, h_cap, h_c;
    __shared__ long long h_M;
    __shared__ unsigned long long h_key;
    auto clampu = [&](int32_t U) { return U < 1 ? 1 : (U > H ? H : U); };
    // c = the pairs with e <= u of a sorted list (8-ary search: eight
    // independent probes per level, one level for up to 8 pairs)
    auto count_le = [&](const int32_t *Ek, int n, int u) {
      int lo = 0, hi = n;
      while (lo < hi) {
        const int len = hi - lo;
        int nlo = lo, nhi = hi;
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // probes cover every position when len <= 8
          const int pi = lo + (len * i) / 8;
          if (Ek[pi] <= u)
            nlo = max(nlo, pi + 1);
          else
            nhi = min(nhi, pi);
        }
        lo = nlo;
        hi = nhi;
      }
      return lo;
    };
    auto key_of = [mc](int k, int q, int cap, int32_t p, long long M) {
      const long long h = static_cast<long long>(cap) - (static_cast<long long>(p) + 1 + M);
      return dispatch_key(h, q, k, mc);
    };
    if (warp == 0) {
      const int k = lane;
      const bool has = k < D;
      int n_r = has ? s_n[k] : 0, q_r = has ? s_q[k] : 0;
      const int base_r = has ? s_base[k] : 0, cap_r = has ? s_cap[k] : 0;
      bool bad = false, have = false;  // have: key, c and M are the current candidate's
      unsigned long long key = ~0ull;
      long long M = 0;
      int c = 0;
      auto score = [&](int32_t pp, int uu) {
        key = ~0ull;
        if (!has) return;
        if (quick && n_r > 0) {
          const long long mub = max(static_cast<long long>(PM[base_r + n_r - 1]),
                                    static_cast<long long>(SS[base_r]) +
                                        static_cast<long long>(uu - 1) * (n_r + 1));
          if (static_cast<long long>(pp) + 1 + mub <= cap_r) {
            key = (static_cast<unsigned long long>(q_r) << 10) | static_cast<unsigned>(k);
            c = -1;   // found at insertion
            M = mub;  // bounds every new cell: no range error (cap <= INT32_MAX)
            return;
          }
        }
        c = count_le(E + base_r, n_r, uu);
        const long long full = c > 0 ? static_cast<long long>(PM[base_r + c - 1]) : LLONG_MIN;
        const long long part = static_cast<long long>(c < n_r ? SS[base_r + c] : 0u) +
                               static_cast<long long>(uu - 1) * (n_r - c + 1);
        M = max(full, part);
        key = key_of(k, q_r, cap_r, pp, M);
      };
      for (int j = 0; j < nb; ++j) {
        const int32_t p = s_cp[j], U = s_cu[j];
        int bk = -1;
        if ((p | U) >= 0) {
          if (!have) score(p, clampu(U));
          // the warp's smallest key: one 32-bit reduction when every value
          // fits 21 bits (inf << 31 | v << 10 | k, the same order), else a ladder
          const unsigned long long kv = (key >> 10) & ((1ull << 53) - 1);
          const bool none = key == ~0ull;
          if (__all_sync(0xffffffffu, none || kv < (1ull << 21))) {
            const uint32_t k32 = none ? 0xffffffffu
                                      : (static_cast<uint32_t>(key >> 63) << 31) |
                                            (static_cast<uint32_t>(kv) << 10) | static_cast<uint32_t>(key & 1023u);
            bk = static_cast<int>(__reduce_min_sync(0xffffffffu, k32) & 1023u);
          } else {
            unsigned long long kk = key;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
              const unsigned long long o = __shfl_xor_sync(0xffffffffu, kk, off);
              kk = o < kk ? o : kk;
            }
            bk = static_cast<int>(kk & 1023u);
          }
          if (lane == bk) {  // the chosen decoder's lane books the decision
            choice[j] = bk;
            bad |= q_r == 0x7fffffff;
            q_r += q_r == 0x7fffffff ? 0 : 1;
            // every new cell K + p + t + 1 (t < u) is at most M + p + 1
            bad |= static_cast<long long>(p) + 1 + M > 0x7fffffffLL;
            h_bk = bk;
            h_pos = c;
            h_n = n_r;
            h_base = base_r;
            h_q = q_r;
            h_cap = cap_r;
            n_r += 1;
          }
        } else if (lane == 0) {
          bad = true;
          choice[j] = -1;
          h_bk = -1;
        }
        named_bar(1, 64);  // the decision goes to warp 1
        const bool nxt = j + 1 < nb;
        const int32_t p1 = nxt ? s_cp[j + 1] : 0, U1 = nxt ? s_cu[j + 1] : 0;
        const bool ok1 = nxt && (p1 | U1) >= 0;
        if (ok1) score(p1, clampu(U1));  // the chosen decoder's key is replaced below
        named_bar(2, 64);  // warp 1 has updated the list and scored it again
        if (ok1 && lane == bk) {
          key = h_key;
          c = h_c;
          M = h_M;
        }
        have = ok1;
      }
      if (__any_sync(0xffffffffu, bad) && lane == 0) flag_error(status, MAPS_E_RANGE);
      if (has) {
        s_n[k] = n_r;
        s_q[k] = q_r;
      }
    } else if (warp == 1) {
      for (int j = 0; j < nb; ++j) {
        named_bar(1, 64);
        const int bk = h_bk;
        if (bk >= 0) {
          const int n = h_n, base = h_base, m = n + 1;
          const int32_t p = s_cp[j];
          const int u = clampu(s_cu[j]);
          int pos = h_pos;  // -1: the scoring took the bound, count the pairs with e <= u here
          if (pos < 0) {
            if (n < 32)
              pos = __popc(__ballot_sync(0xffffffffu, lane < n && E[base + lane] <= u));
            else
              pos = count_le(E + base, n, u);
          }
          const bool nxt = j + 1 < nb;
          const int32_t p1 = nxt ? s_cp[j + 1] : 0, U1 = nxt ? s_cu[j + 1] : 0;
          const bool ok1 = nxt && (p1 | U1) >= 0;
          const int u1 = clampu(U1);
          int c1 = 0;
          long long M1 = 0;
          if (m <= 32) {
            // one round: lane i takes pair i of the new list; the suffix sums
            // follow from the old ones (b more before the new pair, the same
            // after it) and one shuffle scan gives the prefix maxima of V, in
            // 32 bits (the booking's check keeps every K + t within INT32_MAX)
            const int src = lane <= pos ? lane : lane - 1;
            const bool old_ok = src < n;
            const int eo = old_ok ? E[base + src] : 0, bo = old_ok ? Bv[base + src] : 0;
            const uint32_t so = old_ok ? SS[base + src] : 0u;
            const uint32_t bnew = static_cast<uint32_t>(p) + 1u;
            const int e2 = lane == pos ? u : eo;
            const int b2 = lane == pos ? static_cast<int>(bnew) : bo;
            const uint32_t suf = lane <= pos ? so + bnew : so;
            uint32_t V = lane < m ? suf + static_cast<uint32_t>(e2 - 1) * static_cast<uint32_t>(m - lane + 1) : 0u;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
              const uint32_t y = __shfl_up_sync(0xffffffffu, V, off);
              if (lane >= off) V = max(V, y);
            }
            __syncwarp();  // every lane has read the old list
            if (lane < m) {
              E[base + lane] = e2;
              Bv[base + lane] = b2;
              SS[base + lane] = suf;
              PM[base + lane] = V;
            }
            // the new list's count and table values at the next candidate's u
            c1 = __popc(__ballot_sync(0xffffffffu, lane < m && e2 <= u1));
            const uint32_t pmb = __shfl_sync(0xffffffffu, V, c1 > 0 ? c1 - 1 : 0);
            const uint32_t ssb = __shfl_sync(0xffffffffu, suf, c1 < m ? c1 : 0);
            const long long full = c1 > 0 ? static_cast<long long>(pmb) : LLONG_MIN;
            const long long part = static_cast<long long>(c1 < m ? ssb : 0u) +
                                   static_cast<long long>(u1 - 1) * (m - c1 + 1);
            M1 = max(full, part);
          } else {
            // a list past 32 pairs: shift [pos, n) up by one (last round
            // first), place the new pair, rebuild the tables
            for (int r = (n - 1) >> 5; r >= 0; --r) {
              const int i = r * 32 + lane;
              const bool mv = i < n && i >= pos;
              const int e = mv ? E[base + i] : 0, b = mv ? Bv[base + i] : 0;
              __syncwarp();
              if (mv) {
                E[base + i + 1] = e;
                Bv[base + i + 1] = b;
              }
              __syncwarp();
            }
            if (lane == 0) {
              E[base + pos] = u;
              Bv[base + pos] = p + 1;
            }
            __syncwarp();
            rebuild_tables(E + base, Bv + base, SS + base, PM + base, m);
            if (ok1) {
              c1 = count_le(E + base, m, u1);
              const long long full = c1 > 0 ? static_cast<long long>(PM[base + c1 - 1]) : LLONG_MIN;
              const long long part = static_cast<long long>(c1 < m ? SS[base + c1] : 0u) +
                                     static_cast<long long>(u1 - 1) * (m - c1 + 1);
              M1 = max(full, part);
            }
          }
          if (ok1 && lane == 0) {
            h_key = key_of(bk, h_q, h_cap, p1, M1);
            h_c = c1;
            h_M = M1;
          }
        }
        named_bar(2, 64);
      }
    }
  } else if (warp == 0) {
    for (int j = 0; j < nb; ++j) {
      const int32_t p = s_cp[j], U = s_cu[j];
      if ((p | U) < 0) {
        if (lane == 0) {
          flag_error(status, MAPS_E_RANGE);
          choice[j] = -1;
        }
        continue;
      }
      const int u = U < 1 ? 1 : (U > H ? H : U);
      unsigned long long key = ~0ull;  // inf << 63 | v << 10 | k, the smallest wins
      long long bM = 0;                // M and c of this lane's best decoder
      int bc = 0;
      for (int k = lane; k < D; k += 32) {
        const int n = s_n[k], base = s_base[k];
        if (quick && n > 0) {  // a sure fit is decided by (Q, index) alone
          const long long mub = max(static_cast<long long>(PM[base + n - 1]),
                                    static_cast<long long>(SS[base]) +
                                        static_cast<long long>(u - 1) * (n + 1));
          if (static_cast<long long>(p) + 1 + mub <= s_cap[k]) {
            const unsigned long long kk = (static_cast<unsigned long long>(s_q[k]) << 10) |
                                          static_cast<unsigned>(k);
            if (kk < key) {
              key = kk;
              bM = mub;
              bc = -1;
            }
            continue;
          }
        }
        int lo = 0, hi = n;  // c = the pairs with e <= u
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (E[base + mid] <= u)
            lo = mid + 1;
          else
            hi = mid;
        }
        const int c = lo;
        const long long full = c > 0 ? static_cast<long long>(PM[base + c - 1]) : LLONG_MIN;
        const long long part = static_cast<long long>(c < n ? SS[base + c] : 0u) +
                               static_cast<long long>(u - 1) * (n - c + 1);
        const long long M = max(full, part);
        const long long h = static_cast<long long>(s_cap[k]) - (static_cast<long long>(p) + 1 + M);
        const unsigned long long kk = dispatch_key(h, s_q[k], k, mc);
        if (kk < key) {
          key = kk;
          bM = M;
          bc = c;
        }
      }
      // The warp's smallest key.  When every value fits 21 bits the key packs
      // into 32 (inf << 31 | v << 10 | k, the same order) and one reduction
      // finds it; otherwise a shuffle ladder over the 64-bit keys.
      const unsigned long long kv = (key >> 10) & ((1ull << 53) - 1);
      const bool none = key == ~0ull;  // a lane without decoders
      int bk;
      if (__all_sync(0xffffffffu, none || kv < (1ull << 21))) {
        const uint32_t k32 = none ? 0xffffffffu
                                  : (static_cast<uint32_t>(key >> 63) << 31) |
                                        (static_cast<uint32_t>(kv) << 10) | static_cast<uint32_t>(key & 1023u);
        bk = static_cast<int>(__reduce_min_sync(0xffffffffu, k32) & 1023u);
      } else {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          const unsigned long long o = __shfl_xor_sync(0xffffffffu, key, off);
          key = o < key ? o : key;
        }
        bk = static_cast<int>(key & 1023u);
      }
      // the winner's lane (decoder bk is lane bk % 32's) hands over M and c
      const long long Mb = __shfl_sync(0xffffffffu, bM, bk & 31);
      int pos = __shfl_sync(0xffffffffu, bc, bk & 31);
      const int n = s_n[bk], base = s_base[bk];
      if (pos < 0) {  // the bound decided it: the pairs with e <= u place the new one
        int lo = 0, hi = n;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (E[base + mid] <= u)
            lo = mid + 1;
          else
            hi = mid;
        }
        pos = lo;
      }
      if (lane == 0) {
        choice[j] = bk;
        if (s_q[bk] == 0x7fffffff)
          flag_error(status, MAPS_E_RANGE);
        else
          s_q[bk] += 1;
        // every new cell K + p + t + 1 (t < u) is at most M + p + 1
        if (static_cast<long long>(p) + 1 + Mb > 0x7fffffffLL) flag_error(status, MAPS_E_RANGE);
      }
      // reserve: (u, p + 1) joins decoder bk's pairs after those with e <= u
      const int m = n + 1;
      if (m <= 32) {
        // One round: lane i takes pair i of the new list.  The suffix sums
        // follow from the old ones (b more before the new pair, the same
        // after it), and the prefix maxima of V take one shuffle scan, in 32
        // bits (the check above keeps every K + t of the new list within
        // INT32_MAX).
        const int src = lane <= pos ? lane : lane - 1;  // the old pair this lane keeps
        const bool old_ok = src < n;
        const int eo = old_ok ? E[base + src] : 0, bo = old_ok ? Bv[base + src] : 0;
        const uint32_t so = old_ok ? SS[base + src] : 0u;
        const uint32_t bnew = static_cast<uint32_t>(p) + 1u;
        const int e2 = lane == pos ? u : eo;
        const int b2 = lane == pos ? static_cast<int>(bnew) : bo;
        const uint32_t suf = lane <= pos ? so + bnew : so;
        uint32_t V = lane < m ? suf + static_cast<uint32_t>(e2 - 1) * static_cast<uint32_t>(m - lane + 1) : 0u;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, V, off);
          if (lane >= off) V = max(V, y);
        }
        __syncwarp();  // every lane has read the old list
        if (lane < m) {
          E[base + lane] = e2;
          Bv[base + lane] = b2;
          SS[base + lane] = suf;
          PM[base + lane] = V;
        }
        if (lane == 0) s_n[bk] = m;
        __syncwarp();
        continue;
      }
      for (int r = (n - 1) >> 5; r >= 0; --r) {  // shift [pos, n) up by one, last round first
        const int i = r * 32 + lane;
        const bool mv = i < n && i >= pos;
        const int e = mv ? E[base + i] : 0, b = mv ? Bv[base + i] : 0;
        __syncwarp();
        if (mv) {
          E[base + i + 1] = e;
          Bv[base + i + 1] = b;
        }
        __syncwarp();
      }
      if (lane == 0) {
        E[base + pos] = u;
        Bv[base + pos] = p + 1;
        s_n[bk] = n + 1;
      }
      __syncwarp();
      rebuild_tables(E + base, Bv + base, SS + base, PM + base, n + 1);
    }
  }
  __syncthreads();
  for (int k = tid; k < D; k += kSt) Q[k] = s_q[k];
}
template <bool kGlobal>
__global__ void __launch_bounds__(kSt, 1)
stream_dispatch_kernel(int D, int H, int nb, int mc, const int64_t *res_off, const int32_t *rp,
                       const int32_t *rg, const int32_t *rU, const int32_t *capv, int32_t *Q,
                       const int32_t *cp, const int32_t *cU, int32_t *choice, int32_t *status,
                       unsigned char *lists, StreamState *S) {
  pdl_prologue();
  extern __shared__ __align__(16) unsigned char sdm[];
  dispatch_block<kGlobal, true>(sdm, lists, D, H, nb, mc, res_off, rp, rg, rU, capv, Q, cp, cU, choice, status,
                               &S->lists, 0);
}

// 5''. Deferral: the listed requests join the waiting queues at act[nact..]:
//      with choices cch (and bounds Uq[nact + i]), or, with cch null, round
//      robin with the horizon as their bound (timed out without one).
__device__ void enqueue_list(int n, int nact, int D, int32_t H, int64_t hi, const int64_t *arrival,
                             const int32_t *ids, const int32_t *cch, const int32_t *Uq,
                             int32_t *choice_out, uint8_t *st, int32_t *dec, long long *disp,
                             int32_t *g, int32_t *U, int32_t *act, StreamState *S, int32_t *status) {
  const long long s = arrival[hi - 1];
  const int stride = gridDim.x * blockDim.x;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const int id = ids[i];
    int c = cch ? cch[i] : id % D;
    if (c < 0 || c >= D) {  // only after a range error (a bound that overflowed)
      flag_error(status, MAPS_E_RANGE);
      c = 0;
    }
    choice_out[id] = c;
    st[id] = kWaiting;
    dec[id] = c;
    disp[id] = s;
    g[id] = 0;
    U[id] = cch ? Uq[nact + i] : H;
    act[nact + i] = id;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) S->nact = nact + n;
}
__global__ void stream_enqueue_list_kernel(int n, int nact, int D, int32_t H, int64_t hi,
                                           const int64_t *arrival, const int32_t *ids,
                                           const int32_t *cch, const int32_t *Uq,
                                           int32_t *choice_out, uint8_t *st, int32_t *dec,
                                           long long *disp, int32_t *g, int32_t *U, int32_t *act,
                                           StreamState *S, int32_t *status) {
  pdl_prologue();
  enqueue_list(n, nact, D, H, hi, arrival, ids, cch, Uq, choice_out, st, dec, disp, g, U, act, S, status);
}

// 6. The batch joins the waiting queues of its decoders.
__device__ void enqueue_batch(int64_t lo, int nb, int nact, int64_t hi, int D, const int64_t *arrival,
                              const int32_t *choice, const int32_t *Uq, uint8_t *st, int32_t *dec,
                              long long *disp, int32_t *g, int32_t *U, int32_t *act,
                              StreamState *S, int32_t *status) {
  const long long s = arrival[hi - 1];
  const int stride = gridDim.x * blockDim.x;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += stride) {
    const int64_t id = lo + i;
    int c = choice[id];
    if (c < 0 || c >= D) {  // only after a range error (a bound that overflowed)
      flag_error(status, MAPS_E_RANGE);
      c = 0;
    }
    st[id] = kWaiting;
    dec[id] = c;
    disp[id] = s;
    g[id] = 0;
    U[id] = Uq[nact + i];
    act[nact + i] = static_cast<int32_t>(id);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) S->nact = nact + nb;
}
__global__ void stream_enqueue_kernel(int64_t lo, int nb, int nact, int64_t hi, int D,
                                      const int64_t *arrival, const int32_t *choice,
                                      const int32_t *Uq, uint8_t *st, int32_t *dec,
                                      long long *disp, int32_t *g, int32_t *U, int32_t *act,
                                      StreamState *S, int32_t *status) {
  pdl_prologue();
  enqueue_batch(lo, nb, nact, hi, D, arrival, choice, Uq, st, dec, disp, g, U, act, S, status);
}

// 7. The waiting requests with their order keys.
__global__ void __launch_bounds__(kSt, 1)
stream_waitlist_kernel(int n, int64_t hi, const int64_t *arrival, const int32_t *act,
                       const uint8_t *st, const int32_t *dec, const int32_t *U,
                       const long long *disp, int32_t *wid, int32_t *wdec, int32_t *wU,
                       int32_t *wwait, int32_t *warr) {
  pdl_prologue();
  __shared__ int s_w[kStWarps];
  const long long s = arrival[hi - 1];
  int nw = 0;
  for (int c0 = 0; c0 < n; c0 += kSt) {
    const int x = c0 + threadIdx.x;
    const int id = x < n ? act[x] : -1;
    const bool f = id >= 0 && st[id] == kWaiting;
    int tot;
    const int pos = block_flag_scan(f, s_w, tot);
    if (f) {
      const int o = nw + pos;
      const long long w = s - disp[id];
      wid[o] = id;
      wdec[o] = dec[id];
      wU[o] = U[id];
      wwait[o] = static_cast<int32_t>(w > 0x7fffffffLL ? 0x7fffffffLL : w);
      warr[o] = id;
    }
    nw += tot;
  }
}

// 8. Admission, one warp per decoder: entry x of the queue is admitted while
//    it and every entry before it satisfy used + (the increments of the
//    entries admitted before) + p + U <= cap, the increment being p, p + U
//    (staged) or 2p + U (held).  Each decoder's statistics gain its queue
//    left waiting times the steps to the next batch, and its admissions.
//    Per-step mode: each admission's sequence number (aseq), the queue's
//    first entry left (qhead), and the waiting requests count for the
//    dispatch step alone (the steps after it are the next interval's).
__device__ void
admit_block(int D, int32_t cap, int acct, int per_step, int nw, int64_t hi, int64_t hi_next,
            const int64_t *arrival, const int64_t *wseg, const int32_t *wperm, const int32_t *wid,
            const int32_t *prompt, const int32_t *U, const long long *used, uint8_t *st, int32_t *g,
            int32_t *res_u, long long *aseq, long long *dseq, int64_t *qhead, const StreamState *S,
            int64_t *stats_b, int64_t *dst) {
  __shared__ int s_adm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long span = per_step ? (hi_next != hi ? 1 : 0) : arrival[hi_next - 1] - arrival[hi - 1];
  if (tid == 0) s_adm = 0;
  __syncthreads();
  for (int k = warp; k < D; k += kStWarps) {
    long long u = used[k];
    const long long x1 = wseg[k + 1];
    int adm = 0;
    bool stop = false;
    for (long long b0 = wseg[k]; b0 < x1 && !stop; b0 += 32) {
      const long long x = b0 + lane;
      const bool valid = x < x1;
      const int id = valid ? wid[wperm[x]] : -1;
      const long long p = valid ? prompt[id] : 0, uu = valid ? U[id] : 0;
      const long long inc = acct == MAPS_STREAM_OCCUPANCY ? p
                            : acct == MAPS_STREAM_STAGED  ? p + uu
                                                          : 2 * p + uu;
      long long incl = inc;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
      }
      const bool ok = valid && u + (incl - inc) + p + uu <= cap;
      const unsigned fail = __ballot_sync(0xffffffffu, valid && !ok);
      const unsigned vmask = __ballot_sync(0xffffffffu, valid);
      const int nadm = fail ? __ffs(fail) - 1 : __popc(vmask);
      if (lane < nadm) {
        st[id] = kRunning;
        g[id] = 0;
        res_u[id] = static_cast<int32_t>(uu);
        if (per_step) aseq[id] = dseq[k] + adm + lane;
      }
      if (nadm > 0) u += __shfl_sync(0xffffffffu, incl, nadm - 1);
      adm += nadm;
      stop = fail != 0;
    }
    if (lane == 0 && adm) atomicAdd(&s_adm, adm);
    if (lane == 0) {  // decoder k is this warp's alone
      if (per_step) {
        dseq[k] += adm;
        qhead[k] = wseg[k] + adm;
      }
      if (dst != nullptr) {
        dst[4 * k] += (x1 - wseg[k] - adm) * span;
        dst[4 * k + 2] += adm;
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    stats_b[1] = s_adm + (per_step ? S->adm_i : 0);
    stats_b[2] = nw - s_adm;
  }
}
__global__ void __launch_bounds__(kSt, 1)
stream_admit_kernel(int D, int32_t cap, int acct, int per_step, int nw, int64_t hi, int64_t hi_next,
                    const int64_t *arrival, const int64_t *wseg, const int32_t *wperm,
                    const int32_t *wid, const int32_t *prompt, const int32_t *U,
                    const long long *used, uint8_t *st, int32_t *g, int32_t *res_u,
                    long long *aseq, long long *dseq, int64_t *qhead, const StreamState *S,
                    int64_t *stats_b, int64_t *dst) {
  pdl_prologue();
  admit_block(D, cap, acct, per_step, nw, hi, hi_next, arrival, wseg, wperm, wid, prompt, U, used, st, g,
              res_u, aseq, dseq, qhead, S, stats_b, dst);
}

struct StreamWs {
  size_t sub_bytes;  // [0, sub_bytes): workspace of the calls the loop makes
  StreamState *S;
  uint8_t *st;
  int32_t *g, *dec, *U, *res_u;
  long long *disp;
  int32_t *act[2];
  int32_t *done_id, *done_rem, *done_perm, *zeros;
  int64_t *done_seg;
  int32_t *win_true, *win_pred, *qpred, *Uq;
  int64_t *res_off;
  int32_t *rp, *rg, *rU, *capv, *Q;
  long long *used;
  int32_t *K;
  int64_t *headroom;
  int32_t *wid, *wdec, *wU, *wwait, *warr, *wperm;
  int64_t *wseg;
  int32_t *q_dev;
  // deferral
  int32_t *pend[2], *cid, *tout, *cp, *cch;
  // per-step mode
  long long *aseq, *dseq;
  int32_t *rbuf, *sbuf;
  int64_t *qhead;
};

// ---------------------------------------------------------------------------
// The loop in one block.  A batch's steps are chains of dependent small passes
// over a few hundred requests, so launched one by one they cost their launches
// (eleven, and the host's read of the counts that size them).  This kernel runs
// batches one after another on one block, steps apart by block barriers, with
// the two sorts and the quantile done in place.  32 decoders, batches of 256: 68
// -> 30 us a batch where no queue forms (30,000 requests 8.1 -> 3.5 ms), and with
// the register walk 210 -> 116 at 16,000 tokens, 330 -> 143 with per-step
// admission and deferral.
//   * the completions and each decoder's waiting requests are sorted by rank
//     (a key's place is the number of smaller keys of its group, one thread
//     counting for a key, or up to eight where the keys are few), groups past
//     kLoopRank by a bitonic network;
//   * the quantile comes from a histogram of the window's scores, as in
//     maps_calibrate's one-block form.
// It stops before a batch that does not fit (the requests in the system, the
// window, the dispatch's shared memory), or at the dispatch of one whose sorted
// lists two warps should walk; the host then runs that batch, or the rest of it, by
// the launches below and comes back when the next one fits.
// ---------------------------------------------------------------------------
// Requests in the system and the batch, at most (their sort keys take 18 bytes each
// of shared memory).  1,024 and 4,096 instead: 20,000 requests on 20 decoders at
// 40,000 tokens, batches of 512, 8.3 and 6.8 against 6.8 ms; batches of 1,024 on 32
// with room 2.8 and 1.7 against 2.6; batches of 256 with room 3.3 all three.
constexpr int kLoopActive = 2048;
constexpr int kLoopWindow = 4096;  // four scores a thread
// Keys of a group ranked by counting, n^2 comparisons by all threads against the
// network's log^2 n barriers.  128, 256 and 1,024 instead: 30,000 requests with room
// 3.65, 3.47 and 3.29 against 3.30 ms (some 250 completions a batch).
constexpr int kLoopRank = 512;
constexpr int kLoopBatches = 256;  // batches of one launch
constexpr int kLoopUsual = 1024;   // requests in the system its shared memory is first sized for
constexpr int kListsD = 16;        // with room for sorted lists below this many decoders

struct LoopArgs {
  maps_stream_cfg c;
  StreamWs w;
  const int64_t *arrival;
  const int32_t *prompt, *true_len, *pred, *pred_delay;
  int32_t *choice, *q_out;
  int64_t *stats, *dst;
  int32_t *status;
  size_t smem;       // dynamic shared memory
  int64_t nbatch;
  int64_t b0;             // the first batch to run
  long long total_done0;  // completions before it
};

// Shared memory the loop's dispatch cannot do without: none for the policies that
// walk nothing; of up to 32 decoders not the sorted lists, whose walk the host can
// launch.
__host__ __device__ inline size_t loop_dispatch_smem(const maps_stream_cfg &c, int nact, int nb) {
  if (c.dispatch_policy != MAPS_STREAM_MAPS && c.dispatch_policy != MAPS_STREAM_MC) return 0;
  return stream_dispatch_smem(c.D, nact, nb) + (c.D <= 32 ? 0 : stream_lists_bytes(c.D, nact, nb));
}

// Sorts groups of unique keys: group i is key[seg[i], seg[i + 1]), with which[x]
// the group of key x; out[x's place] gets the key.  Every thread of the block.
__device__ void sort_groups(const unsigned long long *key, const int32_t *seg, const int16_t *which,
                            int n, int groups, unsigned long long *out) {
  int tp = 1;  // threads a key: they share its comparisons
  while (tp < 8 && 2 * tp * n <= kSt) tp *= 2;
  const int sub = threadIdx.x & (tp - 1);
  for (int x0 = 0; x0 < n; x0 += kSt / tp) {
    const int x = x0 + static_cast<int>(threadIdx.x) / tp;
    int a = 0, r = 0;
    unsigned long long k = 0;
    bool rank = false;
    if (x < n) {
      a = seg[which[x]];
      const int b = seg[which[x] + 1];
      k = key[x];
      rank = b - a <= kLoopRank;
      if (rank) {
#pragma unroll 4
        for (int y = a + sub; y < b; y += tp) r += key[y] < k;
      } else if (sub == 0) {
        out[x] = k;
      }
    }
    for (int o = 1; o < tp; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (rank && sub == 0) out[a + r] = k;
  }
  __syncthreads();
  for (int i = 0; i < groups; ++i) {  // the long groups, one after another
    const int a = seg[i], m = seg[i + 1] - a;
    if (m <= kLoopRank) continue;
    unsigned long long *v = out + a;
    int P = 1;
    while (P < m) P <<= 1;
    // a network over P places, those past m holding the largest value: the
    // compare-exchanges with them never move anything (ascending runs only)
    for (int k = 2; k <= P; k <<= 1) {
      for (int x = threadIdx.x; x < P; x += kSt) {  // mirror step: both runs ascending
        const int base = x & ~(k - 1), o = x & (k - 1);
        const int y = base + (k - 1 - o);
        if (o < k / 2 && y < m && v[x] > v[y]) {
          const unsigned long long t = v[x];
          v[x] = v[y];
          v[y] = t;
        }
      }
      __syncthreads();
      for (int j = k >> 2; j > 0; j >>= 1) {
        for (int x = threadIdx.x; x < P; x += kSt) {
          const int y = x + j;
          if ((x & j) == 0 && y < m && v[x] > v[y]) {
            const unsigned long long t = v[x];
            v[x] = v[y];
            v[y] = t;
          }
        }
        __syncthreads();
      }
    }
  }
}

// The k-th smallest score of the window (n <= kLoopWindow), by the passes of
// maps_calibrate: hist has 4,096 words of shared memory.
__device__ uint32_t window_quantile(const int32_t *win_true, const int32_t *win_pred, int n, uint32_t k,
                                    uint32_t *hist) {
  __shared__ uint32_t s_warp[kStWarps], s_lo, s_k;
  __shared__ int s_wl;
  constexpr int kItems = kLoopWindow / kSt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t sv[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const int x = i * kSt + tid;
    sv[i] = x < n ? score(win_true[x], win_pred[x]) : 0u;
  }
  uint32_t lo = 0;
  int w = 32;
  for (int pass = 0; pass < 3 && w > 0; ++pass) {  // three passes always close the range
    const bool first = pass == 0;
    const int shift = w > kStepBits ? w - kStepBits : 0;
    reinterpret_cast<uint4 *>(hist)[tid] = make_uint4(0, 0, 0, 0);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      if (i * kSt >= n) break;
      int d = -1;
      if (i * kSt + tid < n && (first || (sv[i] >= lo && sv[i] - lo < (1u << w))))
        d = first ? first_bin(sv[i]) : static_cast<int>((sv[i] - lo) >> shift);
      const unsigned peers = __match_any_sync(0xffffffffu, d);
      if (d >= 0 && lane == __ffs(peers) - 1) atomicAdd(&hist[d], static_cast<uint32_t>(__popc(peers)));
    }
    __syncthreads();
    const uint4 c = reinterpret_cast<const uint4 *>(hist)[tid];
    const uint32_t tot = c.x + c.y + c.z + c.w;
    uint32_t incl = tot;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += y;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t cum = __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane] : 0u) + incl - tot;
    if (cum < k && k <= cum + tot) {
      int d = 4 * tid;
      if (k > cum + c.x) {
        cum += c.x, ++d;
        if (k > cum + c.y) {
          cum += c.y, ++d;
          if (k > cum + c.z) cum += c.z, ++d;
        }
      }
      uint32_t nlo = lo + (static_cast<uint32_t>(d) << shift);
      int nw = shift;
      if (first) first_range(d, nlo, nw);
      s_lo = nlo;
      s_wl = nw;
      s_k = k - cum;
    }
    __syncthreads();
    lo = s_lo;
    w = s_wl;
    k = s_k;
    __syncthreads();  // s_lo and the histogram are written again
  }
  return lo;
}

// (kPerStep apart: the interval's code costs the other loop registers, 5% of a
// batch that is mostly dispatch walk.)
template <bool kPerStep>
__global__ void __launch_bounds__(kSt, 1)
stream_loop_kernel(const __grid_constant__ LoopArgs a) {
  pdl_prologue();
  extern __shared__ __align__(16) unsigned char ldm[];
  __shared__ int32_t scratch[3 * kStreamMaxD];
  __shared__ int s_w[kStWarps];
  const maps_stream_cfg &c = a.c;
  const StreamWs &w = a.w;
  StreamState *const S = w.S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int D = c.D;
  const int64_t N = c.N, B = c.batch;
  const bool defer = c.beta >= 0;
  const int mc = c.dispatch_policy == MAPS_STREAM_MC ? 1 : 0;
  // groups of the sorts over the dispatch's shared memory: keys, sorted keys, ids
  unsigned long long *const key = reinterpret_cast<unsigned long long *>(ldm);
  unsigned long long *const sorted = key + kLoopActive;
  int16_t *const which = reinterpret_cast<int16_t *>(sorted + kLoopActive);
  int32_t *const seg = scratch;                    // [D + 1] group starts
  int32_t *const cur = scratch + kStreamMaxD + 8;  // [D] cursors
  int64_t b = a.b0;
  long long total_done = a.total_done0;
  __shared__ int32_t s_lists;
  if (tid == 0) s_lists = 0;  // (2 at the end: batch b stopped at its dispatch in this launch)
  for (int run = 0; run < kLoopBatches && b < a.nbatch; ++run, ++b) {
    const int64_t lo = b * B, hi = min(lo + B, N);
    const int nb = static_cast<int>(hi - lo);
    int32_t *const act_in = w.act[b & 1], *const act = w.act[(b & 1) ^ 1];
    int64_t *const stats_b = a.stats + 4 * b;
    const int npend = S->npend;
    if (defer) {
      __syncthreads();
      select_block(lo, nb, hi, c.beta, b + 1 == a.nbatch ? 1 : 0, a.arrival, a.pred_delay, w.pend[b & 1],
                   w.pend[(b & 1) ^ 1], w.cid, w.tout, S);
      __syncthreads();
    }
    const int nc = defer ? S->nc : nb, nto = defer ? S->nto : 0;
    const int most = S->nact + nto;  // requests in the system before this batch's, at most
    if (most + nc > kLoopActive || loop_dispatch_smem(c, most, nc) > a.smem) {
      __syncthreads();
      if (tid == 0) S->npend = npend;  // the batch is not started
      break;
    }
    __syncthreads();
    if (kPerStep) {  // 1'.
      interval_block(scratch, hi, D, c.cap, c.accounting, a.arrival, a.prompt, a.true_len, w.U, w.res_u, w.st,
                     w.g, w.dec, act_in, w.wid, w.wperm, w.wseg, w.qhead, w.aseq, w.dseq, w.rbuf, w.sbuf,
                     w.done_id, w.done_rem, S, a.dst);
      __syncthreads();
    }
    advance_block(hi, D, c.cap, c.accounting, kPerStep ? 1 : 0, a.arrival, a.prompt, a.true_len, w.res_u, w.st, w.g,
                  w.dec, act_in, act, w.done_id, w.done_rem, w.used, S, stats_b, a.dst);
    __syncthreads();
    int nact = S->nact;
    const int ndone = S->ndone, nwait = S->nwait;
    if (ndone > 0) {  // 2. by (step, id) into the ring
      for (int x = tid; x < ndone; x += kSt) {
        key[x] = (static_cast<unsigned long long>(w.done_rem[x]) << 32) | static_cast<uint32_t>(w.done_id[x]);
        which[x] = 0;
      }
      if (tid == 0) {
        seg[0] = 0;
        seg[1] = ndone;
      }
      __syncthreads();
      sort_groups(key, seg, which, ndone, 1, sorted);
      for (int x = max(0, ndone - c.window) + tid; x < ndone; x += kSt) {
        const int id = static_cast<int>(sorted[x] & 0xffffffffull);
        const int slot = static_cast<int>((total_done + x) % c.window);
        w.win_true[slot] = a.true_len[id];
        w.win_pred[slot] = a.pred[id];
      }
      total_done += ndone;
      __syncthreads();
    }
    // 3. the quantile; U = pred + q of the requests in the system and the candidates
    const int win = static_cast<int>(min(total_done, static_cast<long long>(c.window)));
    const long long rank = (static_cast<long long>(1000000u - c.alpha_ppm) * (win + 1) + 999999) / 1000000;
    const bool rr = rank > win;
    int32_t q = 0;
    if (!rr) {
      const uint32_t qq = window_quantile(w.win_true, w.win_pred, win, static_cast<uint32_t>(rank),
                                          reinterpret_cast<uint32_t *>(ldm));
      if (qq > 0x7fffffffu) {
        if (tid == 0) flag_error(a.status, MAPS_E_RANGE);
      } else {
        q = static_cast<int32_t>(qq);
      }
    }
    if (tid == 0) *w.q_dev = q;
    if (nto > 0) {  // timed out: round robin with the horizon as bound
      __syncthreads();  // every thread has read S->nact, which the enqueue sets
      enqueue_list(nto, nact, D, c.H, hi, a.arrival, w.tout, nullptr, w.Uq, a.choice, w.st, w.dec, w.disp, w.g,
                   w.U, act, S, a.status);
      nact += nto;
      __syncthreads();
    }
    const int32_t *const cids = defer ? w.cid : nullptr;
    int32_t *const cch = defer ? w.cch : a.choice + lo;
    const int32_t *const cpr = defer ? w.cp : a.prompt + lo;
    for (int x = tid; x < nact + nc; x += kSt) {
      const int id = x < nact ? act[x] : cids ? cids[x - nact] : static_cast<int>(lo + (x - nact));
      const long long u = static_cast<long long>(a.pred[id]) + q;  // Eq. (conformal_upper)
      if (u > 0x7fffffffLL) flag_error(a.status, MAPS_E_RANGE);
      w.Uq[x] = static_cast<int32_t>(u > 0x7fffffffLL ? 0x7fffffffLL : u);
      if (x >= nact && cids) w.cp[x - nact] = a.prompt[id];
    }
    if (rr || c.dispatch_policy == MAPS_STREAM_RR)  // 3'., 5'.
      for (int x = tid; x < nc; x += kSt)
        cch[x] = static_cast<int32_t>((cids ? static_cast<int64_t>(cids[x]) : lo + x) % D);
    __syncthreads();
    csr_block(scratch, nact, D, rr ? 1 : 0, w.q_dev, a.q_out + b, act, w.st, w.g, w.dec, a.prompt, w.Uq, w.U,
              w.res_off, w.rp, w.rg, w.rU, w.Q, a.arrival, defer ? a.pred_delay : nullptr, hi, c.H);  // 4.
    __syncthreads();
    if (nc > 0 && !rr && c.dispatch_policy == MAPS_STREAM_LR) {
      if (warp == 0) lr_warp(reinterpret_cast<uint32_t *>(scratch), D, nc, w.res_off, cch);
      __syncthreads();
    } else if (nc > 0 && !rr && c.dispatch_policy != MAPS_STREAM_RR) {  // 5.
      dispatch_block<false, false>(ldm, nullptr, D, c.H, nc, mc, w.res_off, w.rp, w.rg, w.rU, w.capv, w.Q, cpr,
                                   w.Uq + nact, cch, a.status, &s_lists, a.smem);
      __syncthreads();
      if (s_lists == 2) break;  // the host takes the batch up from here
    }
    if (!defer)  // 6.
      enqueue_batch(lo, nb, nact, hi, D, a.arrival, a.choice, w.Uq, w.st, w.dec, w.disp, w.g, w.U, act, S,
                    a.status);
    else if (nc > 0)
      enqueue_list(nc, nact, D, c.H, hi, a.arrival, w.cid, w.cch, w.Uq, a.choice, w.st, w.dec, w.disp, w.g, w.U,
                   act, S, a.status);
    // 7. each decoder's waiting requests in local order
    const int n_all = nact + nc, nw = nwait + nto + nc;
    for (int k = tid; k <= D; k += kSt) seg[k] = 0;
    __syncthreads();
    const long long s_b = a.arrival[hi - 1];
    for (int x = tid; x < n_all; x += kSt) {
      const int id = act[x];
      if (w.st[id] == kWaiting) atomicAdd(&seg[w.dec[id] + 1], 1);
    }
    __syncthreads();
    {  // inclusive scan of the counts: seg[k] becomes decoder k's start (D <= kSt)
      int v = tid < D ? seg[tid + 1] : 0;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += y;
      }
      if (lane == 31) s_w[warp] = v;
      __syncthreads();
      v += static_cast<int>(__reduce_add_sync(0xffffffffu, lane < warp ? static_cast<unsigned>(s_w[lane]) : 0u));
      if (tid < D) {
        seg[tid + 1] = v;
        w.wseg[tid + 1] = v;
        if (tid + 1 < D) cur[tid + 1] = v;
      }
      if (tid == 0) {
        w.wseg[0] = 0;
        cur[0] = 0;
      }
      __syncthreads();
    }
    for (int x = tid; x < n_all; x += kSt) {
      const int id = act[x];
      if (w.st[id] == kWaiting) {
        const int k = w.dec[id];
        // promoted (waited past max_wait, or FCFS) before the rest, then the
        // bound of the others, then the index, which is the arrival order
        const bool promoted = c.local_order == MAPS_STREAM_FCFS || min(s_b - w.disp[id], 0x7fffffffLL) > c.max_wait;
        const int o = atomicAdd(&cur[k], 1);
        key[o] = (promoted ? 0ull : (1ull << 62) | (static_cast<unsigned long long>(w.U[id]) << 31)) |
                 static_cast<uint32_t>(id);
        which[o] = static_cast<int16_t>(k);
      }
    }
    __syncthreads();
    sort_groups(key, seg, which, nw, D, sorted);
    for (int x = tid; x < nw; x += kSt) {
      w.wid[x] = static_cast<int32_t>(sorted[x] & 0x7fffffffull);
      w.wperm[x] = x;
    }
    __syncthreads();
    const int64_t hi_next = b + 1 < a.nbatch ? min(hi + B, N) : hi;
    admit_block(D, c.cap, c.accounting, kPerStep ? 1 : 0, nw, hi, hi_next, a.arrival, w.wseg, w.wperm, w.wid, a.prompt,
                w.U, w.used, w.st, w.g, w.res_u, w.aseq, w.dseq, w.qhead, S, stats_b, a.dst);  // 8.
    __syncthreads();
  }
  __syncthreads();
  if (tid == 0) {
    S->next_b = b;
    S->total_done = total_done;
    S->lists = s_lists;
  }
}

size_t stream_sub_bytes(const maps_stream_cfg &c) {
  size_t b = maps_calibrate_workspace_size(c.window, c.N);
  b = std::max(b, maps_project_occupancy_workspace_size(c.D, c.H, c.N));
  b = std::max(b, maps_dispatch_workspace_size(MAPS_MODE_SEQUENTIAL, c.D, c.H, c.batch));
  b = std::max(b, maps_order_local_workspace_size(c.N, c.D));
  b = std::max(b, maps_order_local_workspace_size(c.N, 1));
  return (b + kAlign - 1) / kAlign * kAlign;
}

StreamWs carve_stream(Carve &c, const maps_stream_cfg &cfg) {
  StreamWs w;
  const size_t N = static_cast<size_t>(cfg.N), D = static_cast<size_t>(cfg.D);
  w.sub_bytes = stream_sub_bytes(cfg);
  c.off = w.sub_bytes;
  w.S = c.take<StreamState>(1);
  w.st = c.take<uint8_t>(N);
  w.g = c.take<int32_t>(N);
  w.dec = c.take<int32_t>(N);
  w.U = c.take<int32_t>(N);
  w.res_u = c.take<int32_t>(N);
  w.disp = c.take<long long>(N);
  w.act[0] = c.take<int32_t>(N);
  w.act[1] = c.take<int32_t>(N);
  w.done_id = c.take<int32_t>(N);
  w.done_rem = c.take<int32_t>(N);
  w.done_perm = c.take<int32_t>(N);
  w.zeros = c.take<int32_t>(N);
  w.done_seg = c.take<int64_t>(2);
  w.win_true = c.take<int32_t>(static_cast<size_t>(cfg.window));
  w.win_pred = c.take<int32_t>(static_cast<size_t>(cfg.window));
  w.qpred = c.take<int32_t>(N);
  w.Uq = c.take<int32_t>(N);
  w.res_off = c.take<int64_t>(D + 1);
  w.rp = c.take<int32_t>(N);
  w.rg = c.take<int32_t>(N);
  w.rU = c.take<int32_t>(N);
  w.capv = c.take<int32_t>(D);
  w.Q = c.take<int32_t>(D);
  w.used = c.take<long long>(D);
  w.K = c.take<int32_t>(D * static_cast<size_t>(cfg.H));
  w.headroom = c.take<int64_t>(static_cast<size_t>(cfg.batch));
  w.wid = c.take<int32_t>(N);
  w.wdec = c.take<int32_t>(N);
  w.wU = c.take<int32_t>(N);
  w.wwait = c.take<int32_t>(N);
  w.warr = c.take<int32_t>(N);
  w.wperm = c.take<int32_t>(N);
  w.wseg = c.take<int64_t>(D + 1);
  w.q_dev = c.take<int32_t>(1);
  const bool defer = cfg.beta >= 0;
  w.pend[0] = c.take<int32_t>(defer ? N : 0);
  w.pend[1] = c.take<int32_t>(defer ? N : 0);
  w.cid = c.take<int32_t>(defer ? N : 0);
  w.tout = c.take<int32_t>(defer ? N : 0);
  w.cp = c.take<int32_t>(defer ? N : 0);
  w.cch = c.take<int32_t>(defer ? N : 0);
  const bool ps = cfg.per_step != 0;
  w.aseq = c.take<long long>(ps ? N : 0);
  w.dseq = c.take<long long>(ps ? D : 0);
  w.rbuf = c.take<int32_t>(ps ? N : 0);
  w.sbuf = c.take<int32_t>(ps ? N : 0);
  w.qhead = c.take<int64_t>(ps ? D : 0);
  return w;
}

bool cfg_ok(const maps_stream_cfg *c) {
  return c != nullptr && c->N >= 1 && c->N <= 0x7fffffffLL && c->D >= 1 && c->D <= kStreamMaxD &&
         c->H >= 1 && c->H <= (1 << 28) && c->cap >= 0 && c->batch >= 1 && c->window >= 1 &&
         c->alpha_ppm > 0 && c->alpha_ppm < 1000000u && c->dispatch_policy >= MAPS_STREAM_MAPS &&
         c->dispatch_policy <= MAPS_STREAM_LR && c->local_order >= MAPS_STREAM_SJF &&
         c->local_order <= MAPS_STREAM_FCFS && c->accounting >= MAPS_STREAM_OCCUPANCY &&
         c->accounting <= MAPS_STREAM_HELD && (c->per_step == 0 || c->per_step == 1);
}

int grid_for(int64_t n, int threads = 256) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads,
                                                                 4LL * sm_count())));
}

}  // namespace
}  // namespace maps

extern "C" {

size_t maps_stream_workspace_size(const maps_stream_cfg *cfg) {
  using namespace maps;
  if (!cfg_ok(cfg)) return kCtrlBytes;
  Carve c(nullptr);
  carve_stream(c, *cfg);
  return c.bytes();
}

int maps_stream_run(const maps_stream_cfg *cfg, const int64_t *arrival_ms, const int32_t *prompt,
                    const int32_t *true_len, const int32_t *pred, const int32_t *pred_delay,
                    int32_t *choice_out, int32_t *q_out, int64_t *stats_out,
                    int64_t *dec_stats_out, void *ws, size_t ws_bytes, void *stream) {
  using namespace maps;
  if (!cfg_ok(cfg) || arrival_ms == nullptr || prompt == nullptr || true_len == nullptr ||
      pred == nullptr || choice_out == nullptr || q_out == nullptr || stats_out == nullptr ||
      (cfg->beta >= 0 && pred_delay == nullptr))
    return MAPS_E_INVALID;
  MAPS_TRY(check_ws(ws, ws_bytes, maps_stream_workspace_size(cfg)));
  const maps_stream_cfg c = *cfg;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int32_t *status = status_word(ws);
  Carve cv(ws);
  const StreamWs w = carve_stream(cv, c);
  const int64_t N = c.N, B = c.batch, nbatch = (N + B - 1) / B;
  const int D = c.D;
  const bool defer = c.beta >= 0;
  const int per_step = c.per_step;
  const int32_t *pdl = defer ? pred_delay : nullptr;

  MAPS_TRY(cuda_ok(cudaMemsetAsync(w.st, 0, static_cast<size_t>(N), s)));
  MAPS_TRY(cuda_ok(cudaMemsetAsync(w.zeros, 0, static_cast<size_t>(N) * sizeof(int32_t), s)));
  if (dec_stats_out != nullptr)
    MAPS_TRY(cuda_ok(cudaMemsetAsync(dec_stats_out, 0, static_cast<size_t>(c.D) * 4 * sizeof(int64_t), s)));
  if (per_step) {
    MAPS_TRY(cuda_ok(cudaMemsetAsync(w.dseq, 0, static_cast<size_t>(D) * sizeof(long long), s)));
    MAPS_TRY(cuda_ok(cudaMemsetAsync(w.qhead, 0, static_cast<size_t>(D) * sizeof(int64_t), s)));
    MAPS_TRY(cuda_ok(cudaMemsetAsync(w.wseg, 0, static_cast<size_t>(D + 1) * sizeof(int64_t), s)));
  }
  launch_pdl(stream_init_kernel, 1, kSt, 0, s, std::min(N, B), D, c.cap, arrival_ms, w.capv, w.S);
  launch_pdl(stream_validate_kernel, grid_for(N), 256, 0, s, N, arrival_ms, prompt, true_len, pred,
             pdl, status);
  MAPS_TRY(launch_ok());
  {
    const int st0 = maps_check(ws, stream);  // a bad input stops the loop before it starts
    if (st0 != MAPS_OK) return st0;
  }

  long long total_done = 0;
  StreamState hs;
  // the one-block loop, where a batch fits it
  void (*const loop)(LoopArgs) = per_step ? stream_loop_kernel<true> : stream_loop_kernel<false>;
  cudaFuncAttributes fa;
  MAPS_TRY(cuda_ok(cudaFuncGetAttributes(&fa, loop)));
  const size_t loop_smem = smem_beside(fa.sharedSizeBytes);
  MAPS_TRY(allow_smem(loop, loop_smem));
  const size_t spare = sizeof(int32_t) * static_cast<size_t>(D) * c.H;  // the dense K, else unused
  // What the loop leaves of the multiprocessor's memory is its L1 cache, which
  // the requests' state then hits: it starts with what the usual batch needs, and
  // takes all of it where a batch does not fit that.  The usual batch has kLoopUsual
  // requests in the system, and sorted lists below kListsD decoders (above, lists
  // past the register walk's 128 pairs are rare in a system of 2,048).
  const int nb0 = static_cast<int>(std::min(B, static_cast<int64_t>(kLoopActive)));
  size_t usual = loop_dispatch_smem(c, D >= kListsD && D <= 32 ? kLoopActive : kLoopUsual, nb0);
  if (usual > 0 && D < kListsD) usual += stream_lists_bytes(D, kLoopUsual, nb0);
  usual = std::max<size_t>({usual, 18 * kLoopActive, sizeof(uint32_t) << kStepBits});  // the sorts, the quantile
  usual = std::min(usual, loop_smem);
  size_t give = usual;
  auto loop_fits = [&](int64_t system, int64_t cands) {  // requests in the system, candidates
    return c.window <= kLoopWindow && system + cands <= kLoopActive &&
           loop_dispatch_smem(c, static_cast<int>(system), static_cast<int>(cands)) <= loop_smem;
  };
  // whether the loop, with all of the memory, walks that batch's lists itself
  auto walks_here = [&](int64_t system, int64_t cands) {
    const int n = static_cast<int>(system), nc = static_cast<int>(cands);
    return !stream_lists_long(D, n, nc) &&
           stream_dispatch_smem(D, n, nc) + stream_lists_bytes(D, n, nc) <= loop_smem;
  };
  bool in_loop = loop_fits(0, std::min(N, B));
  int64_t left = -1;  // the batch the loop last left at its dispatch
  for (int64_t b = 0; b < nbatch; ++b) {
    bool resume = false;  // the loop has taken batch b up to its dispatch
    if (in_loop) {
      LoopArgs la;
      la.c = c;
      la.w = w;
      la.arrival = arrival_ms;
      la.prompt = prompt;
      la.true_len = true_len;
      la.pred = pred;
      la.pred_delay = pred_delay;
      la.choice = choice_out;
      la.q_out = q_out;
      la.stats = stats_out;
      la.dst = dec_stats_out;
      la.status = status;
      la.smem = give;
      la.nbatch = nbatch;
      la.b0 = b;
      la.total_done0 = total_done;
      launch_pdl(loop, 1, kSt, give, s, la);
      MAPS_TRY(launch_ok());
      MAPS_TRY(cuda_ok(cudaMemcpyAsync(&hs, w.S, sizeof(hs), cudaMemcpyDeviceToHost, s)));
      MAPS_TRY(cuda_ok(cudaStreamSynchronize(s)));
      const bool stopped = hs.next_b < nbatch && hs.next_b < b + kLoopBatches;
      b = hs.next_b;
      total_done = hs.total_done;
      resume = hs.lists == 2;
      if (resume && walks_here(hs.nact, defer ? hs.nc : std::min(B, N - b * B))) give = loop_smem;
      if (!resume && (!stopped || give < loop_smem)) {
        --b;  // all done, or a launch's worth, or on with all of the memory
        give = stopped ? loop_smem : usual;
        continue;
      }
      in_loop = false;  // batch b does not fit, or its lists are long: it runs here
    }
    const int64_t lo = b * B, hi = std::min(lo + B, N);
    const int nb = static_cast<int>(hi - lo);
    int32_t *act_in = w.act[b & 1], *act = w.act[(b & 1) ^ 1];
    int64_t *stats_b = stats_out + 4 * b;
    if (!resume) {
      if (defer)  // 4 (first half): who is dispatched at this step
        launch_pdl(stream_select_kernel, 1, kSt, 0, s, lo, nb, hi, c.beta, b + 1 == nbatch ? 1 : 0,
                   arrival_ms, pred_delay, w.pend[b & 1], w.pend[(b & 1) ^ 1], w.cid, w.tout, w.S);
      if (per_step)  // 1'.
        launch_pdl(stream_interval_kernel, 1, kSt, 0, s, hi, D, c.cap, c.accounting, arrival_ms,
                   prompt, true_len, w.U, w.res_u, w.st, w.g, w.dec, act_in, w.wid, w.wperm, w.wseg,
                   w.qhead, w.aseq, w.dseq, w.rbuf, w.sbuf, w.done_id, w.done_rem, w.S, dec_stats_out);
      launch_pdl(stream_advance_kernel, 1, kSt, 0, s, hi, D, c.cap, c.accounting, per_step, arrival_ms,
                 prompt, true_len, w.res_u, w.st, w.g, w.dec, act_in, act, w.done_id, w.done_rem,
                 w.used, w.S, stats_b, dec_stats_out);
      MAPS_TRY(launch_ok());
      MAPS_TRY(cuda_ok(cudaMemcpyAsync(&hs, w.S, sizeof(hs), cudaMemcpyDeviceToHost, s)));
      MAPS_TRY(cuda_ok(cudaStreamSynchronize(s)));
    }
    int nact = hs.nact;
    const int ndone = hs.ndone, nwait = hs.nwait;
    // the policy's candidates: the batch, or (deferral) the listed ids
    const int nc = defer ? hs.nc : nb, nto = defer ? hs.nto : 0;
    const int32_t *cids = defer ? w.cid : nullptr;
    const int32_t *cpr = defer ? w.cp : prompt + lo;
    int32_t *cch = defer ? w.cch : choice_out + lo;

    bool rr = false;  // (a batch taken up has a bound)
    if (!resume) {
      if (ndone > 0) {  // 2.
        MAPS_TRY(maps_order_local(ndone, 1, w.zeros, w.done_rem, w.zeros, w.done_id, 0, w.done_perm,
                                  w.done_seg, ws, w.sub_bytes, stream));
        launch_pdl(stream_window_kernel, grid_for(ndone), 256, 0, s, ndone, total_done, c.window,
                                                             w.done_perm, w.done_id, true_len, pred,
                                                             w.win_true, w.win_pred);
        total_done += ndone;
      }
      const int64_t win_len = std::min<long long>(total_done, c.window);
      if (nto > 0) {  // 4 (second half): timed out, round robin with the horizon as bound
        launch_pdl(stream_enqueue_list_kernel, grid_for(nto), 256, 0, s, nto, nact, D, c.H, hi,
                   arrival_ms, w.tout, nullptr, w.Uq, choice_out, w.st, w.dec, w.disp, w.g, w.U, act,
                   w.S, status);
        nact += nto;
      }

      launch_pdl(stream_gather_kernel, grid_for(nact + nc), 256, 0, s, nact, nc, lo, act, cids, pred,
                 prompt, w.qpred, w.cp);
      const int cs = maps_calibrate(w.win_true, w.win_pred, win_len, c.alpha_ppm, w.qpred, nact + nc,
                                    w.Uq, w.q_dev, nullptr, ws, w.sub_bytes, stream);  // 3.
      rr = cs == MAPS_E_UNBOUNDED;
      if (cs != MAPS_OK && !rr) return cs;
      if (rr)
        launch_pdl(stream_rr_kernel, grid_for(nact + nc), 256, 0, s, nact + nc, nc, lo, D, 1, w.qpred,
                   w.Uq, cids, cch);
      launch_pdl(stream_csr_kernel, 1, kSt, 0, s, nact, D, rr ? 1 : 0, w.q_dev, q_out + b, act, w.st, w.g,
                 w.dec, prompt, w.Uq, w.U, w.res_off, w.rp, w.rg, w.rU, w.Q, arrival_ms, pdl, hi,
                 c.H);  // 4.
      MAPS_TRY(launch_ok());
    }
    const int mc = c.dispatch_policy == MAPS_STREAM_MC ? 1 : 0;
    if (nc == 0) {
      // nobody to dispatch at this step
    } else if (!rr && c.dispatch_policy == MAPS_STREAM_RR) {  // 5'.
      launch_pdl(stream_rr_kernel, grid_for(nc), 256, 0, s, nc, nc, lo, D, 0, w.qpred, w.Uq, cids, cch);
      MAPS_TRY(launch_ok());
    } else if (!rr && c.dispatch_policy == MAPS_STREAM_LR) {
      launch_pdl(stream_lr_kernel, 1, 32, 0, s, D, nc, w.res_off, cch);
      MAPS_TRY(launch_ok());
    } else if (!rr) {  // 5.
      const size_t most = smem_beside(4096);  // (the kernel's static arrays take 1.2 KB)
      const int place = stream_lists_place(D, nact, nc, most, spare);
      if (place != 0) {
        // the decoders' pairs and the batch fit in shared memory: no dense projection
        const size_t dsm = stream_dispatch_smem(D, nact, nc) + (place == 1 ? stream_lists_bytes(D, nact, nc) : 0);
        const auto kern = place == 1 ? stream_dispatch_kernel<false> : stream_dispatch_kernel<true>;
        MAPS_TRY(allow_smem(kern, most));
        launch_pdl(kern, 1, kSt, dsm, s, D, c.H, nc, mc, w.res_off, w.rp, w.rg, w.rU, w.capv, w.Q, cpr,
                   w.Uq + nact, cch, status,
                   place == 1 ? nullptr : reinterpret_cast<unsigned char *>(w.K), w.S);
        MAPS_TRY(launch_ok());
      } else {
        MAPS_TRY(maps_project_occupancy(D, c.H, w.res_off, nact, w.rp, w.rg, w.rU, w.K, nullptr, ws,
                                        w.sub_bytes, stream));
        MAPS_TRY(dispatch_sequential(D, c.H, w.K, w.capv, w.Q, nc, cpr, w.Uq + nact, cch,
                                     w.headroom, mc != 0, ws, s));
      }
    }
    if (defer) {
      if (nc > 0)
        launch_pdl(stream_enqueue_list_kernel, grid_for(nc), 256, 0, s, nc, nact, D, c.H, hi,
                   arrival_ms, w.cid, w.cch, w.Uq, choice_out, w.st, w.dec, w.disp, w.g, w.U, act,
                   w.S, status);  // 6.
    } else {
      launch_pdl(stream_enqueue_kernel, grid_for(nb), 256, 0, s, lo, nb, nact, hi, D, arrival_ms,
                 choice_out, w.Uq, w.st, w.dec, w.disp, w.g, w.U, act, w.S, status);  // 6.
    }
    const int n_all = nact + nc, nw = nwait + nto + nc;
    launch_pdl(stream_waitlist_kernel, 1, kSt, 0, s, n_all, hi, arrival_ms, act, w.st, w.dec, w.U, w.disp,
                                             w.wid, w.wdec, w.wU, w.wwait, w.warr);  // 7.
    MAPS_TRY(launch_ok());
    // FCFS: every wait is >= 0 > -1, so every entry is promoted: arrival order
    const int32_t mw = c.local_order == MAPS_STREAM_FCFS ? -1 : c.max_wait;
    MAPS_TRY(maps_order_local(nw, D, w.wdec, w.wU, w.wwait, w.warr, mw, w.wperm, w.wseg, ws,
                              w.sub_bytes, stream));
    const int64_t hi_next = b + 1 < nbatch ? std::min(hi + B, N) : hi;
    launch_pdl(stream_admit_kernel, 1, kSt, 0, s, D, c.cap, c.accounting, per_step, nw, hi, hi_next,
               arrival_ms, w.wseg, w.wperm, w.wid, prompt, w.U, w.used, w.st, w.g, w.res_u, w.aseq,
               w.dseq, w.qhead, w.S, stats_b, dec_stats_out);  // 8.
    MAPS_TRY(launch_ok());
    // back to the one block once the next batch is sure to fit; but not while lists
    // that it leaves to the host are walked (as of the batch before), or right after
    // two such batches in a row
    const bool again = walks_here(nact, nc) || (resume ? left != b - 1 : hs.lists == 0);
    if (resume) left = b;
    in_loop = again && loop_fits(n_all, B + hs.npend);
  }
  return maps_check(ws, stream);
}

}  // extern "C"
