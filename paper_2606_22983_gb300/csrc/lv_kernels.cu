// CUDA kernels of the KV swap path (sm_103a).
//
//   ranking   k_select; k_rank_census -> k_rank_emit          (Section 5.1, Eq. 4)
//   allocate  k_alloc                                        (lowest free, Section 5.1)
//   move      k_swap_out / k_swap_in                         (Section 5, Fig. 6; Section 5.2)
//             k_exchange_plan -> k_exchange_copy             (both directions in one step)
//             k_stage_tasks (TMA) / k_stage_tasks_lsu         (staged copy-engine path)
//   commit    k_remap (-> k_release), k_cancel, k_append     (Section 6 side tables)
//   monitor   k_events                                       (Section 3, Sections 5.1-5.2)
//   step      k_step -> k_exchange_copy                      (a whole turn, preload or eviction
//                                                             decided on the device)
//   verify    k_checksum                                     (page checksums)
//
// The only waits are the TMA stage kernel's mbarrier waits for its own copies,
// each limited by %globaltimer to one second, after which the kernel reports
// LV_ERR_TIMEOUT and returns, and the barriers of a cluster's CTAs, which run together; no
// kernel waits on another kernel or agent.  Every
// index read from memory is range-checked and a bad item is skipped with the
// sticky error set.
#include <cooperative_groups.h>
#include <cstdint>
#include <utility>

#include "lv_internal.cuh"

namespace cg = cooperative_groups;

namespace lv {

namespace {

__device__ __forceinline__ void set_error(long long* ctl, int code, long long detail) {
  if (atomicCAS(reinterpret_cast<unsigned long long*>(&ctl[C_ERR]), 0ull,
                (unsigned long long)code) == 0ull) {
    ctl[C_ERR_DETAIL] = detail;
  }
}

// Programmatic dependent launch.  Most kernels are launched so that each may be
// scheduled while the previous kernel on the stream still runs (its launch
// latency overlaps that kernel).  pdl_entry() waits until the previous kernel
// has completed and its writes are visible, and then lets the next kernel of
// the stream be scheduled.  Before it a kernel may read only what never changes
// after the pool's creation (k_exchange_copy: the sub-page arrays' addresses).
// In a kernel launched the ordinary way both instructions have no effect.
__device__ __forceinline__ void pdl_entry() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The same two steps apart, for a kernel with a large grid: it waits at its start and
// lets the next kernel be scheduled only when its own work is done, so that the next
// kernel's CTAs do not sit on SMs, waiting, while this grid still needs them.  A CTA
// that returns early counts as having let it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Blocks of a context of `ctx` tokens, at most maxB (a 32-bit division: a 64-bit one costs
// some 100 instructions in the chain of dependent reads).
__device__ __forceinline__ int32_t blocks_of_context(const DevPool& p, int32_t ctx) {
  if (ctx <= 0) return 0;
  const uint32_t nb = ((uint32_t)ctx + (uint32_t)p.T - 1u) / (uint32_t)p.T;
  return nb > (uint32_t)p.maxB ? p.maxB : (int32_t)nb;
}

__device__ __forceinline__ int32_t nblocks_of(const DevPool& p, int32_t sid) {
  return blocks_of_context(p, p.sess[sid].ctx_tokens);
}

// Exclusive scan over the block of NT threads; *total receives the sum.
template <int NT>
__device__ long long block_excl_scan(long long v, long long* total) {
  static_assert(NT % 32 == 0 && NT <= 1024, "block size");
  __shared__ long long warp_sums[NT / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[wid] = x;
  __syncthreads();
  if (wid == 0) {
    long long w = lane < NT / 32 ? warp_sums[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      long long y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < NT / 32) warp_sums[lane] = w;
  }
  __syncthreads();
  long long before = wid > 0 ? warp_sums[wid - 1] : 0;
  *total = warp_sums[NT / 32 - 1];
  __syncthreads();
  return before + x - v;
}

// Inclusive tiers: the host slot holding victim x's clean copy, or -1.
__device__ __forceinline__ int32_t clean_copy_of(const DevPool& p, const lv_victim& x) {
  if (!p.incl || x.sid < 0 || x.sid >= p.S || x.blk < 0 || x.blk >= p.maxB) return -1;
  return p.shadow[(size_t)x.sid * p.maxB + x.blk];
}

// ---------------------------------------------------------------- counts
// p.cnt[s] holds session s's blocks in HBM (x) and in the host tier (y): what a scan of its
// table row for entries >= 0 and <= -2 would count.  Every kernel that writes a table entry
// keeps it (import, remap, the exchange's plan, append), so that a decision reads S counts
// instead of S table rows.
__device__ __forceinline__ int2 tier_of(int32_t e) { return make_int2(e >= 0 ? 1 : 0, e <= -2 ? 1 : 0); }

// Both counts change by one 64-bit addition of dd * 2^32 + dh (a negative dh borrows from the
// upper half what the sum gives back).
__device__ __forceinline__ void add_counts(unsigned long long* cnt, int dh, int dd) {
  atomicAdd(cnt, ((unsigned long long)(unsigned)dd << 32) + (unsigned long long)(long long)dh);
}
__device__ __forceinline__ unsigned long long* counts_of(const DevPool& p, int32_t s) {
  return reinterpret_cast<unsigned long long*>(&p.cnt[s]);
}

// Adds (dh, dd) to the counts of session s, for the whole warp at once: lanes that share the
// first adding lane's session add through one reduction, the others by themselves.
// All 32 lanes must call it; a lane with nothing to add passes zeros.  cnt: where this lane
// adds, [S] words.
__device__ __forceinline__ void warp_count(unsigned long long* cnt, int32_t s, int dh, int dd) {
  const unsigned act = __ballot_sync(0xffffffffu, dh != 0 || dd != 0);
  if (!act) return;
  const int lead = __ffs(act) - 1;
  const int32_t s0 = __shfl_sync(0xffffffffu, s, lead);
  const bool adds = act >> (threadIdx.x & 31) & 1u, mine = adds && s == s0;
  const int h = __reduce_add_sync(0xffffffffu, mine ? dh : 0);
  const int d = __reduce_add_sync(0xffffffffu, mine ? dd : 0);
  if ((int)(threadIdx.x & 31) == lead) {
    add_counts(cnt + s0, h, d);
  } else if (adds && !mine) {
    add_counts(cnt + s, dh, dd);
  }
}

// The same for the E changes of each lane, v[j] = dd * 2^16 + dh for session s[j]: where the
// warp's sessions are all one, through one reduction.
template <int E>
__device__ __forceinline__ void warp_counts(unsigned long long* cnt, const int32_t* s, const int* v) {
  const int32_t s0 = __shfl_sync(0xffffffffu, s[0], 0);
  bool one = true;
  int sum = 0;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    one = one && (v[j] == 0 || s[j] == s0);
    sum += v[j];
  }
  if (__all_sync(0xffffffffu, one)) {
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((threadIdx.x & 31) == 0 && sum) add_counts(cnt + s0, (int)(int16_t)sum, (sum - (int)(int16_t)sum) >> 16);
    return;
  }
#pragma unroll
  for (int j = 0; j < E; ++j) warp_count(cnt, s[j], (int)(int16_t)v[j], (v[j] - (int)(int16_t)v[j]) >> 16);
}

// ---------------------------------------------------------------- import
__device__ __forceinline__ int32_t import_block(const DevPool& p, const int32_t* __restrict__ placement,
                                                const int32_t* __restrict__ ctx, long long idx, int32_t s,
                                                int32_t b);

// One thread per table entry; whole warps stay in the loop so that they can add up counts.
__global__ void k_import(DevPool p, const int32_t* __restrict__ placement,
                         const int32_t* __restrict__ ctx) {
  const long long total = (long long)p.S * p.maxB;
  int in_hbm = 0, in_host = 0;
  for (long long base = blockIdx.x * (long long)blockDim.x; base < total;
       base += (long long)gridDim.x * blockDim.x) {
    const long long idx = base + threadIdx.x;
    int32_t s = 0, e = -1;
    if (idx < total) {
      s = (int32_t)(idx / p.maxB);
      e = import_block(p, placement, ctx, idx, s, (int32_t)(idx % p.maxB));
    }
    const int2 t = tier_of(e);
    warp_count(counts_of(p, 0), s, t.x, t.y);
    in_hbm += t.x;
    in_host += t.y;
  }
  // the allocation counts, once per warp (a million blocks counted one by one queue on two words)
  in_hbm = __reduce_add_sync(0xffffffffu, in_hbm);
  in_host = __reduce_add_sync(0xffffffffu, in_host);
  if ((threadIdx.x & 31) == 0) {
    if (in_hbm) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HBM_ALLOC]), (unsigned long long)in_hbm);
    if (in_host) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HOST_ALLOC]), (unsigned long long)in_host);
  }
}

// The table entry that block b of session s gets (-1: none, or refused).
__device__ __forceinline__ int32_t import_block(const DevPool& p, const int32_t* __restrict__ placement,
                                                const int32_t* __restrict__ ctx, long long idx, int32_t s,
                                                int32_t b) {
  const long long c = ctx[s];
  long long nb = (c + p.T - 1) / p.T;
  if (b == 0) {
    if (c < 0 || nb > p.maxB) {
      set_error(p.ctl, LV_ERR_BOUNDS, s);
    }
    p.sess[s].ctx_tokens = (c < 0 || nb > p.maxB) ? 0 : (int32_t)c;
  }
  if (c < 0 || nb > p.maxB) nb = 0;
  const int32_t e = placement[idx];
  p.table[idx] = -1;
  p.mark[idx] = 0;
  p.shadow[idx] = -1;
  if (b >= nb) {
    if (e != -1) set_error(p.ctl, LV_ERR_BOUNDS, idx);
    return -1;
  }
  const uint32_t key = owner_key(s, b);
  if (e >= 0) {
    if (e >= p.hbm_pages) { set_error(p.ctl, LV_ERR_BOUNDS, idx); return -1; }
    if (atomicCAS(&p.own_hbm[e], kOwnerNone, key) != kOwnerNone) {
      set_error(p.ctl, LV_ERR_DOUBLE_MAP, idx);
      return -1;
    }
    atomicOr(&p.bits_hbm[e >> 5], 1u << (e & 31));
  } else if (e <= -2) {
    const long long h = -(long long)e - 2;
    if (h >= p.host_pages) { set_error(p.ctl, LV_ERR_BOUNDS, idx); return -1; }
    if (atomicCAS(&p.own_host[h], kOwnerNone, key) != kOwnerNone) {
      set_error(p.ctl, LV_ERR_DOUBLE_MAP, idx);
      return -1;
    }
    atomicOr(&p.bits_host[h >> 5], 1u << (h & 31));
  } else {
    set_error(p.ctl, LV_ERR_BOUNDS, idx);   // a block inside the context with no location
    return -1;
  }
  p.table[idx] = e;
  return e;
}

__global__ void k_check_budget(DevPool p) {
  if (p.ctl[C_HBM_ALLOC] > p.budget) set_error(p.ctl, LV_ERR_BUDGET, p.ctl[C_HBM_ALLOC]);
}

// -------------------------------------------------------------- sessions
__global__ void k_session_set(DevPool p, const lv_session_state* __restrict__ in, int32_t first,
                              int32_t n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  lv_session_state st = in[i];
  st.ctx_tokens = p.sess[first + i].ctx_tokens;   // owned by import / append
  p.sess[first + i] = st;
}

// One monitor event applied to a session's state (Section 3 signals; Section
// 5.1 reply interval and immediate reuse; Section 5.2 protection).
__device__ __forceinline__ void apply_event(const DevPool& p, lv_session_state& st, const lv_event& x) {
  switch (x.kind) {
    case LV_EV_TURN_BEGIN:
      st.flags = (st.flags | LV_RUNNING) & ~LV_IMMEDIATE;
      st.protect_until_us = 0;
      st.last_use_us = x.t_us;
      break;
    case LV_EV_TURN_END:
      st.last_use_us = x.t_us;
      st.flags &= ~(LV_RUNNING | LV_DONE_VALID);
      st.gen_us = x.a;
      st.play_us = 0;
      st.reply_tokens = x.b;
      if (st.gen_us > 0) {
        st.flags |= LV_RESP_OPEN;
      } else {
        st.flags = (st.flags & ~LV_RESP_OPEN) | LV_DONE_VALID;
        st.t_done_us = x.t_us;
      }
      break;
    case LV_EV_PLAYBACK:
      if (st.flags & LV_RESP_OPEN) {
        const long long np = st.play_us + x.a;
        st.play_us = np < st.gen_us ? np : st.gen_us;
        if (st.play_us >= st.gen_us) {
          st.flags = (st.flags & ~LV_RESP_OPEN) | LV_DONE_VALID;
          st.t_done_us = x.t_us;
        }
      }
      break;
    case LV_EV_SPEECH_START:
      st.flags |= LV_IMMEDIATE;
      break;
    case LV_EV_BARGE_IN:
      st.gen_us = st.play_us;
      st.flags = (st.flags | LV_IMMEDIATE) & ~(LV_RESP_OPEN | LV_DONE_VALID);
      break;
    case LV_EV_SPEECH_STOP:
      if (st.flags & LV_DONE_VALID) {
        long long xs = x.t_us - st.t_done_us;
        if (xs < 0) xs = 0;
        st.reply_ema_us = st.reply_n == 0 ? xs : (3 * st.reply_ema_us + xs) / 4;
        if (st.reply_n < 0x7fffffff) st.reply_n += 1;
      }
      st.flags &= ~(LV_IMMEDIATE | LV_DONE_VALID);
      break;
    case LV_EV_PRELOADED:
      st.protect_until_us = x.t_us + p.protect_us;
      break;
    case LV_EV_UNPROTECT:
      st.protect_until_us = 0;
      break;
    default:
      break;   // reported by the caller
  }
}

// One thread per session applies, in order, the events addressed to it.
constexpr int kEventThreads = 128;
constexpr int kEventChunk = 512;   // events staged in shared memory at a time (16 KiB)

// One thread per session.  The CTA stages the event list in shared memory, a
// chunk at a time (coalesced loads, each event read once per CTA), and every
// thread applies, in list order, the events of its own session.  CTA 0 checks
// every event's kind and session and counts them.
__global__ void __launch_bounds__(kEventThreads)
k_events(DevPool p, const lv_event* __restrict__ ev, long long n) {
  pdl_entry();
  __shared__ lv_event chunk[kEventChunk];
  const int s = blockIdx.x * kEventThreads + threadIdx.x;
  lv_session_state st;
  if (s < p.S) st = p.sess[s];
  bool touched = false;
  for (long long c0 = 0; c0 < n; c0 += kEventChunk) {
    const int m = (int)(n - c0 < kEventChunk ? n - c0 : kEventChunk);
    __syncthreads();   // the previous chunk is no longer read
    for (int e = threadIdx.x; e < m; e += kEventThreads) {
      const lv_event x = ev[c0 + e];
      chunk[e] = x;
      if (blockIdx.x == 0 && (x.kind < LV_EV_TURN_BEGIN || x.kind > LV_EV_UNPROTECT || x.sid < 0 ||
                              x.sid >= p.S))
        set_error(p.ctl, LV_ERR_BOUNDS, c0 + e);
    }
    __syncthreads();
    if (s < p.S) {
      for (int e = 0; e < m; ++e) {
        if (chunk[e].sid != s) continue;
        touched = true;
        apply_event(p, st, chunk[e]);
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_EVENTS]), (unsigned long long)n);
  if (s < p.S && touched) p.sess[s] = st;
}

// --------------------------------------------------------------- ranking
// Order key of a session, 0 when it is not a candidate.  Larger keys are
// evicted first: bit 63 = normal tier, bits 31..62 = T_next (Eq. 4), bits
// 0..30 = 2^31-1-sid so that equal T_next rank by ascending session id.
__device__ __forceinline__ unsigned long long session_key(const DevPool& p, const lv_session_state& st,
                                                          int32_t s, long long now_us, bool fallback) {
  if (p.policy == LV_POLICY_LRU) {
    // least recently used first: every non-running session is a candidate
    if (st.flags & LV_RUNNING) return 0ull;
    long long t = st.last_use_us;
    if (t < 0) t = 0;
    if (t > kKeyMax) t = kKeyMax;
    return (1ull << 63) | ((unsigned long long)(kKeyMax - t) << 31) |
           (unsigned long long)(0x7fffffff - s);
  }
  const bool normal = !(st.flags & (LV_RUNNING | LV_IMMEDIATE)) && !(now_us < st.protect_until_us);
  if (!normal && !(fallback && !(st.flags & LV_RUNNING))) return 0ull;
  long long t_play;
  if (p.tplay == LV_PLAY_PLAYBACK) {
    const long long d = st.gen_us - st.play_us;            // remaining playback horizon
    t_play = d > 0 ? d : 0;
  } else {
    // progress counters: a longer unfinished reply means later reuse
    if (!(st.flags & LV_RESP_OPEN) || st.reply_tokens <= 0) t_play = 0;
    else if (st.reply_tokens > kKeyMax / p.unit_us) t_play = kKeyMax;
    else t_play = st.reply_tokens * p.unit_us;
  }
  long long t_reply = st.reply_n > 0 ? st.reply_ema_us : p.reply_prior_us;
  if (t_reply < 0) t_reply = 0;
  if (t_play > kKeyMax) t_play = kKeyMax;
  if (t_reply > kKeyMax) t_reply = kKeyMax;
  long long t_next = t_play + t_reply;
  if (t_next > kKeyMax) t_next = kKeyMax;
  return ((normal ? 1ull : 0ull) << 63) | ((unsigned long long)t_next << 31) |
         (unsigned long long)(0x7fffffff - s);
}

constexpr int kCensusThreads = 256;
// Up to this many sessions every emit CTA finds its session's place by reading all
// S keys itself (S^2 key reads, from L2); above it, k_rank_prefix computes every place
// once, between the census and the emission (S^2 key comparisons, but S^2 / 256 key
// reads), at the cost of one more launch in the chain.
#ifndef LV_EMIT_SCAN_MAX
#define LV_EMIT_SCAN_MAX 1024
#endif
constexpr int kEmitScanMax = LV_EMIT_SCAN_MAX;

// Every session's key and its count of HBM-resident blocks.  kRow: threads of a row's
// session -- a CTA, or a warp (eight sessions a CTA) where rows are short: 4096 rows of 256
// words took 8.8 us with a CTA each.
template <int kRow>
__global__ void __launch_bounds__(kCensusThreads)
k_rank_census(DevPool p, long long now_us, bool fallback) {
  pdl_wait();
  const int32_t s = (blockIdx.x * kCensusThreads + threadIdx.x) / kRow;
  const int t = threadIdx.x % kRow;
  unsigned long long key = 0ull;
  int c = 0;
  if (s < p.S) {
    key = session_key(p, p.sess[s], s, now_us, fallback);
    if (key != 0ull) {
      const int32_t nb = nblocks_of(p, s);
      const int32_t* row = p.table + (size_t)s * p.maxB;
#pragma unroll 4
      for (int32_t b = t; b < nb; b += kRow) c += row[b] >= 0 ? 1 : 0;
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (kRow > 32) {
    __shared__ int part[kCensusThreads / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
    __syncthreads();
    c = 0;
    if (t == 0)
      for (int w = 0; w < kCensusThreads / 32; ++w) c += part[w];
  }
  if (t == 0 && s < p.S) {
    p.skey[s] = key;
    p.scount[s] = c;
    if (p.S > kEmitScanMax) {       // k_rank_prefix accumulates into these
      p.sbefore[s] = 0;
      if (s == 0) p.ctl[C_RANK_TOTAL] = 0;
    }
  }
  pdl_trigger();
}

constexpr int kPrefixTile = 128;    // sessions placed by one CTA (one per thread)
constexpr int kPrefixChunk = 256;   // keys staged by one CTA in shared memory

// The place of every candidate session in the victim order, for S > kEmitScanMax:
// sbefore[s] = the resident blocks of the candidate sessions with a larger key
// (keys are distinct).  CTA (x, y) compares the sessions of tile x with the keys
// of chunk y, read once into shared memory (every thread reads the same key at
// once: a broadcast), and adds its partial sums; the CTAs of tile 0 also add up
// all candidates' blocks into C_RANK_TOTAL.  The census zeroed both.
__global__ void __launch_bounds__(kPrefixTile)
k_rank_prefix(DevPool p) {
  pdl_wait();   // the census is complete and visible
  __shared__ unsigned long long kc[kPrefixChunk];
  __shared__ int32_t cc[kPrefixChunk];
  __shared__ long long part[kPrefixTile / 32];
  const int32_t j0 = blockIdx.y * kPrefixChunk;
  const int32_t nj = min(kPrefixChunk, p.S - j0);
  for (int32_t j = threadIdx.x; j < nj; j += kPrefixTile) {
    const unsigned long long kj = p.skey[j0 + j];
    kc[j] = kj;
    cc[j] = kj ? p.scount[j0 + j] : 0;
  }
  __syncthreads();
  const int32_t s = blockIdx.x * kPrefixTile + threadIdx.x;
  const unsigned long long key = s < p.S ? p.skey[s] : 0ull;
  if (key != 0ull) {
    long long before = 0;
#pragma unroll 8
    for (int32_t j = 0; j < nj; ++j) before += kc[j] > key ? cc[j] : 0;
    if (before) atomicAdd(reinterpret_cast<unsigned long long*>(&p.sbefore[s]), (unsigned long long)before);
  }
  if (blockIdx.x == 0) {
    long long t = 0;
    for (int32_t j = threadIdx.x; j < nj; j += kPrefixTile) t += cc[j];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      long long all = 0;
      for (int w = 0; w < kPrefixTile / 32; ++w) all += part[w];
      if (all) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_RANK_TOTAL]), (unsigned long long)all);
    }
  }
  pdl_trigger();
}

constexpr int kEmitThreads = 256;

// One CTA per session.  The victim order takes the sessions by decreasing key
// (keys are distinct: each holds its session id), so a session's first
// position in the order is the number of resident blocks of the sessions with
// a larger key; the CTA sums those counts over the census, then writes its
// own resident blocks, suffix first (or ascending), while positions stay below
// the selection count min(k, all resident candidates).  CTA 0 publishes the
// count and the counters.
__global__ void __launch_bounds__(kEmitThreads)
k_rank_emit(DevPool p, long long k, bool fallback, long long* count_dev,
            lv_victim* __restrict__ out) {
  pdl_wait();   // the census (and the places) are complete and visible
  const int32_t sid = blockIdx.x;
  const unsigned long long key = p.skey[sid];
  if (key == 0ull && sid != 0) return;
  long long off, total;
  if (p.S > kEmitScanMax) {      // placed by k_rank_prefix
    off = key ? p.sbefore[sid] : 0;
    total = p.ctl[C_RANK_TOTAL];
  } else {
    long long before = 0, all = 0;
    for (int32_t j = threadIdx.x; j < p.S; j += kEmitThreads) {
      const unsigned long long kj = p.skey[j];
      const long long cj = kj ? p.scount[j] : 0;
      all += cj;
      before += kj > key ? cj : 0;
    }
    block_excl_scan<kEmitThreads>(before, &off);
    block_excl_scan<kEmitThreads>(all, &total);
  }
  const long long n_out = k < total ? k : total;
  if (sid == 0 && threadIdx.x == 0) {
    p.ctl[C_SEL_COUNT] = n_out;
    p.ctl[C_SEL_TOTAL] = total;
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_SELECTS]), 1ull);
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_VICTIMS]), (unsigned long long)n_out);
    if (k != INT64_MAX && total < k)
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_SHORTFALLS]), 1ull);
    if (fallback) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_FALLBACK]), 1ull);
    if (count_dev) *count_dev = n_out;
  }
  if (key == 0ull || off >= n_out) return;
  const int32_t nb = nblocks_of(p, sid);
  const int32_t* row = p.table + (size_t)sid * p.maxB;
  const bool suffix = p.within == LV_SUFFIX_FIRST;
  long long run = 0;
  for (int32_t q0 = 0; q0 < nb && off + run < n_out; q0 += kEmitThreads) {
    const int32_t q = q0 + threadIdx.x;
    const int32_t b = suffix ? nb - 1 - q : q;
    int32_t e = -1;
    if (q < nb) e = row[b];
    const long long flag = e >= 0 ? 1 : 0;
    long long chunk;
    const long long pos = off + run + block_excl_scan<kEmitThreads>(flag, &chunk);
    if (flag && pos < n_out) out[pos] = lv_victim{sid, b, e};
    run += chunk;
  }
  pdl_trigger();
}

// ------------------------------------------------------------------ copy
constexpr int kCopyThreads = 256;
constexpr int kCopyUnroll = 4;

// Copies one sub-page: 16-byte vectors, kCopyUnroll loads in flight per thread.
__device__ __forceinline__ void copy_subpage(const int4* __restrict__ src, int4* __restrict__ dst,
                                             int nvec) {
  for (int base = threadIdx.x; base < nvec; base += kCopyThreads * kCopyUnroll) {
    int4 r[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
      const int q = base + u * kCopyThreads;
      if (q < nvec) r[u] = src[q];
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
      const int q = base + u * kCopyThreads;
      if (q < nvec) dst[q] = r[u];
    }
  }
}

// Unit u = (victim i, sub-page j): hbm_kv[j][page_i] -> host[slot_i][j].
__global__ void __launch_bounds__(kCopyThreads)
k_swap_out(DevPool p, const lv_victim* __restrict__ v, const int32_t* __restrict__ slots,
           long long n, lv_remap_entry* __restrict__ commit) {
  pdl_wait();
  const long long units = n * p.J;
  const int nvec = (int)(p.P >> 4);
  for (long long u = blockIdx.x; u < units; u += gridDim.x) {
    const long long i = u / p.J;
    const int j = (int)(u % p.J);
    const lv_victim x = v[i];
    const int32_t slot = slots[i];
    if (slot < 0) continue;                          // reservation failed (error already set)
    bool ok = x.sid >= 0 && x.sid < p.S && x.blk >= 0 && x.page >= 0 && x.page < p.hbm_pages &&
              slot < p.host_pages;
    ok = ok && x.blk < nblocks_of(p, x.sid);
    ok = ok && p.table[(size_t)x.sid * p.maxB + x.blk] == x.page &&
         p.own_hbm[x.page] == owner_key(x.sid, x.blk);
    const bool clean = ok && clean_copy_of(p, x) == slot;   // its clean copy: nothing to move
    if (j == 0 && threadIdx.x == 0) {
      if (!ok) set_error(p.ctl, LV_ERR_STATE, i);
      else atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PAGES_OUT]), 1ull);
      if (clean) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN_OUT]), 1ull);
      if (commit) commit[i] = lv_remap_entry{x.sid, x.blk, ok ? -(slot + 2) : -1};
    }
    if (!ok || clean) continue;
    const int4* src = reinterpret_cast<const int4*>(p.kv[j] + (size_t)x.page * p.P);
    int4* dst = reinterpret_cast<int4*>(p.host + ((size_t)slot * p.J + j) * p.P);
    copy_subpage(src, dst, nvec);
  }
  pdl_trigger();
}

// Unit u = (block i, sub-page j): host[slot(blk_i)][j] -> hbm_kv[j][page_i].
__global__ void __launch_bounds__(kCopyThreads)
k_swap_in(DevPool p, int32_t sid, const int32_t* __restrict__ blks,
          const int32_t* __restrict__ pages, long long n, lv_remap_entry* __restrict__ commit) {
  pdl_wait();
  const long long units = n * p.J;
  const int nvec = (int)(p.P >> 4);
  const bool sid_ok = sid >= 0 && sid < p.S;
  const int32_t nb = sid_ok ? nblocks_of(p, sid) : 0;
  for (long long u = blockIdx.x; u < units; u += gridDim.x) {
    const long long i = u / p.J;
    const int j = (int)(u % p.J);
    const int32_t blk = blks[i];
    const int32_t page = pages[i];
    if (page < 0) continue;                          // reservation failed (error already set)
    bool ok = sid_ok && blk >= 0 && blk < nb && page < p.hbm_pages;
    long long slot = -1;
    if (ok) {
      const int32_t e = p.table[(size_t)sid * p.maxB + blk];
      slot = -(long long)e - 2;
      ok = e <= -2 && slot < p.host_pages && p.own_host[slot] == owner_key(sid, blk);
    }
    if (j == 0 && threadIdx.x == 0) {
      if (!ok) set_error(p.ctl, sid_ok ? LV_ERR_STATE : LV_ERR_BOUNDS, i);
      else atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PAGES_IN]), 1ull);
      if (commit) commit[i] = lv_remap_entry{sid, blk, ok ? page : -1};
    }
    if (!ok) continue;
    const int4* src = reinterpret_cast<const int4*>(p.host + ((size_t)slot * p.J + j) * p.P);
    int4* dst = reinterpret_cast<int4*>(p.kv[j] + (size_t)page * p.P);
    copy_subpage(src, dst, nvec);
  }
  pdl_trigger();
}

// ------------------------------------------------------- one-CTA decisions
// The decision kernels (k_step, k_exchange_plan, k_append) run as one CTA: what they do is a
// chain of dependent reads of a few hundred table words, so their time is the number of
// links, each a trip to L2 or a barrier, and not the work in them.  Lists of up to
// kStepItems entries and the allocation bitmaps are therefore kept in shared memory, reads
// that depend on nothing are issued at the start, and a scan costs one barrier.  The other
// cost is scattered access: a warp's 32 stores or reductions to 32 places keep the SM's
// memory pipe busy for 32 cycles (measured: 31 a warp), and whatever comes next, a barrier's
// shared-memory word too, queues behind them.  So the bitmaps change in shared memory alone
// and only the words that differ at the end are written, a page that is freed and taken
// again in one step gets one owner word, and the session table is read in whole lines.
// The third cost is instructions: a jump to a line outside the small instruction buffer costs
// about 110 cycles, warm or not (measured with 160 taken branches over short blocks), while
// straight code is fetched ahead.  So these kernels do not unroll loops that mostly run once,
// and what is rare is marked and laid out of line.
#define LV_RARE(x) __builtin_expect(!!(x), 0)
#define LV_MOSTLY(x) __builtin_expect(!!(x), 1)
constexpr int kStepThreads = 512;
constexpr int kStepWarps = kStepThreads / 32;
constexpr int kStepItems = 1024;   // victims, and loads, whose lists stay in shared memory

// Prefix sums over the CTA with one barrier each: consecutive calls alternate between two
// sets of warp totals, so a set is written again only after the barrier of the call between.
struct BlockScan {
  int* ws;   // [2][kStepWarps] in shared memory
  int ph;
  __device__ int sum(int v, int* total) {          // exclusive prefix of v
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    return warps(x, lane, wid, total) + x - v;
  }
  __device__ int rank(bool flag, int* total) {      // flagged threads before this one
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    return warps(__popc(m & (0xffffffffu >> (31 - lane))), lane, wid, total) +
           __popc(m & ((1u << lane) - 1u));
  }

 private:
  // x: the warp's inclusive sums (lane 31 holds its total); returns the total of the warps before
  __device__ int warps(int x, int lane, int wid, int* total) {
    int* w = ws + ph * kStepWarps;
    ph ^= 1;
    if (lane == 31) w[wid] = x;
    __syncthreads();
    int y = lane < kStepWarps ? w[lane] : 0;
#pragma unroll
    for (int o = 1; o < kStepWarps; o <<= 1) {
      const int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    *total = __shfl_sync(0xffffffffu, y, kStepWarps - 1);
    const int before = __shfl_sync(0xffffffffu, y, wid > 0 ? wid - 1 : 0);
    return wid > 0 ? before : 0;
  }
};

// One tier's allocation bitmap: the pool's words, and what this kernel works on: a copy in
// shared memory (with the words as they were beside it, for bits_back), or where that does
// not fit the pool's words themselves.
// Which pages are free is read off these words alone, not off the tier's allocation count in
// p.ctl: a free on another stream may run meanwhile, and it clears a bit and lowers that count
// one after the other, so the two read apart may disagree, and two threads may read different
// counts.
struct TierBits {
  uint32_t* gl;
  uint32_t* cur;
  uint32_t* old;
  long long nbits;
  int taken;       // set bits among the words that this thread read
  __device__ uint32_t word(int w) const { return cur != gl ? cur[w] : __ldcg(&gl[w]); }
  __device__ bool has(int32_t i) const { return word(i >> 5) >> (i & 31) & 1u; }
  __device__ void set(int w, uint32_t m) const {           // a word only this thread changes now
    if (cur != gl) cur[w] |= m;
    else atomicOr(&gl[w], m);
  }
  __device__ void clear(int32_t i) const { atomicAnd(&cur[i >> 5], ~(1u << (i & 31))); }
};

// Reads a bitmap of W words into shared memory at `copy` (2 W words; null: used in place).
// me: the thread's place in a permutation of the CTA's threads, of which the first copy the
// first words.
__device__ __forceinline__ TierBits bits_copy(uint32_t* gl, long long nbits, uint32_t* copy, int me) {
  const int W = (int)((nbits + 31) >> 5);
  TierBits t{gl, gl, gl, nbits, 0};
  if (LV_RARE(!copy)) {
#pragma unroll 8
    for (int w = threadIdx.x; w < W; w += kStepThreads) t.taken += __popc(gl[w]);
    return t;
  }
  t.cur = copy;
  t.old = copy + W;
#pragma unroll 1
  for (int w = me; w < W; w += kStepThreads) {
    const uint32_t x = gl[w];
    copy[w] = copy[W + w] = x;
    t.taken += __popc(x);
  }
  return t;
}

// Writes the words that changed, as reductions of the bits that changed: a free of other
// pages on another stream may run meanwhile.  After a barrier.
__device__ __forceinline__ void bits_back(const TierBits& t) {
  if (t.cur == t.gl) return;
  const int W = (int)((t.nbits + 31) >> 5);
#pragma unroll 1
  for (int w = threadIdx.x; w < W; w += kStepThreads) {
    const uint32_t now = t.cur[w], was = t.old[w];
    if (now & ~was) atomicOr(&t.gl[w], now & ~was);
    if (was & ~now) atomicAnd(&t.gl[w], ~(was & ~now));
  }
}

// Position of the k-th set bit of f (k counted from 0, below popc(f)).
__device__ __forceinline__ int nth_bit(uint32_t f, int k) {
  int at = 0;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) {
    const int c = __popc(f & ((1u << w) - 1u));
    if (k >= c) {
      k -= c;
      at += w;
      f >>= w;
    }
  }
  return at;
}

// The n lowest free bits, ascending, into out[0..n); sets them.  Each thread owns a
// contiguous run of words and counts its free bits; then thread i finds the i-th one by
// binary search among the threads' counts (in `base`), so that a tier with whole free words
// takes as long as one with a free bit here and there.  Without a copy of the bitmap each
// thread writes its own words' bits, and no more than it counted: a free on another stream
// may add bits meanwhile.  Returns false, with nothing changed, when n and `spare` more are
// not free (the searches below end only because n are); other threads may read out when it
// returns.
__device__ bool take_lowest(const TierBits& t, int n, long long spare, int32_t* out, BlockScan& scan, int* base) {
  const int W = (int)((t.nbits + 31) >> 5);
  const int per = (W + kStepThreads - 1) / kStepThreads;
  const int w0 = threadIdx.x * per;
  const uint32_t last = (t.nbits & 31) ? (1u << (t.nbits & 31)) - 1u : 0xffffffffu;
  auto free_of = [&](int w) { return w < W ? ~t.word(w) & (w == W - 1 ? last : 0xffffffffu) : 0u; };
  int cnt = 0;
#pragma unroll 1
  for (int i = 0; i < per; ++i) cnt += __popc(free_of(w0 + i));
  int total;
  int r = scan.sum(cnt, &total);
  const bool enough = total - spare >= n;
  if (!enough) n = 0;
  if (LV_RARE(t.cur == t.gl)) {
    const int r_end = min(n, r + cnt);
#pragma unroll 1
    for (int i = 0; i < per && r < r_end; ++i) {
      uint32_t f = free_of(w0 + i), take = 0;
#pragma unroll 1
      while (f && r < r_end) {
        const int b = __ffs(f) - 1;
        f &= f - 1;
        out[r++] = (w0 + i) * 32 + b;
        take |= 1u << b;
      }
      if (take) t.set(w0 + i, take);
    }
    __syncthreads();
    return enough;
  }
  base[threadIdx.x] = r;
  __syncthreads();
#pragma unroll 1
  for (int i = threadIdx.x; i < n; i += kStepThreads) {
    int o = 0;                 // the last thread whose run starts at or before the i-th bit
#pragma unroll
    for (int step = kStepThreads / 2; step > 0; step >>= 1)
      if (base[o + step] <= i) o += step;
    int left = i - base[o], w = o * per;
    uint32_t f = free_of(w);
#pragma unroll 1
    for (int c = __popc(f); left >= c; c = __popc(f)) {
      left -= c;
      f = free_of(++w);
    }
    out[i] = w * 32 + nth_bit(f, left);
  }
  __syncthreads();             // every thread has read the words
#pragma unroll 1
  for (int i = 0; i < per && r < n; ++i) {
    const uint32_t f = free_of(w0 + i);
    const int c = __popc(f);
    const uint32_t take = c <= n - r ? f : f & ((1u << nth_bit(f, n - r)) - 1u);
    if (take) t.set(w0 + i, take);
    r += c;
  }
  return enough;
}

// Spreads the nd slots out[0..nd) so that the r-th victim without a clean copy has the r-th of
// them and every other victim its copy.  In place, from the last chunk to the first: a
// victim's rank among those without a copy is at most its index, so each read position
// still holds its compact value when it is read.
__device__ void spread_slots(const DevPool& p, const lv_victim* v, long long n, int nd, int32_t* out,
                             BlockScan& scan) {
  long long after = 0;   // victims without a copy in the chunks already spread
#pragma unroll 1
  for (long long c = (n + kStepThreads - 1) / kStepThreads - 1; c >= 0; --c) {
    const long long i = c * kStepThreads + threadIdx.x;
    const int32_t cp = i < n ? clean_copy_of(p, v[i]) : 0;
    int chunk;
    const int excl = scan.rank(cp < 0, &chunk);
    const int32_t val = cp < 0 ? out[nd - after - chunk + excl] : cp;
    __syncthreads();
    if (i < n) out[i] = val;
    __syncthreads();
    after += chunk;
  }
}

// ------------------------------------------------------------ allocation
// Reserves n pages or slots, the lowest free ones (one CTA).  v: a swap-out's victims under
// inclusive tiers -- those with a clean copy take it, only the others count against the
// host tier.
__global__ void __launch_bounds__(kStepThreads, 1)
k_alloc(DevPool p, bool in_hbm, const lv_victim* v, long long n, int32_t* out, bool injected_fail,
        int copy_bits) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ int ws[2 * kStepWarps];
  __shared__ int base[kStepThreads];
  pdl_entry();
  BlockScan scan{ws, 0};
  uint32_t* copy = copy_bits ? reinterpret_cast<uint32_t*>(dyn) : nullptr;
  const TierBits t = in_hbm ? bits_copy(p.bits_hbm, p.hbm_pages, copy, threadIdx.x)
                            : bits_copy(p.bits_host, p.host_pages, copy, threadIdx.x);
  int nd = (int)n;
  if (LV_RARE(v != nullptr)) {
    int cnt = 0;
#pragma unroll 1
    for (long long i = threadIdx.x; i < n; i += kStepThreads) cnt += clean_copy_of(p, v[i]) < 0 ? 1 : 0;
    scan.sum(cnt, &nd);
  }
  __syncthreads();             // the bitmap's copy is complete
  const long long spare = in_hbm ? p.hbm_pages - p.budget : 0;
  if (LV_RARE(injected_fail || (nd > 0 && !take_lowest(t, nd, spare, out, scan, base)))) {
    if (threadIdx.x == 0) set_error(p.ctl, in_hbm ? LV_ERR_NO_HBM : LV_ERR_NO_HOST, nd);
#pragma unroll 1
    for (long long i = threadIdx.x; i < n; i += kStepThreads) out[i] = -1;
    return;
  }
  uint32_t* own = in_hbm ? p.own_hbm : p.own_host;
#pragma unroll 1
  for (int i = threadIdx.x; i < nd; i += kStepThreads) own[out[i]] = kOwnerReserved;
  __syncthreads();
  if (LV_RARE(nd < n)) spread_slots(p, v, n, nd, out, scan);
  bits_back(t);
  if (threadIdx.x == 0)
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[in_hbm ? C_HBM_ALLOC : C_HOST_ALLOC]), (unsigned long long)nd);
}

// -------------------------------------------------------------- exchange
// Evict n_out victims and load n_in host blocks of one session in a single
// stream-ordered step whose result equals swap-out, commit, swap-in, commit
// done one after the other.  plan_moves takes every metadata decision in that
// order -- validation, host slots (lowest free, victim order), out-commit, HBM
// pages (lowest free after the frees, list order), in-commit -- and emits copy
// tasks {out page, out slot, in slot, in page}.
// An incoming block that lands on a victim's old page shares that victim's
// task, so one thread reads the old bytes before it writes the new ones and
// both directions of the host link carry data at the same time.
constexpr unsigned long long kPairedBit = 1ull << 31;

// Words that a device-driven step leaves for the kernels after it.
enum ResWord : int {
  R_N_IN = 2,       // host blocks listed (for k_order_loads)
  R_N_TASKS = 6,
  R_SID = 9,        // lv_turn: the turn's session (-1 when the pick failed)
  R_CURSOR = 10     // the exchange copy's next unit (zeroed by the plan)
};

// What plan_moves works on.  v, slots, blks, gslot and pages may lie in shared memory
// (lists of up to kStepItems entries) or in global memory.
struct MovePlan {
  const lv_victim* v;
  int64_t n_out;
  int32_t sid;
  const int32_t* blks;
  const int32_t* gslot;     // the loads' host slots, or null: read from the table
  int64_t n_in;
  int32_t* slots;
  int32_t* pages;
  int32_t* slots_out;       // global results
  int32_t* pages_out;
  int4* tasks;
  long long* n_tasks;
  int32_t epoch;
  unsigned long long* page_tag;
};

// Shared memory of the one-CTA kernels.
struct StepLists {
  lv_victim v[kStepItems];
  int32_t slots[kStepItems], blks[kStepItems], gslot[kStepItems], pages[kStepItems], pair[kStepItems];
};
struct StepShared {
  int ws[2 * kStepWarps];
  unsigned long long best[2][kStepWarps];
  int2 sums[kStepWarps];
  int taken[kStepWarps];            // HBM pages allocated, by the warps that read their bits
  int2 pick[kStepWarps + 1];
  int sel_sid[12], sel_off[12];     // [kSelectRounds]
  uint32_t done[kStepItems / 32];   // victims that need no out task of their own
  int base[kStepThreads];
  union {
    StepLists l;
    // at the start, 32 sessions' states of each warp
    __align__(16) long long states[kStepWarps][32 * sizeof(lv_session_state) / 8];
  };
};

// Plans and commits m's moves; every thread of the CTA calls it.  kListed: the lists come
// from the caller and may be wrong or hold a block twice (checked, with the epoch marks);
// else they were just read from the tables, and checked there: bad_out and bad_in are a
// thread's first wrong victim and load, or -1.  Returns false, with nothing changed, the
// outputs -1 and no tasks, when an item is refused or a tier is too full.
// hbm_alloc: the HBM pages allocated as the kernel found them.
template <bool kListed>
__device__ bool plan_moves(const DevPool& p, const MovePlan& m, const TierBits& hbm, const TierBits& host,
                           long long hbm_alloc, long long bad_out, long long bad_in,
                           StepShared& sh, BlockScan& scan) {
  const long long n_out = m.n_out;
  long long n_in = m.n_in;
  const bool sid_ok = m.sid >= 0 && m.sid < p.S;
  const size_t row = sid_ok ? (size_t)m.sid * p.maxB : 0;
  const int32_t nb_in = kListed && sid_ok ? nblocks_of(p, m.sid) : 0;
  const bool few = n_out <= kStepItems;      // victims are tracked in shared memory
  static_assert(kStepItems / 32 <= kStepThreads, "one word of `done` per thread");
  if (few && threadIdx.x < kStepItems / 32) sh.done[threadIdx.x] = 0u;
  // validation: every victim is resident where it says, every incoming block is in the
  // host tier, and no block appears twice (victims and incoming blocks side by side: item
  // i < n_out is victim i, item n_out + i incoming block i)
  bool bad = false;
  int dirty = 0;             // victims without a clean copy: all of them unless the tiers are inclusive
  if (kListed) {
#pragma unroll 1
    for (long long it = threadIdx.x; it < n_out + n_in; it += kStepThreads) {
      bool ok;
      if (it < n_out) {
        const lv_victim x = m.v[it];
        ok = x.sid >= 0 && x.sid < p.S && x.blk >= 0 && x.page >= 0 && x.page < p.hbm_pages;
        ok = ok && x.blk < nblocks_of(p, x.sid);
        ok = ok && p.table[(size_t)x.sid * p.maxB + x.blk] == x.page &&
             p.own_hbm[x.page] == owner_key(x.sid, x.blk);
        ok = ok && atomicExch(&p.mark[(size_t)x.sid * p.maxB + x.blk], m.epoch) != m.epoch;
      } else {
        const int32_t b = m.blks[it - n_out];
        ok = sid_ok && b >= 0 && b < nb_in;
        if (ok) {
          const int32_t e = p.table[row + b];
          const long long h = -(long long)e - 2;
          ok = e <= -2 && h < p.host_pages && p.own_host[h] == owner_key(m.sid, b);
          ok = ok && atomicExch(&p.mark[row + b], m.epoch) != m.epoch;
        }
      }
      if (!ok) { set_error(p.ctl, sid_ok || it < n_out ? LV_ERR_STATE : LV_ERR_BOUNDS, it); bad = true; }
    }
  } else {
    if (LV_RARE(n_out > 0 && bad_out >= 0)) { set_error(p.ctl, LV_ERR_STATE, bad_out); bad = true; }
    if (LV_RARE(n_in > 0 && bad_in >= 0)) { set_error(p.ctl, LV_ERR_STATE, n_out + bad_in); bad = true; }
  }
  if (LV_RARE(p.incl))
#pragma unroll 1
    for (long long i = threadIdx.x; i < n_out; i += kStepThreads) dirty += clean_copy_of(p, m.v[i]) < 0 ? 1 : 0;
  bad = __syncthreads_or(bad);
  int n_dirty = (int)n_out;
  if (LV_RARE(p.incl)) scan.sum(dirty, &n_dirty);
  // capacity, as the sequential calls see it: host slots before any is freed,
  // HBM pages after the victims' pages are freed
  const bool no_hbm = hbm_alloc - n_out + n_in > p.budget;
  bool no_host = false;
  if (LV_RARE(no_hbm)) {
    int mine = 0, used;
#pragma unroll 1
    for (int w = threadIdx.x; w < (int)((p.host_pages + 31) >> 5); w += kStepThreads) mine += __popc(host.word(w));
    scan.sum(mine, &used);
    no_host = used + (long long)n_dirty > p.host_pages;
  } else if (LV_MOSTLY(n_dirty > 0 && !bad)) {
    // host slots for the victims: a clean copy, or the lowest free slots in victim order
    no_host = !take_lowest(host, n_dirty, 0, m.slots, scan, sh.base);
  }
  if (LV_RARE(bad || no_host || no_hbm)) {
    if (!bad && threadIdx.x == 0)
      set_error(p.ctl, no_host ? LV_ERR_NO_HOST : LV_ERR_NO_HBM, no_host ? (long long)n_dirty : n_in);
#pragma unroll 1
    for (long long i = threadIdx.x; i < n_out; i += kStepThreads) m.slots_out[i] = -1;
#pragma unroll 1
    for (long long i = threadIdx.x; i < n_in; i += kStepThreads) m.pages_out[i] = -1;
    if (threadIdx.x == 0) *m.n_tasks = 0;
    return false;
  }
  if (LV_RARE(n_dirty < n_out)) {
    __syncthreads();
    spread_slots(p, m.v, n_out, n_dirty, m.slots, scan);
  }
  // out-commit: victims now live in their slots, their pages are free.  A page that an
  // incoming block takes pairs that block's task with its victim's: found by looking the
  // victim's page up among the pages taken (ascending), or for longer lists through a tag
  // that the victim leaves in page_tag.  A clean victim has nothing to read and no pair.
  const bool look_up = few && n_in <= kStepItems;
  const unsigned long long tag = (unsigned long long)(uint32_t)m.epoch << 32;
#pragma unroll 1
  for (long long i0 = 0; i0 < n_out; i0 += kStepThreads) {
    const long long i = i0 + threadIdx.x;
    if (i < n_out) {
      const lv_victim x = m.v[i];
      const int32_t slot = m.slots[i];
      const size_t ti = (size_t)x.sid * p.maxB + x.blk;
      bool clean = false;
      if (LV_RARE(p.incl)) clean = p.shadow[ti] == slot;
      p.table[ti] = -(slot + 2);
      if (LV_RARE(clean)) p.shadow[ti] = -1;
      p.own_host[slot] = owner_key(x.sid, x.blk);
      hbm.clear(x.page);
      if (LV_RARE(clean && few)) atomicOr(&sh.done[i >> 5], 1u << (i & 31));
      if (LV_RARE(!clean && !look_up)) m.page_tag[x.page] = tag | (unsigned long long)i;
      if (LV_MOSTLY(m.slots_out != m.slots)) m.slots_out[i] = slot;
    }
    if (kListed) {
      const bool mine = i < n_out;
      warp_count(counts_of(p, 0), mine ? m.v[i].sid : 0, mine ? -1 : 0, mine ? 1 : 0);
    }
  }
  if (LV_MOSTLY(look_up))
#pragma unroll 1
    for (int i = threadIdx.x; i < n_in; i += kStepThreads) sh.l.pair[i] = -1;
  __syncthreads();
  // HBM pages for the incoming blocks
  if (n_in > 0) {
    // (too few only if a victim's page had no bit: then nothing is loaded)
    n_in = take_lowest(hbm, (int)n_in, 0, m.pages, scan, sh.base) ? n_in : 0;
    __syncthreads();
  }
  // a victim's page is now taken again, or free
  int paired = 0;
#pragma unroll 1
  for (long long i = threadIdx.x; i < n_out; i += kStepThreads) {
    const int32_t pg = m.v[i].page;
    if (LV_RARE(!hbm.has(pg))) {
      p.own_hbm[pg] = kOwnerNone;
    } else if (LV_MOSTLY(look_up && !(sh.done[i >> 5] >> (i & 31) & 1u))) {
      int lo = 0;
#pragma unroll
      for (int step = kStepItems / 2; step > 0; step >>= 1)
        if (lo + step < n_in && m.pages[lo + step] <= pg) lo += step;
      sh.l.pair[lo] = m.slots[i];
      atomicOr(&sh.done[i >> 5], 1u << (i & 31));
      ++paired;
    }
  }
  int all_paired = 0;
  if (LV_MOSTLY(look_up)) scan.sum(paired, &all_paired);
  else __syncthreads();
  // in-commit, and one task per incoming block
#pragma unroll 1
  for (long long i = threadIdx.x; i < n_in; i += kStepThreads) {
    const int32_t b = m.blks[i];
    const size_t ti = row + b;
    const long long g = m.gslot ? (long long)m.gslot[i] : -(long long)p.table[ti] - 2;
    const int32_t pg = m.pages[i];
    int4 t = make_int4(-1, -1, (int32_t)g, pg);
    if (LV_MOSTLY(look_up)) {
      t.y = sh.l.pair[i];
      if (t.y >= 0) t.x = pg;
    } else if (n_out > 0) {
      const unsigned long long pt = m.page_tag[pg];
      if ((pt >> 32) == (unsigned long long)(uint32_t)m.epoch && !(pt & kPairedBit)) {
        const long long vi = (long long)(pt & 0x7fffffffull);
        t.x = pg;
        t.y = m.slots[vi];
        ++paired;
        if (few) atomicOr(&sh.done[vi >> 5], 1u << (vi & 31));
        else m.page_tag[pg] = pt | kPairedBit;
      }
    }
    p.table[ti] = pg;
    p.own_hbm[pg] = owner_key(m.sid, b);
    if (LV_RARE(p.incl)) {
      p.shadow[ti] = (int32_t)g;             // the host slot stays as its clean copy
    } else {
      p.own_host[g] = kOwnerNone;
      host.clear((int32_t)g);
    }
    m.tasks[i] = t;
    if (LV_MOSTLY(m.pages_out != m.pages)) m.pages_out[i] = pg;
  }
  if (LV_RARE(!look_up)) scan.sum(paired, &all_paired);
  // victims whose page no incoming block takes: out-only tasks, in victim order.  (Mostly
  // there are none: a full tier's lowest free pages are the victims' own.)
  const bool more = all_paired < n_dirty;
  long long run = 0;
#pragma unroll 1
  for (long long i0 = 0; LV_RARE(more && i0 < n_out); i0 += kStepThreads) {
    const long long i = i0 + threadIdx.x;
    bool flag = false;
    int32_t pg = -1;
    if (i < n_out) {
      pg = m.v[i].page;
      if (few) {
        flag = !(sh.done[i >> 5] >> (i & 31) & 1u);
      } else {
        const unsigned long long pt = m.page_tag[pg];
        flag = (pt >> 32) == (unsigned long long)(uint32_t)m.epoch && !(pt & kPairedBit) &&
               (long long)(pt & 0x7fffffffull) == i;
      }
    }
    int chunk;
    const long long pos = run + scan.rank(flag, &chunk);
    if (flag) m.tasks[n_in + pos] = make_int4(pg, m.slots[i], -1, -1);
    run += chunk;
  }
  if (threadIdx.x == 0) {
    if (LV_RARE(n_in < m.n_in)) set_error(p.ctl, LV_ERR_STATE, n_out);
    *m.n_tasks = n_in + run;
    const long long n_clean = n_out - n_dirty;
    const long long host_delta = p.incl ? n_dirty : n_dirty - n_in;
    if (n_in) add_counts(counts_of(p, m.sid), (int)n_in, -(int)n_in);
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HOST_ALLOC]), (unsigned long long)host_delta);
    if (LV_RARE(p.incl)) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN]), (unsigned long long)(n_in - n_clean));
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN_OUT]), (unsigned long long)n_clean);
    }
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HBM_ALLOC]), (unsigned long long)(n_in - n_out));
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PAGES_OUT]), (unsigned long long)n_out);
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PAGES_IN]), (unsigned long long)n_in);
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_REMAP]), (unsigned long long)(n_out + n_in));
  }
  return true;
}

// The words of both bitmaps, twice each (bits_copy).
__host__ __device__ inline size_t bits_words(const DevPool& p) {
  return 2 * (size_t)(((p.hbm_pages + 31) >> 5) + ((p.host_pages + 31) >> 5));
}

// The exchange of a caller's lists (lv_swap_exchange).
__global__ void __launch_bounds__(kStepThreads, 1)
k_exchange_plan(DevPool p, const lv_victim* __restrict__ v, long long n_out, int32_t sid,
                const int32_t* __restrict__ blks, long long n_in, int32_t* slots, int32_t* pages,
                int4* tasks, long long* n_tasks, int32_t epoch, unsigned long long* page_tag,
                long long* cursor, int copy_bits) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ StepShared sh;
  pdl_entry();
  BlockScan scan{sh.ws, 0};
  uint32_t* copy = copy_bits ? reinterpret_cast<uint32_t*>(dyn) : nullptr;
  const TierBits hbm = bits_copy(p.bits_hbm, p.hbm_pages, copy, threadIdx.x);
  const TierBits host = bits_copy(p.bits_host, p.host_pages, copy ? copy + 2 * ((p.hbm_pages + 31) >> 5) : nullptr,
                                  threadIdx.x);
  if (threadIdx.x == 0 && cursor) *cursor = 0;
  int hbm_alloc;
  scan.sum(hbm.taken, &hbm_alloc);
  MovePlan m{v, n_out, sid, blks, nullptr, n_in, n_out <= kStepItems ? sh.l.slots : slots,
             n_in <= kStepItems ? sh.l.pages : pages, slots, pages, tasks, n_tasks, epoch, page_tag};
  plan_moves<true>(p, m, hbm, host, hbm_alloc, -1, -1, sh, scan);
  __syncthreads();
  bits_back(hbm);
  bits_back(host);
}

// Grows session sid, of ctx tokens, by n_tokens (every thread of the CTA calls it): the new
// blocks take the lowest free HBM pages, in block order.  near: room for kStepItems page ids
// in shared memory.  Returns the pages appended, -1 on an error.
__device__ long long append_tokens_to(const DevPool& p, int32_t sid, int32_t ctx, int32_t n_tokens,
                                      int32_t* pages, const TierBits& hbm, const TierBits& host,
                                      int32_t* near, BlockScan& scan, int* base) {
  const int32_t nb = (int32_t)(((uint32_t)ctx + (uint32_t)p.T - 1u) / (uint32_t)p.T);
  const uint32_t nctx = (uint32_t)ctx + (uint32_t)n_tokens;
  // (nctx past 2^31 is refused: its block count only has to be defined)
  const long long nnb = nctx > 0x7fffffffu ? 0 : (nctx + (uint32_t)p.T - 1u) / (uint32_t)p.T;
  const long long m = nnb - nb;
  if (LV_RARE(nnb > p.maxB || nctx > 0x7fffffffu)) {
    if (threadIdx.x == 0) set_error(p.ctl, LV_ERR_BOUNDS, sid);
    return -1;
  }
  if (m > 0) {
    int32_t* list = m <= kStepItems ? near : pages;
    if (LV_RARE(!take_lowest(hbm, (int)m, p.hbm_pages - p.budget, list, scan, base))) {
      if (threadIdx.x == 0) set_error(p.ctl, LV_ERR_NO_HBM, sid);
      return -1;
    }
#pragma unroll 1
    for (long long i = threadIdx.x; i < m; i += kStepThreads) {
      const int32_t pg = list[i];
      const int32_t b = (int32_t)(nb + i);
      p.table[(size_t)sid * p.maxB + b] = pg;
      p.own_hbm[pg] = owner_key(sid, b);
      if (list != pages) pages[i] = pg;
    }
  }
  if (threadIdx.x == 0) {
    if (m > 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HBM_ALLOC]), (unsigned long long)m);
      add_counts(counts_of(p, sid), (int)m, 0);
    }
    // inclusive tiers: the partially filled last block gains rows, its clean copy is stale
    if (LV_RARE(p.incl) && n_tokens > 0 && nb > 0 && ctx % p.T != 0) {
      const size_t ti = (size_t)sid * p.maxB + (nb - 1);
      const int32_t g = p.shadow[ti];
      if (g >= 0 && g < p.host_pages) {
        p.shadow[ti] = -1;
        p.own_host[g] = kOwnerNone;
        host.clear(g);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HOST_ALLOC]), (unsigned long long)-1ll);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN]), (unsigned long long)-1ll);
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN_DROPPED]), 1ull);
      }
    }
    p.sess[sid].ctx_tokens = (int32_t)nctx;
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_APPENDED]), (unsigned long long)m);
  }
  return m;
}

__global__ void __launch_bounds__(kStepThreads)
k_append(DevPool p, int32_t sid, int32_t n_tokens, int32_t* pages, int32_t* count, int copy_bits) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ int ws[2 * kStepWarps];
  __shared__ int32_t near[kStepItems];
  __shared__ int base[kStepThreads];
  pdl_entry();
  BlockScan scan{ws, 0};
  const TierBits hbm = bits_copy(p.bits_hbm, p.hbm_pages, copy_bits ? reinterpret_cast<uint32_t*>(dyn) : nullptr,
                                 threadIdx.x);
  const TierBits host = bits_copy(p.bits_host, p.host_pages, nullptr, 0);   // one bit of it at most
  const int32_t ctx = p.sess[sid].ctx_tokens;
  __syncthreads();      // every thread has read it and the bitmap
  const long long m = append_tokens_to(p, sid, ctx, n_tokens, pages, hbm, host, near, scan, base);
  if (m > 0) {
    __syncthreads();
    bits_back(hbm);
  }
  if (threadIdx.x == 0 && count) *count = m > 0 ? (int32_t)m : 0;
}

// Unit u = (task t, chunk c): kUnitVecs 16-byte vectors of the task's page, taken as one
// run of J * P bytes (which it is in the host slot; in HBM vector q of the page lies in
// sub-page q / nvec).  The out half copies the HBM page to its host slot, the in half a
// host slot to its HBM page; each thread loads both before it stores either, so a paired
// task reads the old page before overwriting it.  CTAs take units in order from a shared
// cursor (zeroed by the plan), the next one fetched while the current one is copied: a CTA
// that starts late, or runs on an SM crowded by other work, simply takes fewer units.
//
// What bounds it: the host link, as long as enough bytes are on their way.  A CTA has one
// unit in flight and 45 CTAs have to cover the link's latency, so a unit is 16 KiB each way
// whatever the sub-page size.  With one sub-page per unit, pages of 4 KiB sub-pages kept a
// quarter of that in flight: a turn that moves 45 pages of 192 KiB each way (1000 sessions)
// took 140 us and takes 106 us; pages of 16 KiB sub-pages are as before (1.90 ms for 203
// pages of 1.5 MiB each way, 336 GB/s).
constexpr int kUnitVecs = kCopyThreads * kCopyUnroll;
constexpr int kCopyKv = 512;      // sub-page arrays whose addresses a CTA keeps in shared memory

__host__ __device__ __forceinline__ long long copy_chunks(const DevPool& p) {
  return ((p.P >> 4) * p.J + kUnitVecs - 1) / kUnitVecs;
}

__global__ void __launch_bounds__(kCopyThreads)
k_exchange_copy(DevPool p, const int4* __restrict__ tasks, const long long* __restrict__ n_tasks,
                long long* __restrict__ cursor) {
  __shared__ uint8_t* kv_s[kCopyKv];
  __shared__ long long next;
  // the arrays' addresses never change: read before the plan is waited for
  for (int j = threadIdx.x; j < p.J && j < kCopyKv; j += kCopyThreads) kv_s[j] = p.kv[j];
  pdl_entry();
  const uint32_t nvec = (uint32_t)(p.P >> 4);
  const long long page_vecs = (long long)nvec * p.J;
  const long long chunks = copy_chunks(p);
  const long long units = *n_tasks * chunks;
  // x / nvec for x < nvec + kUnitVecs: at most 1 for sub-pages of a unit or more, else the
  // high half of x times ceil(2^32 / nvec) (exact: x < 2^11, nvec < 2^10)
  const uint32_t inverse = 0xffffffffu / nvec + 1u;
  if (threadIdx.x == 0) next = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(cursor), 1ull);
  __syncthreads();
  for (long long u = next; u < units; u = next) {
    // thread 0 fetches the next unit now and publishes it after the copy, so that its
    // warp does not wait for the atomic's result meanwhile
    unsigned long long fetched = 0;
    if (threadIdx.x == 0) fetched = atomicAdd(reinterpret_cast<unsigned long long*>(cursor), 1ull);
    const long long ti = u / chunks;
    const int4 t = tasks[ti];
    const long long q0 = (u - ti * chunks) * kUnitVecs;       // the unit's first vector
    const long long j0 = q0 / nvec;
    const uint32_t r0 = (uint32_t)(q0 - j0 * nvec);
    const int left = (int)(page_vecs - q0 < kUnitVecs ? page_vecs - q0 : kUnitVecs);
    const bool has_out = t.x >= 0, has_in = t.z >= 0;
    int4* dout = has_out ? reinterpret_cast<int4*>(p.host) + (size_t)t.y * page_vecs + q0 : nullptr;
    const int4* si = has_in ? reinterpret_cast<const int4*>(p.host) + (size_t)t.z * page_vecs + q0 : nullptr;
    int4 ro[kCopyUnroll], ri[kCopyUnroll];
    int4* din[kCopyUnroll];
#pragma unroll
    for (int k = 0; k < kCopyUnroll; ++k) {
      const int q = threadIdx.x + k * kCopyThreads;
      if (q < left) {
        if (has_in) ri[k] = si[q];
        const uint32_t x = r0 + q;
        const uint32_t dj = nvec >= kUnitVecs ? (uint32_t)(x >= nvec) : nvec == 1 ? x : __umulhi(x, inverse);
        const long long j = j0 + dj;
        uint8_t* base = j < kCopyKv ? kv_s[j] : p.kv[j];
        const size_t at = (size_t)(x - dj * nvec);
        din[k] = reinterpret_cast<int4*>(base + (size_t)t.w * p.P) + at;
        if (has_out) ro[k] = *(reinterpret_cast<const int4*>(base + (size_t)t.x * p.P) + at);
      }
    }
#pragma unroll
    for (int k = 0; k < kCopyUnroll; ++k) {
      const int q = threadIdx.x + k * kCopyThreads;
      if (q < left) {
        if (has_out) dout[q] = ro[k];
        if (has_in) *din[k] = ri[k];
      }
    }
    __syncthreads();   // every thread holds u before `next` is replaced
    if (threadIdx.x == 0) next = (long long)fetched;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- staged
// The staged path moves pages through a contiguous HBM staging run so that the
// copy engines can carry them over the host link: tasks (the exchange's
// {out page, out slot, in slot, in page}) are built and validated first, then
// k_stage_tasks<true> gathers every out page's 2L sub-pages into staging[t] and
// k_stage_tasks<false> scatters staging[t] into every in page.  Both move
// whole sub-pages with TMA bulk copies (global -> shared -> global), issued by
// one thread per CTA through a ring of shared-memory stages.

// Validated out-tasks of a swap-out: {page, slot, -1, -1} (all -1 when invalid).
__global__ void k_tasks_out(DevPool p, const lv_victim* __restrict__ v, const int32_t* __restrict__ slots,
                            long long n, int4* __restrict__ tasks, lv_remap_entry* __restrict__ commit) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const lv_victim x = v[i];
  const int32_t slot = slots[i];
  int4 t = make_int4(-1, -1, -1, -1);
  if (slot >= 0) {
    bool ok = x.sid >= 0 && x.sid < p.S && x.blk >= 0 && x.page >= 0 && x.page < p.hbm_pages &&
              slot < p.host_pages;
    ok = ok && x.blk < nblocks_of(p, x.sid);
    ok = ok && p.table[(size_t)x.sid * p.maxB + x.blk] == x.page &&
         p.own_hbm[x.page] == owner_key(x.sid, x.blk);
    if (!ok) set_error(p.ctl, LV_ERR_STATE, i);
    else {
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PAGES_OUT]), 1ull);
      if (clean_copy_of(p, x) == slot)        // its clean copy: no task
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN_OUT]), 1ull);
      else
        t = make_int4(x.page, slot, -1, -1);
    }
    if (commit) commit[i] = lv_remap_entry{x.sid, x.blk, ok ? -(slot + 2) : -1};
  } else if (commit) {
    commit[i] = lv_remap_entry{x.sid, x.blk, -1};
  }
  tasks[i] = t;
}

// Validated in-tasks of a swap-in: {-1, -1, slot, page} (all -1 when invalid).
__global__ void k_tasks_in(DevPool p, int32_t sid, const int32_t* __restrict__ blks,
                           const int32_t* __restrict__ pages, long long n, int4* __restrict__ tasks,
                           lv_remap_entry* __restrict__ commit) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t blk = blks[i], page = pages[i];
  int4 t = make_int4(-1, -1, -1, -1);
  const bool sid_ok = sid >= 0 && sid < p.S;
  if (page >= 0) {
    bool ok = sid_ok && blk >= 0 && blk < nblocks_of(p, sid) && page < p.hbm_pages;
    long long slot = -1;
    if (ok) {
      const int32_t e = p.table[(size_t)sid * p.maxB + blk];
      slot = -(long long)e - 2;
      ok = e <= -2 && slot < p.host_pages && p.own_host[slot] == owner_key(sid, blk);
    }
    if (!ok) set_error(p.ctl, sid_ok ? LV_ERR_STATE : LV_ERR_BOUNDS, i);
    else {
      t = make_int4(-1, -1, (int32_t)slot, page);
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PAGES_IN]), 1ull);
    }
    if (commit) commit[i] = lv_remap_entry{sid, blk, ok ? page : -1};
  } else if (commit) {
    commit[i] = lv_remap_entry{sid, blk, -1};
  }
  tasks[i] = t;
}

__device__ __forceinline__ uint32_t smem_addr(const void* ptr) {
  return (uint32_t)__cvta_generic_to_shared(ptr);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// 1-D bulk copy global -> this CTA's shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_load(void* dst_smem, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst_smem)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// 1-D bulk copy shared -> global, tracked by the bulk async-group.
__device__ __forceinline__ void bulk_store(void* dst, const void* src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
               "r"(smem_addr(src_smem)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read_1() {
  asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait on a stage barrier: false once `limit_ns` have passed (the data never came).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long limit_ns) {
  const unsigned long long t0 = global_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((long long)(global_ns() - t0) > limit_ns) return false;
  }
}

constexpr int kStageThreads = 32;     // one warp per CTA; lane 0 issues the bulk copies
constexpr int kMaxStages = 16;
constexpr long long kWaitLimitNs = 1000000000ll;   // one second per stage wait

// The HBM page of unit (t, j) of a stage kernel, -1 when the unit is skipped.
template <bool kPack, bool kPages>
__device__ __forceinline__ int32_t stage_page(const DevPool& p, const void* __restrict__ list, long long t, int j) {
  if (kPages) {
    const int32_t pg = static_cast<const int32_t*>(list)[t];
    if (pg >= 0 && pg < p.hbm_pages) return pg;
    if (j == 0) set_error(p.ctl, LV_ERR_BOUNDS, t);
    return -1;
  }
  const int4 tk = static_cast<const int4*>(list)[t];
  if (kPack) return tk.x;
  return tk.z < 0 ? -1 : tk.w;
}

// Moves units u = (task t, sub-page j) of P bytes through `stages` shared-memory
// buffers: unit i's load is issued `stages` units ahead of its store.
// pack:   staging[t][j] <- hbm_kv[j][task.x]   for tasks with task.x >= 0
// unpack: hbm_kv[j][task.w] <- staging[t][j]   for tasks with task.z >= 0
// kPages: `list` holds page ids instead of tasks (lv_pack_pages, lv_unpack_pages); a page
// outside the pool is reported and skipped.
template <bool kPack, bool kPages>
__global__ void __launch_bounds__(kStageThreads)
k_stage_tasks(DevPool p, const void* __restrict__ list, long long t_begin, long long t_end,
              uint8_t* __restrict__ staging, int stages) {
  extern __shared__ __align__(128) unsigned char stage_mem[];
  __shared__ __align__(8) uint64_t bars[kMaxStages];
  pdl_wait();
  if (threadIdx.x != 0) return;
  const uint32_t P = (uint32_t)p.P;
  for (int s = 0; s < stages; ++s) mbar_init(&bars[s], 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  const long long units = (t_end - t_begin) * p.J;
  // the units of this CTA, in order: u = blockIdx.x + k * gridDim.x
  auto unit_ptrs = [&](long long k, const uint8_t** src, uint8_t** dst) -> bool {
    const long long u = blockIdx.x + k * (long long)gridDim.x;
    const long long t = t_begin + u / p.J;
    const int j = (int)(u % p.J);
    uint8_t* st = staging + ((size_t)t * p.J + j) * P;
    const int32_t pg = stage_page<kPack, kPages>(p, list, t, j);
    if (pg < 0) return false;
    uint8_t* page = p.kv[j] + (size_t)pg * P;
    *src = kPack ? page : st;
    *dst = kPack ? st : page;
    return true;
  };
  const long long mine = units > blockIdx.x ? (units - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  uint8_t* dsts[kMaxStages];
  bool live[kMaxStages];
  uint32_t phase[kMaxStages];
  for (int s = 0; s < stages; ++s) { live[s] = false; phase[s] = 0; }
  bool failed = false;
  auto issue = [&](long long k) {
    const int s = (int)(k % stages);
    const uint8_t* src;
    live[s] = unit_ptrs(k, &src, &dsts[s]);
    if (live[s]) {
      mbar_expect_tx(&bars[s], P);
      bulk_load(stage_mem + (size_t)s * P, src, P, &bars[s]);
    }
  };
  // prologue: one load in flight per stage
  for (long long k = 0; k < mine && k < stages; ++k) issue(k);
  for (long long k = 0; k < mine; ++k) {
    const int s = (int)(k % stages);
    bool stored = false;
    if (live[s]) {
      if (!mbar_wait_bounded(&bars[s], phase[s], kWaitLimitNs)) {
        failed = true;
        break;
      }
      phase[s] ^= 1u;
      bulk_store(dsts[s], stage_mem + (size_t)s * P, P);
      bulk_commit();
      stored = true;
    }
    // refill the stage of unit k-1 once its store has read it; unit k's store may still run
    if (k >= 1 && k - 1 + stages < mine) {
      if (stored) bulk_wait_read_1();
      else bulk_wait_read_all();
      issue(k - 1 + stages);
    }
  }
  if (failed) {
    set_error(p.ctl, LV_ERR_TIMEOUT, blockIdx.x);
    // let every load still in flight land before the shared memory is released
    for (int s = 0; s < stages; ++s)
      if (live[s]) mbar_wait_bounded(&bars[s], phase[s], kWaitLimitNs);
  }
  bulk_wait_all();
}

// The exchange's copies with TMA bulk copies instead of the SMs' loads and stores:
// one thread per CTA moves units u = (task, sub-page j) through `stages`
// shared-memory stages of 2P bytes.  A unit's out half (old HBM page -> its new host
// slot) and in half (host slot -> its new HBM page) are loaded into one stage
// together and stored from it once both have arrived, so a paired task's page is
// read before it is overwritten.  Units come from the shared cursor (zeroed by the
// plan) kXBatch at a time; a CTA refills the stage of unit k-1 while unit k's stores
// still run.  The CTA issues a few instructions per 2P bytes, so its SM stays free
// for other work; every barrier wait is bounded (LV_ERR_TIMEOUT).
constexpr int kXStageMax = 8;
constexpr int kXBatch = 8;

__global__ void __launch_bounds__(kStageThreads)
k_exchange_copy_tma(DevPool p, const int4* __restrict__ tasks, const long long* __restrict__ n_tasks,
                    long long* __restrict__ cursor) {
  extern __shared__ __align__(128) unsigned char xmem[];
  __shared__ __align__(8) uint64_t bars[kXStageMax];
  pdl_entry();
  if (threadIdx.x != 0) return;
  const int stages = p.xstages;
  const uint32_t P = (uint32_t)p.P;
  const long long units = *n_tasks * p.J;
  for (int s = 0; s < stages; ++s) mbar_init(&bars[s], 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  uint8_t* dout[kXStageMax];
  uint8_t* din[kXStageMax];
  bool pending[kXStageMax];
  uint32_t phase[kXStageMax];
  for (int s = 0; s < stages; ++s) {
    dout[s] = din[s] = nullptr;
    pending[s] = false;
    phase[s] = 0;
  }
  long long ub = 0, ue = 0, taken = 0;
  bool exhausted = false;
  // takes the CTA's unit number k (its k-th, in order) into stage k % stages
  auto take = [&](long long k) {
    if (exhausted) return;
    if (ub == ue) {
      ub = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(cursor), (unsigned long long)kXBatch);
      ue = ub + kXBatch < units ? ub + kXBatch : units;
      if (ub >= units) {
        exhausted = true;
        return;
      }
    }
    const long long u = ub++;
    const int s = (int)(k % stages);
    const int4 t = tasks[u / p.J];
    const int j = (int)(u % p.J);
    unsigned char* so = xmem + (size_t)s * 2 * P;
    dout[s] = t.x >= 0 ? p.host + ((size_t)t.y * p.J + j) * P : nullptr;
    din[s] = t.z >= 0 ? p.kv[j] + (size_t)t.w * P : nullptr;
    const uint32_t bytes = (t.x >= 0 ? P : 0u) + (t.z >= 0 ? P : 0u);
    pending[s] = bytes > 0;
    if (bytes) {
      mbar_expect_tx(&bars[s], bytes);
      if (t.x >= 0) bulk_load(so, p.kv[j] + (size_t)t.x * P, P, &bars[s]);
      if (t.z >= 0) bulk_load(so + P, p.host + ((size_t)t.z * p.J + j) * P, P, &bars[s]);
    }
    taken = k + 1;
  };
  for (long long k = 0; k < stages; ++k) take(k);
  bool failed = false;
  for (long long k = 0; k < taken; ++k) {
    const int s = (int)(k % stages);
    bool stored = false;
    if (pending[s]) {
      if (!mbar_wait_bounded(&bars[s], phase[s], kWaitLimitNs)) {
        failed = true;
        break;
      }
      pending[s] = false;
      phase[s] ^= 1u;
      unsigned char* so = xmem + (size_t)s * 2 * P;
      if (dout[s]) bulk_store(dout[s], so, P);
      if (din[s]) bulk_store(din[s], so + P, P);
      bulk_commit();
      stored = true;
    }
    // refill the stage of unit k-1 once its stores have read it; unit k's may still run
    if (k >= 1 && !exhausted) {
      if (stored) bulk_wait_read_1();
      else bulk_wait_read_all();
      take(k - 1 + stages);
    }
  }
  if (failed) {
    set_error(p.ctl, LV_ERR_TIMEOUT, blockIdx.x);
    // let every load still in flight land before the shared memory is released
    for (int s = 0; s < stages; ++s)
      if (pending[s]) mbar_wait_bounded(&bars[s], phase[s], kWaitLimitNs);
  }
  bulk_wait_all();
}

// The same moves with plain 16-byte loads and stores (256 threads per CTA).
template <bool kPack, bool kPages>
__global__ void __launch_bounds__(kCopyThreads)
k_stage_tasks_lsu(DevPool p, const void* __restrict__ list, long long t_begin, long long t_end,
                  uint8_t* __restrict__ staging) {
  pdl_wait();
  const long long units = (t_end - t_begin) * p.J;
  const int nvec = (int)(p.P >> 4);
  for (long long u = blockIdx.x; u < units; u += gridDim.x) {
    const long long t = t_begin + u / p.J;
    const int j = (int)(u % p.J);
    int4* st = reinterpret_cast<int4*>(staging + ((size_t)t * p.J + j) * p.P);
    const int32_t pg = stage_page<kPack, kPages>(p, list, t, threadIdx.x == 0 ? j : 1);
    if (pg < 0) continue;
    int4* page = reinterpret_cast<int4*>(p.kv[j] + (size_t)pg * p.P);
    if (kPack) copy_subpage(page, st, nvec);
    else copy_subpage(st, page, nvec);
  }
}

// Self-test of the bounded wait: one thread arms a stage barrier for bytes that no
// copy will ever deliver and waits on it with the given limit; the timeout must be
// reported in the error word and the kernel must return.
__global__ void k_selftest_wait(long long* ctl, long long limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  mbar_expect_tx(&bar, 16);                       // 16 bytes that never arrive
  if (!mbar_wait_bounded(&bar, 0, limit_ns)) set_error(ctl, LV_ERR_TIMEOUT, limit_ns);
}

// ---------------------------------------------------------------- commit
constexpr int kRemapThreads = 256;
constexpr int kReleaseThreads = 256;

// The reads of one entry that do not depend on a check.
struct RemapRead {
  lv_remap_entry x;
  size_t ti;            // table index (0 when out of range)
  int32_t old;          // the block's current location
  int32_t g;            // its clean-copy slot (inclusive tiers), or -1
  int32_t nb;           // blocks of its session
  bool in_range;
};

struct RemapCounts {
  int ok, hbm, host, clean;
  int dh, dd;           // the last settled entry's change of its session's counts
};

__device__ __forceinline__ void remap_read_entry(const DevPool& p, const lv_remap_entry* e, long long i,
                                                 long long n, RemapRead& r) {
  r.x = i < n ? e[i] : lv_remap_entry{-1, -1, -1};
  r.in_range = i < n && r.x.sid >= 0 && r.x.sid < p.S && r.x.blk >= 0 && r.x.blk < p.maxB;
  r.ti = r.in_range ? (size_t)r.x.sid * p.maxB + r.x.blk : 0;
}

__device__ __forceinline__ void remap_read_table(const DevPool& p, RemapRead& r) {
  r.old = r.in_range ? p.table[r.ti] : -1;
  r.g = (r.in_range && p.incl) ? p.shadow[r.ti] : -1;
  r.nb = r.in_range ? nblocks_of(p, r.x.sid) : 0;
}

// The block's epoch mark: one accepted entry per block per call.  It depends on
// the entry alone, so it is issued with the entry's table reads; a mark made for
// a block past its session's context is harmless (every entry naming that block
// fails the same range check).  A returning atomic: the caller issues every
// entry's mark before it looks at any result.
__device__ __forceinline__ void remap_mark(const DevPool& p, const RemapRead& r, int32_t epoch,
                                           int32_t& seen) {
  seen = r.in_range ? atomicExch(&p.mark[r.ti], epoch) : 0;
}

// The entry's error once its table reads and mark are back: range first, then
// a second entry for the same block.
__device__ __forceinline__ int remap_judge(const RemapRead& r, int32_t epoch, int32_t seen) {
  if (!r.in_range || r.x.blk >= r.nb) return LV_ERR_BOUNDS;
  if (seen == epoch) return LV_ERR_DOUBLE_MAP;
  return 0;
}

// Round 3 of an entry that passed its range check and its mark.  The claim of the
// new location (one CAS checks that it is a reservation nobody owns and takes it)
// goes out together with the entry's own writes, made before the claim's result
// is known: the table word, and the old location exchanged to kOwnerFreeing
// (which returns its owner word into `was`, for the consistency check).  The
// release pass after the commit makes a kOwnerFreeing word free and clears its
// bitmap bit.  A claim that fails undoes the writes in remap_settle; until then
// no other entry of the call can see them, since only an entry for the same
// block reads its table word (and the mark turned it away), and every claim of
// an owned location fails, kOwnerFreeing or not.
template <bool kDirect>
__device__ __forceinline__ int remap_claim(const DevPool& p, const RemapRead& r, int err,
                                           uint32_t& got, uint32_t& was) {
  if (err) return err;
  const lv_remap_entry& x = r.x;
  const uint32_t key = owner_key(x.sid, x.blk);
  uint32_t* own;
  if (x.loc >= 0) {
    if (x.loc >= p.hbm_pages) return LV_ERR_BOUNDS;
    own = &p.own_hbm[x.loc];
  } else if (x.loc <= -2) {
    if (-(long long)x.loc - 2 >= p.host_pages) return LV_ERR_BOUNDS;
    own = &p.own_host[-(long long)x.loc - 2];
  } else {
    return LV_ERR_BOUNDS;
  }
  got = atomicCAS(own, kOwnerReserved, key);
  const int32_t old = r.old;
  const long long old_slot = -(long long)old - 2;
  if (old >= 0 && old < p.hbm_pages) {
    was = atomicExch(&p.own_hbm[old], kDirect ? kOwnerNone : kOwnerFreeing);
  } else if (old <= -2 && old_slot < p.host_pages) {
    if (p.incl && x.loc >= 0) was = p.own_host[old_slot];   // back in HBM: the slot stays as its clean copy
    else was = atomicExch(&p.own_host[old_slot], kDirect ? kOwnerNone : kOwnerFreeing);
  }
  p.table[r.ti] = x.loc;
  return 0;
}

// Judges the claim once its result is back.  A failed claim is a double map and
// its entry's writes are put back; an accepted entry settles its clean copy
// (inclusive tiers) and is counted, and a freed location that this block did not
// own means the tables were inconsistent.
template <bool kDirect>
__device__ __forceinline__ void remap_settle(const DevPool& p, const RemapRead& r, int err,
                                             uint32_t got, uint32_t was, long long i,
                                             RemapCounts& c) {
  const lv_remap_entry& x = r.x;
  const int32_t old = r.old, g = r.g;
  const long long old_slot = -(long long)old - 2;
  const bool old_hbm = old >= 0 && old < p.hbm_pages;
  const bool old_host = old <= -2 && old_slot < p.host_pages;
  const long long h = -(long long)x.loc - 2;
  const uint32_t key = owner_key(x.sid, x.blk);
  if (!err && got != kOwnerReserved) {
    // a host location already owned by this block is fine only as its own clean copy
    if (!(x.loc <= -2 && p.incl && (long long)g == h && got == key)) {
      err = LV_ERR_DOUBLE_MAP;
      p.table[r.ti] = old;
      if (old_hbm) p.own_hbm[old] = was;
      else if (old_host && !(p.incl && x.loc >= 0)) p.own_host[old_slot] = was;
    }
  }
  c.dh = c.dd = 0;
  if (err) {
    set_error(p.ctl, err, i);
    return;
  }
  const int2 from = tier_of(old), to = tier_of(x.loc);
  c.dh = to.x - from.x;
  c.dd = to.y - from.y;
  if (x.loc <= -2 && g >= 0) {          // the copy becomes the location, or goes
    p.shadow[r.ti] = -1;
    c.clean -= 1;
    if ((long long)g != h) {
      atomicExch(&p.own_host[g], kDirect ? kOwnerNone : kOwnerFreeing);
      if (kDirect) atomicAnd(&p.bits_host[g >> 5], ~(1u << (g & 31)));
      c.host += 1;
    }
  }
  if (old_hbm) {
    if (kDirect) atomicAnd(&p.bits_hbm[old >> 5], ~(1u << (old & 31)));
    c.hbm += 1;
  } else if (old_host) {
    if (p.incl && x.loc >= 0) {
      p.shadow[r.ti] = (int32_t)old_slot;
      c.clean += 1;
    } else {
      if (kDirect) atomicAnd(&p.bits_host[old_slot >> 5], ~(1u << (old_slot & 31)));
      c.host += 1;
    }
  }
  if (was != kOwnerNone && was != key) set_error(p.ctl, LV_ERR_STATE, i);
  c.ok += 1;
}

// Each thread commits E entries, a CTA's threads apart, so that a warp's entries are
// contiguous and a CTA's mostly of one session.  The allocation counts and the
// commit counter change by block totals (one atomic per block and counter).
// Inclusive tiers: a host location may be the block's own clean copy; a block
// committed to HBM from the host tier keeps its slot as its clean copy; a
// block committed to another host slot loses its copy.
//
// The kernel is bound by the latency of dependent scattered accesses, so each
// round of requests is issued for all E entries of the thread before any of its
// results is used, and requests that do not depend on one another share a
// round: (1) the entries; (2) the block's table word, its session's block count
// and the block's epoch mark; (3) the claim of the new location, the table word
// and the exchange of the old location's owner word (only for an entry that
// passed its range check and its mark; the writes are undone if the claim
// fails).  E chains then wait together.  The early reads are race-free within
// one call: a block has at most one accepted entry (the epoch mark), a location
// freed by one entry is never the new location of another (new locations are
// reservations), and another entry can take an owned location only through a
// CAS, which then fails.  A thread's own entries are issued in order, so a
// duplicate among them meets the epoch mark too.
//
// kDirect: the freed locations' owner words and bitmap bits are cleared by the entries
// themselves and there is no release pass.  That pass reads both tiers' owner words, whatever
// the number of entries, and is a launch of its own: a commit of 1024 of 2^20 pages takes 7 to
// 9 us without it and 11 with it.
//
// The sessions' counts are what many entries wait for one another at: a warp whose entries
// are of one session adds once, but a warp of mixed ones adds 32 times to a few lines, and 16
// sessions of 65536 blocks each in order 8192 times to each of 16 words.  So the form with a
// release pass adds to one of spread_copies arrays, which that pass adds up: 2^20 entries of
// 16 sessions 57 us without the copies and 25.7 with them, in mixed order 310 and 50; of 512
// sessions 27.5 and 25.7, in mixed order 106 and 45 (26 and 37.5 when no counts were kept).
// The direct form has no such pass, so it ends where mixed orders make it the longer one:
// 2^14 entries of 16 sessions 11.5 us, of 2 13, and 2^16 25, against 13 to 15.
template <int E, bool kDirect>
__global__ void __launch_bounds__(kRemapThreads, 4)
k_remap(DevPool p, const lv_remap_entry* __restrict__ e, long long n, int32_t epoch) {
  if (kDirect) pdl_entry();
  else pdl_wait();          // a large grid: the release pass is scheduled behind it
  const long long i0 = blockIdx.x * (long long)(E * kRemapThreads) + threadIdx.x;
  RemapRead r[E];
  int32_t seen[E];
#pragma unroll
  for (int j = 0; j < E; ++j) remap_read_entry(p, e, i0 + j * kRemapThreads, n, r[j]);
#pragma unroll
  for (int j = 0; j < E; ++j) {
    remap_read_table(p, r[j]);
    remap_mark(p, r[j], epoch, seen[j]);
  }
  int err[E];
  uint32_t got[E], was[E];
#pragma unroll
  for (int j = 0; j < E; ++j) {
    got[j] = kOwnerReserved;
    was[j] = kOwnerNone;
    err[j] = i0 + j * kRemapThreads < n ? remap_judge(r[j], epoch, seen[j]) : -1;
    if (err[j] >= 0) err[j] = remap_claim<kDirect>(p, r[j], err[j], got[j], was[j]);
  }
  RemapCounts c{0, 0, 0, 0, 0, 0};
  unsigned long long* cnt = counts_of(p, 0);
  if (!kDirect) cnt = p.spread + (size_t)(i0 & (p.spread_copies - 1)) * p.S;
  int32_t sid[E];
  int change[E];
#pragma unroll
  for (int j = 0; j < E; ++j) {
    c.dh = c.dd = 0;
    if (err[j] >= 0) remap_settle<kDirect>(p, r[j], err[j], got[j], was[j], i0 + j * kRemapThreads, c);
    sid[j] = r[j].x.sid;
    change[j] = c.dd * 65536 + c.dh;
  }
  warp_counts<E>(cnt, sid, change);
  // block totals: warp sums, one shared atomic per warp, one global atomic per block
  __shared__ int tot[4];
  if (threadIdx.x < 4) tot[threadIdx.x] = 0;
  __syncthreads();
  const int ok = __reduce_add_sync(0xffffffffu, c.ok), fh = __reduce_add_sync(0xffffffffu, c.hbm);
  const int fo = __reduce_add_sync(0xffffffffu, c.host), cl = __reduce_add_sync(0xffffffffu, c.clean);
  if ((threadIdx.x & 31) == 0) {
    if (ok) atomicAdd(&tot[0], ok);
    if (fh) atomicAdd(&tot[1], fh);
    if (fo) atomicAdd(&tot[2], fo);
    if (cl) atomicAdd(&tot[3], cl);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (tot[1]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HBM_ALLOC]), (unsigned long long)-(long long)tot[1]);
    if (tot[2]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_HOST_ALLOC]), (unsigned long long)-(long long)tot[2]);
    if (tot[0]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_REMAP]), (unsigned long long)tot[0]);
    if (tot[3]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CLEAN]), (unsigned long long)(long long)tot[3]);
  }
}

// The commit's second pass: every owner word that the commit exchanged to
// kOwnerFreeing becomes kOwnerNone, and its bit is cleared in the allocation
// bitmap with one reduction per bitmap word (the commit itself would issue one
// reduction per freed page, 32 to a word when a whole run of pages is freed).
// Thread q reads owner words 4q..4q+3 of its tier with one 16-byte load; the 8
// threads of a bitmap word combine their bits with shuffles.  Quads [0, qh) are
// the HBM pages and [qh, qh + qo) the host slots; qh and qo are multiples of 8,
// so the 8 threads of a word are always 8 aligned lanes of one tier.  Each thread
// issues the loads of kReleaseUnroll quads, a grid's width apart, before it looks
// at any of them.  Only the freed words are written, so concurrent work on other
// pages is left alone.
constexpr int kReleaseUnroll = 2;

__device__ __forceinline__ uint4 release_load(const DevPool& p, long long q, long long qh,
                                              long long total) {
  uint4 v = make_uint4(kOwnerNone, kOwnerNone, kOwnerNone, kOwnerNone);
  if (q >= total) return v;
  const bool hbm = q < qh;
  const uint32_t* own = hbm ? p.own_hbm : p.own_host;
  const long long n = hbm ? p.hbm_pages : p.host_pages;
  const long long base = (hbm ? q : q - qh) * 4;
  if (base + 3 < n) {
    v = *reinterpret_cast<const uint4*>(own + base);
  } else {
    if (base < n) v.x = own[base];
    if (base + 1 < n) v.y = own[base + 1];
    if (base + 2 < n) v.z = own[base + 2];
  }
  return v;
}

__device__ __forceinline__ void release_apply(const DevPool& p, long long q, long long qh,
                                              long long total, uint4 v, int lane8) {
  const bool hbm = q < qh;
  uint32_t* own = hbm ? p.own_hbm : p.own_host;
  const long long base = (hbm ? q : q - qh) * 4;
  uint32_t m = 0;
  if (q < total) {
    m = (uint32_t)(v.x == kOwnerFreeing) | (uint32_t)(v.y == kOwnerFreeing) << 1 |
        (uint32_t)(v.z == kOwnerFreeing) << 2 | (uint32_t)(v.w == kOwnerFreeing) << 3;
    for (int k = 0; k < 4; ++k)
      if (m >> k & 1u) own[base + k] = kOwnerNone;
  }
  uint32_t w = m << (4 * lane8);
  w |= __shfl_xor_sync(0xffffffffu, w, 1);
  w |= __shfl_xor_sync(0xffffffffu, w, 2);
  w |= __shfl_xor_sync(0xffffffffu, w, 4);
  if (lane8 == 0 && w) atomicAnd(&(hbm ? p.bits_hbm : p.bits_host)[base >> 5], ~w);
}

__global__ void __launch_bounds__(kReleaseThreads)
k_release(DevPool p, long long qh, long long qo) {
  pdl_wait();   // the commit is complete and visible
  const long long total = qh + qo;
  const long long step = (long long)gridDim.x * kReleaseThreads;
  const int lane8 = threadIdx.x & 7;
  // the sessions' counts (whichever commit's changes they are, each is taken once)
  const int changes = p.spread_copies * p.S;
  for (long long i = (long long)blockIdx.x * kReleaseThreads + threadIdx.x; i < changes; i += step) {
    if (p.spread[i] == 0ull) continue;
    const unsigned long long x = atomicExch(&p.spread[i], 0ull);
    if (x) atomicAdd(counts_of(p, (int32_t)(i % p.S)), x);
  }
  for (long long q0 = (long long)blockIdx.x * kReleaseThreads + threadIdx.x;
       q0 - threadIdx.x < total; q0 += kReleaseUnroll * step) {
    uint4 v[kReleaseUnroll];
#pragma unroll
    for (int u = 0; u < kReleaseUnroll; ++u) v[u] = release_load(p, q0 + u * step, qh, total);
#pragma unroll
    for (int u = 0; u < kReleaseUnroll; ++u) release_apply(p, q0 + u * step, qh, total, v[u], lane8);
  }
}

__global__ void k_cancel(DevPool p, const int32_t* __restrict__ locs, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t loc = locs[i];
  uint32_t* bits;
  uint32_t* own;
  long long idx;
  int which;
  if (loc >= 0 && loc < p.hbm_pages) {
    bits = p.bits_hbm; own = p.own_hbm; idx = loc; which = C_HBM_ALLOC;
  } else if (loc <= -2 && (-(long long)loc - 2) < p.host_pages) {
    bits = p.bits_host; own = p.own_host; idx = -(long long)loc - 2; which = C_HOST_ALLOC;
  } else {
    set_error(p.ctl, LV_ERR_BOUNDS, i);
    return;
  }
  // only a pending reservation can be released; a clean copy was never reserved
  const uint32_t o = atomicCAS(&own[idx], kOwnerReserved, kOwnerNone);
  if (o != kOwnerReserved) {
    const int32_t os = (int32_t)(o >> 16), ob = (int32_t)(o & 0xFFFFu);
    const bool copy = p.incl && which == C_HOST_ALLOC && o != kOwnerNone && os < p.S &&
                      ob < p.maxB && p.shadow[(size_t)os * p.maxB + ob] == idx;
    if (!copy) set_error(p.ctl, LV_ERR_STATE, i);
    return;
  }
  const uint32_t m = 1u << (idx & 31);
  atomicAnd(&bits[idx >> 5], ~m);
  atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[which]), (unsigned long long)-1ll);
  atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_CANCELS]), 1ull);
}

// ---------------------------------------------------------------- step
// A device-driven step -- lv_turn, lv_make_resident, lv_evict -- as one kernel of one CTA,
// followed by the exchange copy: pick the turn's session, begin the turn, list its host-tier
// blocks, the deficit, the ranking, the victims, the plan and its commits, the growth, and
// the step's end.  It reads per-session counts, the rows of the sessions concerned and the
// bitmaps, so what bounds it is the chain of dependent reads and the instructions between
// them.  As six to eight kernels in a row (pick, prepare, order, census of every table row,
// emission, plan, append) these decisions took 25-27 us of a turn of 16 or 1000 sessions, and
// 24 us of an eviction; as one kernel 17-19 and 12 us; with the session table read in whole
// lines, the bitmaps changed in shared memory and rare branches out of line 11 us for 16
// sessions.  Whole turns, when the copy took 16 KiB units already: eight sessions that move 24
// pages of 16 KiB each way 47 us with the kernels in a row, 22.8 as one, 19.1 now; 1000
// sessions and 45 pages of 192 KiB in scattered order 106, 81.8 and 75.2.
constexpr int kSelectRounds = 12;   // sessions found by repeated maximum at most
constexpr int kCountedLoads = 128;  // loads ordered by counting; more are sorted

// The step's arguments beyond the pool.
struct StepArgs {
  ResidentScratch rs;
  int32_t sid;                      // -1: lv_turn picks from cand
  const int32_t* cand;
  int32_t n_cand;
  const unsigned long long* keys;   // the loads' order, or null: ascending block id
  long long now_us;
  long long audio_us, units;        // lv_turn: LV_EV_TURN_END's a and b
  long long max_load;               // preload admission (< 0: no limit)
  long long evict;                  // lv_evict: pages to free; -1 for the other steps
  int32_t append_tokens;
  int32_t epoch;
  int turn, preload;
  // kStepAll, or in two parts around k_order_loads: kStepList up to the list of loads,
  // kStepMove the rest
  int part;
  int copy_bits;                    // the bitmaps fit in shared memory
  lv_resident_result* out;          // may be null
};
enum { kStepAll = 0, kStepList = 1, kStepMove = 2 };

// Dynamic shared memory of k_step: [n2] keys, places, blocks in HBM, blocks in the host tier
// and blocks of the sessions, [kStepItems] keys and indexes of the loads' order, both bitmaps.
struct StepLayout {
  int n2;
  size_t off, cnt, away, nb, load, bits, total;
};

__host__ __device__ inline StepLayout step_layout(const DevPool& p, bool ordered, bool copy_bits) {
  StepLayout l{};
  l.n2 = 32;
#pragma unroll 1
  while (l.n2 < p.S) l.n2 *= 2;
  l.off = (size_t)l.n2 * 8;
  l.cnt = l.off + (size_t)l.n2 * 4;
  l.away = l.cnt + (size_t)l.n2 * 4;
  l.nb = l.away + (size_t)l.n2 * 4;
  l.load = l.nb + (size_t)l.n2 * 4;
  l.bits = l.load + (ordered ? (size_t)kStepItems * 12 : 0);
  l.total = l.bits + (copy_bits ? bits_words(p) * 4 : 0);
  return l;
}

// Bitonic sort of n (a power of two) entries in shared memory: keys descending, or, with an
// index per key, (key, index) ascending.
template <bool kIndexed>
__device__ void sort_entries(unsigned long long* key, int* idx, int n) {
#pragma unroll 1
  for (int k = 2; k <= n; k <<= 1) {
#pragma unroll 1
    for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll 1
      for (int i = threadIdx.x; i < n / 2; i += kStepThreads) {
        const int lo = ((i & ~(j - 1)) << 1) | (i & (j - 1)), hi = lo | j;
        const unsigned long long x = key[lo], y = key[hi];
        const bool first = (lo & k) == 0;
        bool less = x < y;                     // lo's entry belongs after hi's in descending order
        bool more = x > y;
        if (kIndexed && x == y) {
          less = idx[lo] < idx[hi];
          more = idx[lo] > idx[hi];
        }
        const bool swap = kIndexed ? (first ? more : less) : (first ? less : more);
        if (swap) {
          key[lo] = y;
          key[hi] = x;
          if (kIndexed) {
            const int t = idx[lo];
            idx[lo] = idx[hi];
            idx[hi] = t;
          }
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ unsigned long long warp_max(unsigned long long x) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(x >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(x >> 32) == hi ? (unsigned)x : 0u);
  return (unsigned long long)hi << 32 | lo;
}

// The largest of every thread's v, to all of them (one barrier; two buffers as BlockScan).
__device__ __forceinline__ unsigned long long block_max(unsigned long long v, StepShared& sh, int ph) {
  v = warp_max(v);
  if ((threadIdx.x & 31) == 0) sh.best[ph][threadIdx.x >> 5] = v;
  __syncthreads();
  return warp_max((threadIdx.x & 31) < kStepWarps ? sh.best[ph][threadIdx.x & 31] : 0ull);
}

__device__ __forceinline__ int32_t session_of_key(unsigned long long key) {
  return 0x7fffffff - (int32_t)(key & 0x7fffffffull);
}

// A check of owner words that does not wait for them: a word is compared when the next one
// is read, or at the end, so that the read is not a link of the chain.
struct OwnerCheck {
  uint32_t owner, key;
  long long pos, bad;       // -1: none
  __device__ void settle() {
    if (pos >= 0 && owner != key && bad < 0) bad = pos;
    pos = -1;
  }
  __device__ void read(const uint32_t* own, long long i, long long n) {
    settle();
    owner = kOwnerNone;
    if (i >= 0 && i < n) owner = own[i];
  }
  __device__ void expect(uint32_t k, long long at) {
    key = k;
    pos = at;
  }
};

// Where victims go, and what their pages' owner words are checked against.
struct VictimList {
  lv_victim* near;          // shared memory, or null
  lv_victim* far;
  const uint32_t* own;      // null: not checked
  long long n_own;
  int n_out;          // positions below this are written
  __device__ void put(int pos, int32_t s, int32_t b, int32_t e) const {
    if (near) near[pos] = lv_victim{s, b, e};
    far[pos] = lv_victim{s, b, e};
  }
};

// The blocks of session s (nb of them) in victim order, by the whole CTA: positions pos0 to
// end of the list, which the session's count gave it.  A block's page has to be its own, and
// every position has to be filled: a row that holds fewer blocks than were counted (a commit
// on another stream between the two) is a wrong victim, of one that holds more the first are
// taken.
__device__ void emit_whole(const DevPool& p, int32_t s, int32_t nb, int pos0, int end,
                           const VictimList& l, OwnerCheck& check, BlockScan& scan) {
  const int32_t* row = p.table + (size_t)s * p.maxB;
  const bool suffix = p.within == LV_SUFFIX_FIRST;
#pragma unroll 1
  for (int32_t q0 = 0; q0 < nb && pos0 < end; q0 += kStepThreads) {
    const int32_t q = q0 + threadIdx.x;
    const int32_t b = suffix ? nb - 1 - q : q;
    const int32_t e = q < nb ? row[b] : -1;
    check.read(l.own, e, l.n_own);
    int chunk;
    const int pos = pos0 + scan.rank(e >= 0, &chunk);
    if (e >= 0 && pos < end) {
      l.put(pos, s, b, e);
      if (l.own) check.expect(owner_key(s, b), pos);
    }
    pos0 += chunk;
  }
  if (LV_RARE(pos0 < end)) check.bad = pos0;
}

// The same for sessions `of(r)`, r = first, first + kStepWarps, ... below m, by one warp, four
// sessions at a time: the first 32 blocks of each are read together (a session of a few
// blocks costs a read's latency, whoever reads it).
template <typename Of>
__device__ void emit_warp(const DevPool& p, const int* nblk, const int* cnt, int m, const VictimList& l,
                          OwnerCheck& check, Of of) {
  const int lane = threadIdx.x & 31;
  const bool suffix = p.within == LV_SUFFIX_FIRST;
#pragma unroll 1
  for (int r0 = threadIdx.x >> 5; r0 < m; r0 += 4 * kStepWarps) {
    int32_t e[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + u * kStepWarps;
      e[u] = -1;
      if (r < m) {
        const int32_t s = of(r).x, nb = nblk[s];
        if (lane < nb) e[u] = p.table[(size_t)s * p.maxB + (suffix ? nb - 1 - lane : lane)];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + u * kStepWarps;
      if (r >= m) break;
      const int2 so = of(r);
      const int32_t s = so.x, nb = nblk[s];
      const int32_t* row = p.table + (size_t)s * p.maxB;
      int pos0 = so.y;
      const int end = min(pos0 + cnt[s], l.n_out);
      int32_t x = e[u];
#pragma unroll 1
      for (int32_t q0 = 0;; ) {
        const int32_t q = q0 + lane;
        check.read(l.own, x, l.n_own);
        const unsigned has = __ballot_sync(0xffffffffu, x >= 0);
        const int pos = pos0 + __popc(has & ((1u << lane) - 1u));
        if (x >= 0 && pos < end) {
          const int32_t b = suffix ? nb - 1 - q : q;
          l.put(pos, s, b, x);
          if (l.own) check.expect(owner_key(s, b), pos);
        }
        pos0 += __popc(has);
        q0 += 32;
        if (q0 >= nb || pos0 >= end) break;
        x = q0 + lane < nb ? row[suffix ? nb - 1 - q0 - lane : q0 + lane] : -1;
      }
      if (LV_RARE(pos0 < end)) check.bad = pos0;
    }
  }
}

// The sessions that the first n_out positions of the victim order touch.
struct Selected {
  int m;                // sessions
  bool sorted;          // in keys / off (the sorted keys), else in sh.sel_sid / sh.sel_off
  long long n_out;      // min(k, total)
  long long total;      // resident blocks of all candidates
};

// The lowest key among those of the first n positions (n of the order's blocks are found for
// certain): the range of the keys that hold position n is narrowed by histograms of
// kStepThreads bins, weighted by the sessions' blocks, over the tight range of the keys left;
// two or three rounds for spread keys, three or four where T_next ties.
__device__ unsigned long long threshold_key(const DevPool& p, const unsigned long long* keys, const int* cnt,
                                            long long n, StepShared& sh, BlockScan& scan) {
  unsigned long long lo = 1, hi = ~0ull;
  long long above = 0;
#pragma unroll 1
  for (;;) {
    unsigned long long high = 0, low = 0;        // low: the largest complement
#pragma unroll 1
    for (int s = threadIdx.x; s < p.S; s += kStepThreads) {
      const unsigned long long x = keys[s];
      const bool in = x >= lo && x <= hi;
      if (in && x > high) high = x;
      if (in && ~x > low) low = ~x;
    }
    high = block_max(high, sh, 0);
    low = ~block_max(low, sh, 1);
    if (low == high) return low;
    const int bits = 64 - __clzll((long long)(high - low));
    const int shift = bits > 9 ? bits - 9 : 0;
    static_assert(kStepThreads == 512, "nine bits of bins");
    sh.base[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll 1
    for (int s = threadIdx.x; s < p.S; s += kStepThreads) {
      const unsigned long long x = keys[s];
      if (x >= low && x <= high) atomicAdd(&sh.base[(x - low) >> shift], cnt[s]);
    }
    __syncthreads();
    const int bin = kStepThreads - 1 - (int)threadIdx.x;    // largest first
    const int w = sh.base[bin];
    int total;
    const long long before = above + scan.sum(w, &total);
    if (before < n && n <= before + w) {
      sh.sel_sid[0] = bin;
      sh.sel_off[0] = (int)before;
    }
    __syncthreads();
    above = sh.sel_off[0];
    lo = low + ((unsigned long long)sh.sel_sid[0] << shift);
    hi = lo + ((1ull << shift) - 1);
    if (hi < lo || hi > high) hi = high;
  }
}

// Ranks by the keys and counts in shared memory (keys[s] != 0 for candidates with at least
// one resident block; session `running` is none, whatever its key) and finds the sessions of
// the first k victims.  Where few sessions should hold k blocks they are found by repeated
// maximum, one barrier each; else, or when kSelectRounds were not enough, by the threshold
// key, and the sessions' places by comparing them with one another, or by a sort of more
// than kCompared.  (4096 sessions, 1500 victims of 7 or 8 sessions: 7.8 us by maximum -- 9.3
// when every round read all keys again instead of a thread's two largest -- and 12.6 by the
// threshold; 256 victims of 128 sessions: 48 us by maximum and a sort of all keys, 13.1 by
// the threshold.)  Keys are distinct (each holds its session).  A thread may call it with
// only its own sessions' keys and counts (s = thread, thread + kStepThreads, ...) written.
constexpr int kCompared = 256;
__device__ Selected select_sessions(const DevPool& p, unsigned long long* keys, int* off, const int* cnt,
                                    long long k, int32_t running, StepShared& sh, BlockScan& scan) {
  Selected r{};
  int mine = 0, cand = 0;
  // a thread's two largest keys: when one of them is taken the other is at hand
  unsigned long long v = 0, v2 = 0;
#pragma unroll 1
  for (int s = threadIdx.x; s < p.S; s += kStepThreads) {
    if (s == running) keys[s] = 0ull;
    const unsigned long long x = keys[s];
    mine += x ? cnt[s] : 0;
    cand += x ? 1 : 0;
    v2 = x > v ? v : x > v2 ? x : v2;
    v = x > v ? x : v;
  }
  mine = __reduce_add_sync(0xffffffffu, mine);
  cand = __reduce_add_sync(0xffffffffu, cand);
  if ((threadIdx.x & 31) == 0) sh.sums[threadIdx.x >> 5] = make_int2(mine, cand);
  unsigned long long last = block_max(v, sh, 0);
  const int2 part = (threadIdx.x & 31) < kStepWarps ? sh.sums[threadIdx.x & 31] : make_int2(0, 0);
  const int total = __reduce_add_sync(0xffffffffu, part.x), cands = __reduce_add_sync(0xffffffffu, part.y);
  r.total = total;
  r.n_out = k < total ? k : total;
  long long at = 0;
  const bool few = r.n_out * cands <= 8ll * total;      // eight sessions of average size
  if (LV_MOSTLY(few)) {
#pragma unroll 1
    while (at < r.n_out) {
      const int32_t s = session_of_key(last);
      if (threadIdx.x == 0) {
        sh.sel_sid[r.m] = s;
        sh.sel_off[r.m] = (int)at;
      }
      at += cnt[s];
      ++r.m;
      if (at >= r.n_out || r.m == kSelectRounds) break;
      if (v == last) {
        v = v2;
        v2 = ~0ull;                               // not known
        if (LV_RARE(v == ~0ull)) {
          v = 0;
#pragma unroll 1
          for (int s2 = threadIdx.x; s2 < p.S; s2 += kStepThreads) {
            const unsigned long long x = keys[s2];
            if (x < last && x > v) v = x;
          }
        }
      }
      last = block_max(v, sh, r.m & 1);
    }
  }
  if (LV_RARE(at < r.n_out)) {
    r.sorted = true;
    __syncthreads();
    const unsigned long long least = threshold_key(p, keys, cnt, r.n_out, sh, scan);
    // the chosen keys to the front of the array
    constexpr int kEach = 4096 / kStepThreads;      // a pool's sessions per thread at most
    unsigned long long x[kEach];
    int chosen = 0;
#pragma unroll
    for (int u = 0; u < kEach; ++u) {
      const int s = threadIdx.x + u * kStepThreads;
      x[u] = s < p.S ? keys[s] : 0ull;
      if (x[u] < least) x[u] = 0ull;
      chosen += x[u] ? 1 : 0;
    }
    int at2 = scan.sum(chosen, &r.m);               // (every thread has read its keys)
#pragma unroll
    for (int u = 0; u < kEach; ++u)
      if (x[u]) keys[at2++] = x[u];
    __syncthreads();
    if (r.m <= kCompared) {
      const int i = threadIdx.x;
      const unsigned long long key = i < r.m ? keys[i] : 0ull;
      if (i < r.m) off[i] = cnt[session_of_key(key)];
      __syncthreads();
      int before = 0;
      if (i < r.m) {
#pragma unroll 4
        for (int j = 0; j < r.m; ++j) before += keys[j] > key ? off[j] : 0;
      }
      __syncthreads();
      if (i < r.m) off[i] = before;
    } else {
      int n2 = 2 * kCompared;
      while (n2 < r.m) n2 *= 2;
#pragma unroll 1
      for (int i = r.m + threadIdx.x; i < n2; i += kStepThreads) keys[i] = 0ull;
      __syncthreads();
      sort_entries<false>(keys, nullptr, n2);
      int run = 0;
#pragma unroll 1
      for (int i0 = 0; i0 < r.m; i0 += kStepThreads) {
        const int i = i0 + threadIdx.x;
        int chunk;
        const int pos = run + scan.sum(i < r.m ? cnt[session_of_key(keys[i])] : 0, &chunk);
        if (i < r.m) off[i] = pos;
        run += chunk;
      }
    }
  }
  __syncthreads();
  return r;
}

// Writes the victims of the selected sessions.
__device__ void emit_selected(const DevPool& p, const Selected& sel, const unsigned long long* keys,
                              const int* off, const int* nblk, const int* cnt, const VictimList& l,
                              OwnerCheck& check, StepShared& sh, BlockScan& scan) {
  if (LV_MOSTLY(sel.m <= 2 && !sel.sorted)) {
#pragma unroll 1
    for (int r = 0; r < sel.m; ++r) {
      const int32_t s = sh.sel_sid[r];
      const int at = sh.sel_off[r];
      emit_whole(p, s, nblk[s], at, min(at + cnt[s], l.n_out), l, check, scan);
    }
  } else if (sel.sorted) {
    emit_warp(p, nblk, cnt, sel.m, l, check, [&](int r) { return make_int2(session_of_key(keys[r]), off[r]); });
  } else {
    emit_warp(p, nblk, cnt, sel.m, l, check, [&](int r) { return make_int2(sh.sel_sid[r], sh.sel_off[r]); });
  }
}

// The states of 32 consecutive sessions (of `left` that there are), one per lane: read by the
// warp as whole lines through its buffer in shared memory.  (Read by each lane for itself,
// 72 bytes apart, every load touches 32 sectors: 3.4 us for 1000 sessions.)
__device__ __forceinline__ lv_session_state load_states(const lv_session_state* q, int left, long long* buf) {
  static_assert(sizeof(lv_session_state) == 72, "nine words");
  const int lane = threadIdx.x & 31;
  const int words = 9 * (left < 32 ? left : 32);
  long long w[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    w[i] = 0;
    if (i * 32 + lane < words) w[i] = reinterpret_cast<const long long*>(q)[i * 32 + lane];
  }
  __syncwarp();                  // the buffer's last reads are over
#pragma unroll
  for (int i = 0; i < 9; ++i) buf[i * 32 + lane] = w[i];
  __syncwarp();
  union {
    lv_session_state st;
    long long w[9];
  } u;
#pragma unroll
  for (int i = 0; i < 9; ++i) u.w[i] = buf[lane * 9 + i];
  return u.st;
}

__global__ void __launch_bounds__(kStepThreads, 1)
k_step(DevPool p, StepArgs a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ StepShared sh;
  pdl_entry();
  const int tid = threadIdx.x, lane = tid & 31;
  const StepLayout lay = step_layout(p, a.keys != nullptr && a.part == kStepAll, a.copy_bits != 0);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(dyn);
  int* off = reinterpret_cast<int*>(dyn + lay.off);
  int* cnt = reinterpret_cast<int*>(dyn + lay.cnt);
  int* away = reinterpret_cast<int*>(dyn + lay.away);
  int* nblk = reinterpret_cast<int*>(dyn + lay.nb);
  BlockScan scan{sh.ws, 0};
  long long* R = a.rs.words;
  const bool evict = a.evict >= 0;

  // reads that depend on nothing: the candidates, bitmaps, every session's state (whole,
  // before anything is decided from it) and counts
  const bool picks = a.turn && a.sid < 0 && a.part != kStepMove;
  int32_t first_cand = -1;
  if (picks && tid < a.n_cand) first_cand = a.cand[tid];
  uint32_t* copy = a.copy_bits && a.part != kStepList ? reinterpret_cast<uint32_t*>(dyn + lay.bits) : nullptr;
  // (the few words of a small pool by warps that have no states to read, each tier's by others:
  // eight sessions 19.1 us a turn so, 19.4 when the first warp reads all three one after the other)
  const TierBits hbm = bits_copy(p.bits_hbm, p.hbm_pages, copy, kStepThreads - 1 - tid);
  const TierBits host = bits_copy(p.bits_host, p.host_pages, copy ? copy + 2 * ((p.hbm_pages + 31) >> 5) : nullptr,
                                  tid ^ (kStepThreads / 2));
  const bool fallback = !evict && !a.preload;
#pragma unroll 1
  for (int s0 = tid & ~31; s0 < p.S; s0 += kStepThreads) {      // 32 sessions of a warp
    const int x = s0 + lane;
    const int2 c = x < p.S ? p.cnt[x] : make_int2(0, 0);
    const lv_session_state st = load_states(p.sess + s0, p.S - s0, sh.states[tid >> 5]);
    if (x < p.S) {
      cnt[x] = c.x;
      away[x] = c.y;
      nblk[x] = blocks_of_context(p, st.ctx_tokens);
      keys[x] = c.x > 0 ? session_key(p, st, x, a.now_us, fallback) : 0ull;
    }
  }
  const int part = __reduce_add_sync(0xffffffffu, hbm.taken);
  if (lane == 0) sh.taken[tid >> 5] = part;
  if (tid == 0) R[R_CURSOR] = 0;
  __syncthreads();
  const int hbm_alloc = __reduce_add_sync(0xffffffffu, lane < kStepWarps ? sh.taken[lane] : 0);

  // the session: given, picked (the first candidate with a host-tier block, else the first), or none
  int32_t sid = a.sid;
  if (LV_RARE(a.part == kStepMove)) {
    sid = (int32_t)R[R_SID];
  } else if (picks) {
    if (tid == 0) sh.pick[kStepWarps] = make_int2(0, first_cand);
    unsigned c = 0x7fffffffu;
    int32_t s = -1;
#pragma unroll 1
    for (int i = tid; i < a.n_cand; i += kStepThreads) {
      const int32_t x = i == tid ? first_cand : a.cand[i];
      if (x >= 0 && x < p.S && away[x] > 0) {
        c = (unsigned)i;
        s = x;
        break;
      }
    }
    __syncwarp();
    const unsigned low = __reduce_min_sync(0xffffffffu, c);
    if (c == low && (low != 0x7fffffffu || lane == 0)) sh.pick[tid >> 5] = make_int2((int)low, s);
    __syncthreads();
    const int2 w = lane < kStepWarps ? sh.pick[lane] : make_int2(0x7fffffff, -1);
    const unsigned first = __reduce_min_sync(0xffffffffu, (unsigned)w.x);
    if (LV_MOSTLY(first != 0x7fffffffu)) {
      const unsigned who = __ballot_sync(0xffffffffu, (unsigned)w.x == first);
      sid = __shfl_sync(0xffffffffu, w.y, __ffs(who) - 1);
    } else {
      sid = sh.pick[kStepWarps].y;
      if (sid < 0 || sid >= p.S) {
        if (tid == 0) set_error(p.ctl, LV_ERR_BOUNDS, 0);
        sid = -1;
      }
    }
  }
  const bool have = sid >= 0 && sid < p.S;      // lv_evict has no session; a failed pick neither
  const int32_t ctx = have ? p.sess[sid].ctx_tokens : 0;
  int32_t flags = 0;                            // the turn's session's, in thread 0
  if (a.turn && have && tid == 0) {
    flags = p.sess[sid].flags;
    if (a.part != kStepMove) {
      // LV_EV_TURN_BEGIN; only the fields it changes are written (others read this state now)
      lv_session_state st{};
      st.flags = flags;
      lv_event x{};
      x.kind = LV_EV_TURN_BEGIN;
      x.sid = sid;
      x.t_us = a.now_us;
      apply_event(p, st, x);
      flags = st.flags;
      p.sess[sid].flags = flags;
      p.sess[sid].protect_until_us = st.protect_until_us;
      p.sess[sid].last_use_us = st.last_use_us;
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_EVENTS]), 1ull);
    }
  }

  // the session's host-tier blocks, in load order
  int status = evict || have ? LV_RESIDENT_DONE : LV_RESIDENT_FAILED;
  long long nh = 0, new_blocks = 0, k = 0;
  const int32_t* blks = a.keys ? a.rs.loads : a.rs.blocks;
  const int32_t* gslot = nullptr;
  OwnerCheck out_check{0, 0, -1, -1}, in_check{0, 0, -1, -1};
  if (!evict && have) {
    const int32_t nb = nblk[sid];
    const uint32_t nctx = (uint32_t)ctx + (uint32_t)a.append_tokens;
    // (nctx past 2^31 is refused anyway: its block count only has to be defined)
    const long long nnb = nctx > 0x7fffffffu ? 0 : (nctx + (uint32_t)p.T - 1u) / (uint32_t)p.T;
    const bool over = nnb > p.maxB || nctx > 0x7fffffffu;
    new_blocks = nnb - nb;
    if (LV_RARE(a.part == kStepMove)) {
      nh = R[R_N_IN];
#pragma unroll 1
      for (long long i = tid; i < nh; i += kStepThreads) {
        // (the order was made by another kernel, from keys read more than once: each block once)
        const int32_t b = a.rs.loads[i];
        const size_t ti = (size_t)sid * p.maxB + b;
        long long h = -1;
        if (b >= 0 && b < nb && atomicExch(&p.mark[ti], a.epoch) != a.epoch) h = -(long long)p.table[ti] - 2;
        in_check.read(p.own_host, h, p.host_pages);
        in_check.expect(owner_key(sid, b), i);
      }
    } else if (away[sid] > 0) {
      const int32_t* row = p.table + (size_t)sid * p.maxB;
#pragma unroll 1
      for (int32_t q0 = 0; q0 < nb; q0 += kStepThreads) {
        const int32_t b = q0 + tid;
        const int32_t e = b < nb ? row[b] : -1;
        const long long h = -(long long)e - 2;
        in_check.read(p.own_host, h, p.host_pages);     // (h < 0 where there is no slot)
        int chunk;
        const long long pos = nh + scan.rank(e <= -2, &chunk);
        if (e <= -2) {
          if (LV_MOSTLY(pos < kStepItems)) {
            sh.l.blks[pos] = b;
            sh.l.gslot[pos] = (int32_t)h;
          }
          a.rs.blocks[pos] = b;
          in_check.expect(owner_key(sid, b), pos);
        }
        nh += chunk;
      }
      __syncthreads();
      if (LV_MOSTLY(nh <= kStepItems)) {
        if (LV_RARE(a.keys && a.part == kStepAll)) {
          // the caller's order: ascending (key, block id); the list is in block order already
          unsigned long long* lk = reinterpret_cast<unsigned long long*>(dyn + lay.load);
          int* li = reinterpret_cast<int*>(lk + kStepItems);
          if (nh <= kCountedLoads) {
            // few: a warp per load counts the loads before it
#pragma unroll 1
            for (int i = tid; i < nh; i += kStepThreads) lk[i] = a.keys[sh.l.blks[i]];
            __syncthreads();
#pragma unroll 1
            for (int i = tid >> 5; i < nh; i += kStepWarps) {
              const unsigned long long ki = lk[i];
              int before = 0;
#pragma unroll 1
              for (int j = lane; j < nh; j += 32) before += lk[j] < ki || (lk[j] == ki && j < i) ? 1 : 0;
              before = __reduce_add_sync(0xffffffffu, before);
              if (lane == 0) li[before] = i;
            }
            __syncthreads();
          } else {
            int n = 2 * kCountedLoads;
#pragma unroll 1
            while (n < nh) n *= 2;
#pragma unroll 1
            for (int i = tid; i < n; i += kStepThreads) {
              lk[i] = i < nh ? a.keys[sh.l.blks[i]] : ~0ull;
              li[i] = i;
            }
            __syncthreads();
            sort_entries<true>(lk, li, n);
          }
          constexpr int kEach = kStepItems / kStepThreads;
          int32_t b[kEach], g[kEach];
#pragma unroll
          for (int u = 0; u < kEach; ++u) {
            const int i = tid + u * kStepThreads;
            if (i < nh) {
              b[u] = sh.l.blks[li[i]];
              g[u] = sh.l.gslot[li[i]];
            }
          }
          __syncthreads();
#pragma unroll
          for (int u = 0; u < kEach; ++u) {
            const int i = tid + u * kStepThreads;
            if (i < nh) {
              sh.l.blks[i] = b[u];
              sh.l.gslot[i] = g[u];
              a.rs.loads[i] = b[u];
            }
          }
          __syncthreads();
        }
        blks = sh.l.blks;
        gslot = sh.l.gslot;
      }
    }
    if (LV_RARE(over)) {
      if (tid == 0 && a.part != kStepMove) set_error(p.ctl, LV_ERR_BOUNDS, sid);
      status = LV_RESIDENT_FAILED;
    } else {
      const long long need = nh + new_blocks, free_pages = p.budget - hbm_alloc;
      k = need - free_pages > 0 ? need - free_pages : 0;
      if (a.preload && nh == 0) status = LV_RESIDENT_NOTHING;
      else if (a.preload && a.max_load >= 0 && nh > a.max_load) status = LV_RESIDENT_SKIPPED;
      if (LV_RARE(status == LV_RESIDENT_SKIPPED) && tid == 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PRELOADS_SKIPPED]), 1ull);
    }
  }
  if (LV_RARE(a.part == kStepList)) {
    if (tid == 0) {
      R[R_SID] = sid;
      R[R_N_IN] = nh;
    }
    return;
  }
  if (evict) k = a.evict;
  const bool go = status == LV_RESIDENT_DONE;
  const long long want = go ? k : 0;            // victims asked for

  Selected sel{};
  // the turn's session is RUNNING by now: never a victim
  if (want > 0) sel = select_sessions(p, keys, off, cnt, want, a.turn ? sid : -1, sh, scan);
  if (tid == 0) {
    p.ctl[C_SEL_COUNT] = sel.n_out;
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_SELECTS]), 1ull);
    if (!evict && !a.preload) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_FALLBACK]), 1ull);
    if (want > 0) {
      p.ctl[C_SEL_TOTAL] = sel.total;
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_VICTIMS]), (unsigned long long)sel.n_out);
      if (sel.total < want) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_SHORTFALLS]), 1ull);
    }
  }
  // the victims of the order's first n_out positions
  lv_victim* near = sel.n_out <= kStepItems ? sh.l.v : nullptr;
  const VictimList list{near, a.rs.victims, p.own_hbm, p.hbm_pages, (int)sel.n_out};
  emit_selected(p, sel, keys, off, nblk, cnt, list, out_check, sh, scan);
  // the gate: a shortfall stops the step (a preload is skipped, a foreground turn fails);
  // lv_evict takes what there is
  long long n_out = sel.n_out, n_in = go ? nh : 0;
  bool grow = go;
  if (evict) {
    if (n_out == 0) status = LV_RESIDENT_NOTHING;
    grow = false;
  } else if (LV_RARE(go && sel.n_out < k)) {
    if (a.preload) {
      status = LV_RESIDENT_SKIPPED;
      if (tid == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PRELOADS_SKIPPED]), 1ull);
    } else {
      status = LV_RESIDENT_FAILED;
      if (tid == 0) set_error(p.ctl, LV_ERR_NO_HBM, k);
    }
    n_out = n_in = 0;
    grow = false;
  }
  __syncthreads();                              // the victims are listed
  MovePlan m{near ? near : a.rs.victims, n_out, sid, blks, gslot, n_in, near ? sh.l.slots : a.rs.slots,
             n_in <= kStepItems ? sh.l.pages : a.rs.pages, a.rs.slots, a.rs.pages, a.rs.tasks,
             R + R_N_TASKS, a.epoch, p.page_tag};
  out_check.settle();
  in_check.settle();
  const bool planned =
      plan_moves<false>(p, m, hbm, host, hbm_alloc, out_check.bad, in_check.bad, sh, scan);
  if (LV_MOSTLY(planned && n_out > 0)) {
    // the victims' sessions: fewer blocks in HBM, more in the host tier
#pragma unroll 1
    for (int r = tid; r < sel.m; r += kStepThreads) {
      const int32_t s = sel.sorted ? session_of_key(keys[r]) : sh.sel_sid[r];
      const long long at = sel.sorted ? off[r] : sh.sel_off[r];
      const int take = (int)(n_out - at < cnt[s] ? n_out - at : cnt[s]);
      add_counts(counts_of(p, s), -take, take);
    }
  }
  long long appended = 0;
  if (LV_RARE(grow && a.append_tokens > 0)) {
    __syncthreads();                            // the commits of the plan
    appended = append_tokens_to(p, sid, ctx, a.append_tokens, a.rs.append, hbm, host, sh.l.pages, scan, sh.base);
    if (appended < 0) appended = 0;
  }
  __syncthreads();
  bits_back(hbm);
  bits_back(host);
  if (tid != 0) return;
  // the step's end: LV_EV_TURN_END unless the turn failed, a completed preload's protection,
  // and the result
  if (a.turn && have && status != LV_RESIDENT_FAILED) {
    lv_session_state st{};
    st.flags = flags;
    lv_event x{};
    x.kind = LV_EV_TURN_END;
    x.sid = sid;
    x.t_us = a.now_us;
    x.a = a.audio_us;
    x.b = a.units;
    apply_event(p, st, x);
    lv_session_state& to = p.sess[sid];
    to.flags = st.flags;
    to.gen_us = st.gen_us;
    to.play_us = st.play_us;
    to.reply_tokens = st.reply_tokens;
    to.last_use_us = st.last_use_us;
    if (st.flags & LV_DONE_VALID) to.t_done_us = st.t_done_us;
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_EVENTS]), 1ull);
  }
  if (a.preload && status == LV_RESIDENT_DONE) {
    p.sess[sid].protect_until_us = a.now_us + p.protect_us;   // warmed KV (Section 5.2)
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_PRELOADS]), 1ull);
  }
  if (a.out) {
    lv_resident_result r;
    r.k = k;
    r.n_found = go ? sel.n_out : 0;
    r.n_victims = n_out;
    r.n_loaded = n_in;
    r.n_appended = appended;
    r.status = status;
    r.sid = sid;
    *a.out = r;
  }
}

// ------------------------------------------------------ ranking by itself
// lv_select_victims for up to kSelectMost victims: one kernel.  The keys of kStepThreads
// sessions are made by each CTA of a cluster and written into the first CTA's shared memory,
// which then selects and lists the victims; it reads one count per session and the rows of
// the sessions chosen, where the census reads every row.  kCensus: no counts are kept for
// these tables (lv_select_victims_noalloc, many sessions); one CTA takes both from the census.
// 256 victims of 1024 sessions with 1024 blocks each: 7.1 us as census and emission, 3.9 as
// one kernel; 1500 of 4096 sessions with 256 blocks: 20.7 and 7.8 us.
// More victims, or victims of some hundred sessions, are written by many CTAs: 4096 victims
// of 1024 sessions take 11.8 us here and 9.2 there, 2048 of at least 1024 sessions with two
// blocks each 32 and 9.2, 256 of 128 such sessions 10.1 and 9.2 (13.1 and 14.9 with 4096
// sessions).
constexpr int kSelectMost = 2048;
constexpr int kSelectSessions = 128;   // k victims are blocks of k / maxB sessions at least

struct SelectLayout {
  int n2;
  size_t off, cnt, nb, total;
};
__host__ __device__ inline SelectLayout select_layout(int S) {
  SelectLayout l{};
  l.n2 = 32;
  while (l.n2 < S) l.n2 *= 2;
  l.off = (size_t)l.n2 * 8;
  l.cnt = l.off + (size_t)l.n2 * 4;
  l.nb = l.cnt + (size_t)l.n2 * 4;
  l.total = l.nb + (size_t)l.n2 * 4;
  return l;
}

template <bool kCensus>
__global__ void __launch_bounds__(kStepThreads, 1)
k_select(DevPool p, long long now_us, long long k, bool fallback, long long* count_dev, lv_victim* out) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ StepShared sh;
  pdl_entry();
  const int tid = threadIdx.x;
  const SelectLayout lay = select_layout(p.S);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(dyn);
  int* off = reinterpret_cast<int*>(dyn + lay.off);
  int* cnt = reinterpret_cast<int*>(dyn + lay.cnt);
  int* nblk = reinterpret_cast<int*>(dyn + lay.nb);
  BlockScan scan{sh.ws, 0};
  if (kCensus) {
    for (int s = tid; s < p.S; s += kStepThreads) {
      const int c = p.scount[s];
      cnt[s] = c;
      keys[s] = c > 0 ? p.skey[s] : 0ull;
      nblk[s] = nblocks_of(p, s);
    }
    __syncthreads();
  } else {
    cg::cluster_group cluster = cg::this_cluster();
    // every CTA says that it runs; nobody writes into the first one before all have said so
    // (the reads of the states lie between, so the wait costs nothing)
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    const int x = blockIdx.x * kStepThreads + tid, s0 = x & ~31;
    unsigned long long key = 0ull;
    int c = 0, nb = 0;
    if (s0 < p.S) {
      if (x < p.S) c = p.cnt[x].x;
      const lv_session_state st = load_states(p.sess + s0, p.S - s0, sh.states[tid >> 5]);
      if (x < p.S) {
        if (c > 0) key = session_key(p, st, x, now_us, fallback);
        nb = blocks_of_context(p, st.ctx_tokens);
      }
    }
    asm volatile("barrier.cluster.wait;" ::: "memory");
    if (x < p.S) {
      cluster.map_shared_rank(keys, 0)[x] = key;
      cluster.map_shared_rank(cnt, 0)[x] = c;
      cluster.map_shared_rank(nblk, 0)[x] = nb;
    }
    cluster.sync();
    if (blockIdx.x > 0) return;
  }
  const Selected sel = select_sessions(p, keys, off, cnt, k, -1, sh, scan);
  OwnerCheck check{0, 0, -1, -1};
  const VictimList list{nullptr, out, nullptr, 0, (int)sel.n_out};
  emit_selected(p, sel, keys, off, nblk, cnt, list, check, sh, scan);
  if (tid == 0) {
    p.ctl[C_SEL_COUNT] = sel.n_out;
    p.ctl[C_SEL_TOTAL] = sel.total;
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_SELECTS]), 1ull);
    atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_VICTIMS]), (unsigned long long)sel.n_out);
    if (sel.total < k) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_SHORTFALLS]), 1ull);
    if (fallback) atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl[C_FALLBACK]), 1ull);
    if (count_dev) *count_dev = sel.n_out;
  }
}

constexpr int kOrderThreads = 256;

// The caller's load order where a session may have more host-tier blocks than k_step sorts
// in shared memory: host-tier block i of the session (ascending in `blocks`, R[R_N_IN] of
// them) goes to position #{j : (key[b_j], b_j) < (key[b_i], b_i)} of `loads` -- ascending
// (key, block id).  One warp per block.
__global__ void __launch_bounds__(kOrderThreads)
k_order_loads(const long long* __restrict__ R, const int32_t* __restrict__ blocks,
              const unsigned long long* __restrict__ key, int32_t* __restrict__ loads) {
  pdl_entry();
  const long long nh = R[R_N_IN];
  const long long i = blockIdx.x * (long long)(kOrderThreads / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= nh) return;
  const int32_t bi = blocks[i];
  const unsigned long long ki = key[bi];
  int rank = 0;
  for (long long j = lane; j < nh; j += 32) {
    const int32_t bj = blocks[j];
    const unsigned long long kj = key[bj];
    rank += (kj < ki || (kj == ki && bj < bi)) ? 1 : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
  if (lane == 0) loads[rank] = bi;
}

// ------------------------------------------------------------- checksums
constexpr int kSumThreads = 256;
constexpr int kSumUnroll = 4;
constexpr int kSumBatch = 4;      // sub-pages taken from the cursor at a time

// Unit u = (page i, sub-page j); the sub-page's words are q0 + k (q0 = j*P/8).
// Each thread keeps kSumUnroll 16-byte loads in flight; the per-unit partial sum
// goes to sums[i] with one atomic add (addition mod 2^64 is order-free).
__global__ void __launch_bounds__(kSumThreads)
k_checksum(DevPool p, const int32_t* __restrict__ pages, long long n, unsigned long long* __restrict__ sums,
           unsigned long long* __restrict__ cursor) {
  __shared__ unsigned long long warp_part[kSumThreads / 32];
  __shared__ long long s_next;
  pdl_wait();
  const long long units = n * p.J;
  const int nvec = (int)(p.P >> 4);                   // 16-byte vectors per sub-page
  // units come from a shared cursor, kSumBatch at a time, the next batch fetched while
  // the current one is read: a CTA that starts late (its SM held by other work) takes
  // fewer units instead of holding up the end of the call
  // (thread 0 keeps the fetched index in a register and publishes it only at the end
  // of the batch, so that its warp does not wait for the atomic's result meanwhile)
  // (null: the grid has a CTA for every batch)
  if (threadIdx.x == 0)
    s_next = cursor ? (long long)atomicAdd(cursor, (unsigned long long)kSumBatch) : (long long)blockIdx.x * kSumBatch;
  __syncthreads();
  for (long long b = s_next; b < units; b = s_next) {
    unsigned long long fetched = (unsigned long long)units;
    if (threadIdx.x == 0 && cursor) fetched = atomicAdd(cursor, (unsigned long long)kSumBatch);
    const long long b_end = b + kSumBatch < units ? b + kSumBatch : units;
    for (long long u = b; u < b_end; ++u) {
      const long long i = u / p.J;
      const int j = (int)(u % p.J);
      const int32_t pg = pages[i];
      const bool ok = pg >= 0 && pg < p.hbm_pages;
      unsigned long long acc = 0;
      if (ok) {
        const ulonglong2* src = reinterpret_cast<const ulonglong2*>(p.kv[j] + (size_t)pg * p.P);
        const unsigned long long q0 = (unsigned long long)j * (unsigned long long)(p.P >> 3);
        for (int base = threadIdx.x; base < nvec; base += kSumThreads * kSumUnroll) {
          ulonglong2 r[kSumUnroll];
#pragma unroll
          for (int k = 0; k < kSumUnroll; ++k) {
            const int v = base + k * kSumThreads;
            if (v < nvec) r[k] = src[v];
          }
#pragma unroll
          for (int k = 0; k < kSumUnroll; ++k) {
            const int v = base + k * kSumThreads;
            if (v < nvec) {
              const unsigned long long q = q0 + 2ull * (unsigned long long)v;   // word index of r.x
              acc += r[k].x * (2ull * q + 1ull) + r[k].y * (2ull * q + 3ull);
            }
          }
        }
      } else if (j == 0 && threadIdx.x == 0) {
        set_error(p.ctl, LV_ERR_BOUNDS, i);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
      if ((threadIdx.x & 31) == 0) warp_part[threadIdx.x >> 5] = acc;
      __syncthreads();
      if (threadIdx.x == 0) {
        unsigned long long t = 0;
#pragma unroll
        for (int w = 0; w < kSumThreads / 32; ++w) t += warp_part[w];
        if (ok) atomicAdd(&sums[i], t);
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) s_next = (long long)fetched;   // every thread has read b
    __syncthreads();
  }
}

// ----------------------------------------------------------------- views
__global__ void __launch_bounds__(kCensusThreads)
k_counts(DevPool p, int32_t* __restrict__ hbm, int32_t* __restrict__ host) {
  const int32_t s = blockIdx.x;
  const int32_t nb = nblocks_of(p, s);
  const int32_t* row = p.table + (size_t)s * p.maxB;
  long long a = 0, h = 0;
  for (int32_t b = threadIdx.x; b < nb; b += kCensusThreads) {
    const int32_t e = row[b];
    a += e >= 0;
    h += e <= -2;
  }
  long long ta, th;
  block_excl_scan<kCensusThreads>(a, &ta);
  block_excl_scan<kCensusThreads>(h, &th);
  if (threadIdx.x == 0) {
    if (hbm) hbm[s] = (int32_t)ta;
    if (host) host[s] = (int32_t)th;
  }
}

__global__ void __launch_bounds__(kStepThreads)
k_blocks(DevPool p, int32_t sid, int32_t where, int32_t* out, long long* count) {
  __shared__ int ws[2 * kStepWarps];
  __shared__ int32_t blocks;
  pdl_entry();
  BlockScan scan{ws, 0};
  // (by one thread: growth on another stream may change it, and it says how many barriers follow)
  if (threadIdx.x == 0) blocks = nblocks_of(p, sid);
  __syncthreads();
  const int32_t nb = blocks;
  const int32_t* row = p.table + (size_t)sid * p.maxB;
  int run = 0;
#pragma unroll 1
  for (int32_t q0 = 0; q0 < nb; q0 += kStepThreads) {
    const int32_t b = q0 + threadIdx.x;
    const int32_t e = b < nb ? row[b] : -1;
    const bool in = where == 0 ? e >= 0 : e <= -2;
    int chunk;
    const int pos = run + scan.rank(in, &chunk);
    if (in) out[pos] = b;
    run += chunk;
  }
  if (threadIdx.x == 0 && count) *count = run;
}

inline unsigned blocks_for(long long n, int threads, long long cap) {
  long long b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

}  // namespace

// ======================================================== launch wrappers
cudaError_t launch_import(const DevPool& p, const int32_t* placement, const int32_t* ctx,
                          cudaStream_t s) {
  k_import<<<blocks_for((long long)p.S * p.maxB, 256, 4096), 256, 0, s>>>(p, placement, ctx);
  return cudaGetLastError();
}

cudaError_t launch_check_budget(const DevPool& p, cudaStream_t s) {
  k_check_budget<<<1, 1, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_session_set(const DevPool& p, const lv_session_state* in, int32_t first,
                               int32_t n, cudaStream_t s) {
  k_session_set<<<blocks_for(n, 256, 1 << 20), 256, 0, s>>>(p, in, first, n);
  return cudaGetLastError();
}

// A launch that lets the kernel be scheduled while the previous kernel on `s`
// still runs; the kernel must call pdl_entry() or pdl_wait() before it reads anything that
// changes after the pool's creation.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem,
                       cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

cudaError_t launch_events(const DevPool& p, const lv_event* ev, int64_t n, cudaStream_t s) {
  return launch_pdl(k_events, blocks_for(p.S, kEventThreads, 1 << 20), kEventThreads, 0, s, p, ev, (long long)n);
}

// One kernel up to kSelectMost victims; more are written by a CTA per session.  Where no
// counts are kept the census comes first, and up to kEmitScanMax sessions the CTAs that then
// write place their own session: 1890 victims of 25 sessions 8.4 us so, 10.0 by one CTA after
// the census, 256 of 1024 sessions 11.6 and 12.6; above, a third kernel would place them: 256
// of 2048 sessions 13.8 us so and 12.6 by one CTA, of 4096 18.2 and 12.9.
cudaError_t launch_select(const DevPool& p, int64_t now_us, int64_t k, bool fallback,
                          lv_victim* out, long long* count_dev, cudaStream_t s) {
  const size_t smem = select_layout(p.S).total;
  const bool one = k <= kSelectMost && k <= (long long)kSelectSessions * p.maxB && (p.cnt || p.S > kEmitScanMax);
  if (one && p.cnt) {
    unsigned ctas = 1;
    while ((int)ctas * kStepThreads < p.S) ctas *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kStepThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = ctas;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = ctas > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k_select<false>, p, (long long)now_us, (long long)k, fallback, count_dev, out);
  }
  const bool by_warp = p.maxB <= 1024;
  cudaError_t e = by_warp ? launch_pdl(k_rank_census<32>, blocks_for(p.S, kCensusThreads / 32, 1 << 20), kCensusThreads,
                                       0, s, p, (long long)now_us, fallback)
                          : launch_pdl(k_rank_census<kCensusThreads>, (unsigned)p.S, kCensusThreads, 0, s, p,
                                       (long long)now_us, fallback);
  if (e != cudaSuccess) return e;
  if (one) {
    e = cudaFuncSetAttribute(k_select<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)select_layout(4096).total);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_select<true>, 1, kStepThreads, smem, s, p, (long long)now_us, (long long)k, fallback, count_dev,
                      out);
  }
  if (p.S > kEmitScanMax) {
    const dim3 grid((unsigned)((p.S + kPrefixTile - 1) / kPrefixTile),
                    (unsigned)((p.S + kPrefixChunk - 1) / kPrefixChunk));
    e = launch_pdl(k_rank_prefix, grid, kPrefixTile, 0, s, p);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(k_rank_emit, (unsigned)p.S, kEmitThreads, 0, s, p, (long long)k, fallback, count_dev, out);
}

// The largest dynamic shared memory of the one-CTA kernels beside their static lists.
constexpr size_t kStepDynamic = 180 * 1024;

cudaError_t launch_alloc(const DevPool& p, bool in_hbm, const lv_victim* v, int64_t n, int32_t* out,
                         cudaStream_t s, bool injected_fail) {
  if (n <= 0) return cudaSuccess;
  const size_t smem = 8 * (size_t)(((in_hbm ? p.hbm_pages : p.host_pages) + 31) >> 5);
  const bool fit = smem <= kStepDynamic;
  return launch_pdl(k_alloc, 1, kStepThreads, fit ? smem : 0, s, p, in_hbm, p.incl ? v : nullptr, (long long)n, out,
                    injected_fail, fit ? 1 : 0);
}

cudaError_t launch_swap_out(const DevPool& p, const lv_victim* v, const int32_t* slots, int64_t n,
                            lv_remap_entry* commit, cudaStream_t s, int num_sms, const EventPair* ev) {
  const long long units = (long long)n * p.J;
  if (ev) cudaEventRecord(ev->start, s);
  const cudaError_t e = launch_pdl(k_swap_out, blocks_for(units, 1, (long long)num_sms * 8), kCopyThreads, 0, s, p, v,
                                   slots, (long long)n, commit);
  if (ev) cudaEventRecord(ev->end, s);
  return e;
}

cudaError_t launch_swap_in(const DevPool& p, int32_t sid, const int32_t* blks, const int32_t* pages,
                           int64_t n, lv_remap_entry* commit, cudaStream_t s, int num_sms,
                           const EventPair* ev) {
  const long long units = (long long)n * p.J;
  if (ev) cudaEventRecord(ev->start, s);
  const cudaError_t e = launch_pdl(k_swap_in, blocks_for(units, 1, (long long)num_sms * 8), kCopyThreads, 0, s, p, sid,
                                   blks, pages, (long long)n, commit);
  if (ev) cudaEventRecord(ev->end, s);
  return e;
}

bool bits_fit(const DevPool& p, size_t others) {
  return others + bits_words(p) * 4 <= kStepDynamic;
}

cudaError_t configure_step_kernels() {
  cudaError_t e = cudaFuncSetAttribute(k_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepDynamic);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_alloc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepDynamic);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_append, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepDynamic);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_select<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)select_layout(4096).total);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_exchange_plan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepDynamic);
}

cudaError_t launch_exchange_plan(const DevPool& p, const lv_victim* v, int64_t n_out, int32_t sid,
                                 const int32_t* blks, int64_t n_in, int32_t* slots, int32_t* pages,
                                 int4* tasks, long long* n_tasks, int32_t epoch,
                                 unsigned long long* page_tag, cudaStream_t s, long long* cursor) {
  const bool fit = bits_fit(p, 0);
  const size_t smem = fit ? bits_words(p) * 4 : 0;
  return launch_pdl(k_exchange_plan, 1, kStepThreads, smem, s, p, v, (long long)n_out, sid, blks,
                    (long long)n_in, slots, pages, tasks, n_tasks, epoch, page_tag, cursor, fit ? 1 : 0);
}

// The copy of a plan's tasks (at most max_pages of them), on s or, with `off`, on the copy
// stream after everything queued on s.
static cudaError_t launch_copy(const DevPool& p, const int4* tasks, const long long* n_tasks,
                               long long* cursor, long long max_pages, cudaStream_t s, int copy_ctas,
                               const EventPair* ev, const CopyOffload* off) {
  cudaStream_t cs = s;
  if (off) {
    cudaError_t e = cudaEventRecord(off->planned, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(off->stream, off->planned, 0);
    if (e != cudaSuccess) return e;
    cs = off->stream;
  }
  if (ev) cudaEventRecord(ev->start, cs);
  else if (off && off->started) cudaEventRecord(off->started, cs);
  // the 16-byte copy takes whole pages in chunks, the TMA copy sub-pages
  const unsigned grid = blocks_for(max_pages * (p.xstages > 0 ? p.J : copy_chunks(p)), 1, copy_ctas);
  cudaError_t le = cudaSuccess;
  if (p.xstages > 0) {
    const size_t smem = (size_t)p.xstages * 2 * p.P;
    if (off || ev) k_exchange_copy_tma<<<grid, kStageThreads, smem, cs>>>(p, tasks, n_tasks, cursor);
    else le = launch_pdl(k_exchange_copy_tma, grid, kStageThreads, smem, cs, p, tasks, n_tasks, cursor);
  } else if (off || ev) {   // after an event wait or record: an ordinary launch
    k_exchange_copy<<<grid, kCopyThreads, 0, cs>>>(p, tasks, n_tasks, cursor);
  } else {
    le = launch_pdl(k_exchange_copy, grid, kCopyThreads, 0, cs, p, tasks, n_tasks, cursor);
  }
  if (le != cudaSuccess) return le;
  if (ev) cudaEventRecord(ev->end, cs);
  else if (off && off->finished) cudaEventRecord(off->finished, cs);
  if (off) {
    const cudaError_t e = cudaEventRecord(off->copied, cs);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_exchange(const DevPool& p, const lv_victim* v, int64_t n_out, int32_t sid,
                            const int32_t* blks, int64_t n_in, int32_t* slots, int32_t* pages,
                            int4* tasks, long long* n_tasks, int32_t epoch,
                            unsigned long long* page_tag, cudaStream_t s, int copy_ctas,
                            const EventPair* ev, long long* cursor) {
  const cudaError_t e = launch_exchange_plan(p, v, n_out, sid, blks, n_in, slots, pages, tasks, n_tasks,
                                             epoch, page_tag, s, cursor);
  if (e != cudaSuccess) return e;
  return launch_copy(p, tasks, n_tasks, cursor, n_out + n_in, s, copy_ctas, ev, nullptr);
}

cudaError_t launch_step(const DevPool& p, const ResidentScratch& rs, const StepCall& c, int32_t epoch,
                        cudaStream_t s, int copy_ctas, const EventPair* ev, const CopyOffload* off) {
  StepArgs a{};
  a.rs = rs;
  a.sid = c.sid;
  a.cand = c.cand;
  a.n_cand = c.n_cand;
  a.keys = c.load_keys;
  a.now_us = c.now_us;
  a.audio_us = c.audio_us;
  a.units = c.units;
  a.max_load = c.max_load;
  a.evict = c.evict;
  a.append_tokens = c.append_tokens;
  a.epoch = epoch;
  a.turn = c.turn;
  a.preload = c.preload;
  a.out = c.out;
  // up to kStepItems loads are ordered inside the step; a session that may have more takes
  // the grid-wide ordering kernel between two parts of it (one warp per block: n^2
  // comparisons over the whole GPU instead of over one CTA)
  const bool split = c.load_keys && p.maxB > kStepItems;
  a.copy_bits = bits_fit(p, step_layout(p, c.load_keys && !split, false).total) ? 1 : 0;
  a.part = split ? kStepList : kStepAll;
  const size_t smem = step_layout(p, c.load_keys && !split, a.copy_bits != 0).total;
  cudaError_t e = launch_pdl(k_step, 1, kStepThreads, smem, s, p, a);
  if (e != cudaSuccess) return e;
  if (split) {
    e = launch_pdl(k_order_loads, blocks_for(p.maxB, kOrderThreads / 32, 1ll << 30), kOrderThreads, 0, s,
                   (const long long*)rs.words, (const int32_t*)rs.blocks, c.load_keys, rs.loads);
    if (e != cudaSuccess) return e;
    a.part = kStepMove;
    e = launch_pdl(k_step, 1, kStepThreads, smem, s, p, a);
    if (e != cudaSuccess) return e;
  }
  const long long most = c.evict >= 0 ? (long long)p.budget : (long long)p.budget + p.maxB;
  return launch_copy(p, rs.tasks, rs.words + R_N_TASKS, rs.words + R_CURSOR, most, s, copy_ctas, ev, off);
}

// Zeroes `words` 32-bit words at q, which may be device memory or the device alias of
// mapped page-locked host memory (a kernel, so that either works), and *cursor.
__global__ void k_zero(uint32_t* __restrict__ q, long long words, unsigned long long* cursor) {
  pdl_entry();
  if (cursor && blockIdx.x == 0 && threadIdx.x == 0) *cursor = 0ull;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < words;
       i += (long long)gridDim.x * blockDim.x)
    q[i] = 0u;
}

cudaError_t launch_zero(void* q, int64_t bytes, cudaStream_t s) {
  const long long words = (long long)(bytes / 4);
  if (words <= 0) return cudaSuccess;
  return launch_pdl(k_zero, blocks_for(words, 256, 1024), 256, 0, s, static_cast<uint32_t*>(q), words,
                    (unsigned long long*)nullptr);
}

bool checksums_need_cursor(const DevPool& p, int64_t n, int ctas) { return n * (long long)p.J > (long long)ctas * kSumBatch; }

cudaError_t launch_checksums(const DevPool& p, const int32_t* pages, int64_t n,
                             unsigned long long* sums, unsigned long long* cursor, cudaStream_t s,
                             int ctas) {
  if (n <= 0) return cudaSuccess;
  const long long words = 2 * (long long)n;
  const cudaError_t e = launch_pdl(k_zero, blocks_for(words, 256, 1024), 256, 0, s, reinterpret_cast<uint32_t*>(sums),
                                   words, cursor);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_checksum, blocks_for((n * (long long)p.J + kSumBatch - 1) / kSumBatch, 1, ctas), kSumThreads, 0, s, p,
                    pages, (long long)n, sums, cursor);
}

cudaError_t launch_selftest_wait(const DevPool& p, long long limit_ns, cudaStream_t s) {
  k_selftest_wait<<<1, 32, 0, s>>>(p.ctl, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_tasks_out(const DevPool& p, const lv_victim* v, const int32_t* slots, int64_t n,
                             int4* tasks, lv_remap_entry* commit, cudaStream_t s) {
  k_tasks_out<<<blocks_for(n, 256, 1ll << 30), 256, 0, s>>>(p, v, slots, n, tasks, commit);
  return cudaGetLastError();
}

cudaError_t launch_tasks_in(const DevPool& p, int32_t sid, const int32_t* blks, const int32_t* pages,
                            int64_t n, int4* tasks, lv_remap_entry* commit, cudaStream_t s) {
  k_tasks_in<<<blocks_for(n, 256, 1ll << 30), 256, 0, s>>>(p, sid, blks, pages, n, tasks, commit);
  return cudaGetLastError();
}

// About 48 KiB of stages per CTA, two CTAs per SM: on GB300 three 16 KiB stages per CTA
// moved 4096 scattered thinker pages at 6.82-6.94 TB/s (read + write), against 6.2-6.4
// with eight stages and one CTA per SM, and 5.5 with two stages.
int stage_count(const DevPool& p) {
  int st = p.stages > 0 ? p.stages : (int)((48 * 1024) / p.P);
  if (st < 3) st = 3;
  if (st > kMaxStages) st = kMaxStages;
  if ((long long)st * p.P > 227 * 1024) st = (int)((227 * 1024) / p.P);
  return st < 2 ? 2 : st;
}

// Pools of different sub-page sizes share these kernels: the limit is set to what the largest
// stages may take, never down to what one pool needs.
cudaError_t configure_stage_kernels(const DevPool& p) {
  const int need = stage_count(p) * (int)p.P;
  const int most = 227 * 1024 - 256 > need ? 227 * 1024 - 256 : need;
  for (const void* f : {(const void*)k_stage_tasks<true, false>, (const void*)k_stage_tasks<false, false>,
                        (const void*)k_stage_tasks<true, true>, (const void*)k_stage_tasks<false, true>}) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int exchange_stage_limit(long long P) {
  const long long per = 2 * P;
  long long n = (227ll * 1024) / per;
  if (n > kXStageMax) n = kXStageMax;
  return n >= 2 ? (int)n : 0;
}

cudaError_t configure_exchange_tma(const DevPool& p) {
  if (p.xstages <= 0) return cudaSuccess;
  return cudaFuncSetAttribute(k_exchange_copy_tma, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)((size_t)p.xstages * 2 * p.P));
}

template <bool kPack, bool kPages>
static cudaError_t launch_stage_as(const DevPool& p, const void* list, int64_t t_begin, int64_t t_end,
                                   uint8_t* staging, cudaStream_t s, int ctas, bool tma) {
  const long long units = (t_end - t_begin) * (long long)p.J;
  if (tma) {
    const int stages = stage_count(p);
    return launch_pdl(k_stage_tasks<kPack, kPages>, blocks_for(units, 1, ctas), kStageThreads, (size_t)stages * p.P, s,
                      p, list, (long long)t_begin, (long long)t_end, staging, stages);
  }
  return launch_pdl(k_stage_tasks_lsu<kPack, kPages>, blocks_for(units, 1, 4ll * ctas), kCopyThreads, 0, s, p, list,
                    (long long)t_begin, (long long)t_end, staging);
}

cudaError_t launch_stage(const DevPool& p, bool pack, bool page_list, const void* list, int64_t t_begin,
                         int64_t t_end, uint8_t* staging, cudaStream_t s, int ctas, const EventPair* ev,
                         bool tma) {
  if (t_end <= t_begin) return cudaSuccess;
  if (ev) cudaEventRecord(ev->start, s);
  auto* launch = pack ? (page_list ? launch_stage_as<true, true> : launch_stage_as<true, false>)
                      : (page_list ? launch_stage_as<false, true> : launch_stage_as<false, false>);
  const cudaError_t e = launch(p, list, t_begin, t_end, staging, s, ctas, tma);
  if (ev) cudaEventRecord(ev->end, s);
  return e;
}

constexpr long long kRemapDirect = 1 << 14;

cudaError_t launch_remap(const DevPool& p, const lv_remap_entry* e, int64_t n, int32_t epoch,
                         cudaStream_t s, int num_sms, int per_thread) {
  if (n <= 0) return cudaSuccess;
  // one entry per thread while the GPU holds every thread at once; beyond that, up
  // to four entries per thread so that their reads overlap
  const long long resident = (long long)(num_sms > 0 ? num_sms : 1) * 2048;
  int E = per_thread;
  if (E != 1 && E != 2 && E != 4) E = n <= resident ? 1 : (n <= 2 * resident ? 2 : 4);
  const unsigned grid = blocks_for((n + E - 1) / E, kRemapThreads, 1ll << 30);
  cudaError_t err;
  const unsigned T = kRemapThreads;
  if (n <= kRemapDirect && per_thread == 0)
    return launch_pdl(k_remap<1, true>, (unsigned)((n + T - 1) / T), T, 0, s, p, e, (long long)n, epoch);
  if (E == 1) err = launch_pdl(k_remap<1, false>, grid, T, 0, s, p, e, (long long)n, epoch);
  else if (E == 2) err = launch_pdl(k_remap<2, false>, grid, T, 0, s, p, e, (long long)n, epoch);
  else err = launch_pdl(k_remap<4, false>, grid, T, 0, s, p, e, (long long)n, epoch);
  if (err != cudaSuccess) return err;
  // the release pass over both tiers' owner words (8 quads of 4 per bitmap word)
  const long long qh = (long long)((p.hbm_pages + 31) / 32) * 8;
  const long long qo = (long long)((p.host_pages + 31) / 32) * 8;
  const long long cap = (long long)(num_sms > 0 ? num_sms : 1) * 8;
  const long long per_cta = (long long)kReleaseThreads * kReleaseUnroll;
  long long rg = (qh + qo + per_cta - 1) / per_cta;
  if (rg > cap) rg = cap;
  err = launch_pdl(k_release, dim3((unsigned)rg), kReleaseThreads, 0, s, p, qh, qo);
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

cudaError_t launch_cancel(const DevPool& p, const int32_t* locs, int64_t n, cudaStream_t s) {
  k_cancel<<<blocks_for(n, 256, 1ll << 30), 256, 0, s>>>(p, locs, n);
  return cudaGetLastError();
}

cudaError_t launch_append(const DevPool& p, int32_t sid, int32_t n_tokens, int32_t* pages,
                          int32_t* count, cudaStream_t s) {
  const size_t smem = 8 * (size_t)((p.hbm_pages + 31) >> 5);
  const bool fit = smem <= kStepDynamic;
  return launch_pdl(k_append, 1, kStepThreads, fit ? smem : 0, s, p, sid, n_tokens, pages, count, fit ? 1 : 0);
}

cudaError_t launch_counts(const DevPool& p, int32_t* hbm, int32_t* host, cudaStream_t s) {
  k_counts<<<p.S, kCensusThreads, 0, s>>>(p, hbm, host);
  return cudaGetLastError();
}

cudaError_t launch_blocks(const DevPool& p, int32_t sid, int32_t where, int32_t* out,
                          long long* count, cudaStream_t s) {
  return launch_pdl(k_blocks, 1, kStepThreads, 0, s, p, sid, where, out, count);
}

}  // namespace lv
