// lv_schedule: the interaction-aware request scheduler of Section 4 (Algorithm 1).
//
// A ready set of up to LV_SCHED_MAX_REQUESTS requests: every request gets a 128-bit key
// (urgency class, the class's own order, its position in the ready set).  One cluster of up
// to eight CTAs takes a round, kChunk requests a CTA.  Each CTA sorts its keys and adds up
// their costs in that order; then every thread finds its request's place among each other
// CTA's sorted keys by binary search in that CTA's shared memory.  The sum of those places
// is its place in the priority order, and the sums of the costs before them say whether it
// lies in the longest prefix that fits the round budgets ("admission stops" at the first
// request that does not fit).
#include <cooperative_groups.h>
#include <cstdint>

#include "lv_internal.cuh"

namespace cg = cooperative_groups;

namespace lv {
namespace {

using u128 = unsigned __int128;
using i128 = __int128;

constexpr int kChunk = 512;                                   // requests of a CTA, one per thread
constexpr int kWarps = kChunk / 32;
static_assert(LV_SCHED_MAX_REQUESTS == 8 * kChunk, "at most eight CTAs, a portable cluster");

__device__ __forceinline__ void sched_error(long long* ctl, int code) {
  atomicCAS(reinterpret_cast<unsigned long long*>(&ctl[C_ERR]), 0ull, (unsigned long long)code);
}

// Bits of v past the top of a class-2 value: |U'| <= bound, so v = bound - U' has at most
// bits(2 * bound) <= 112 of its 114 bits.
struct UtilityScale {
  i128 bound;
  int shift;
};

__device__ UtilityScale utility_scale(const lv_sched_params& q) {
  UtilityScale u;
  u.bound = (i128)q.beta * (1ll << 24) * q.occupied * q.p_safe_us + (i128)q.alpha * (1ll << 40) * q.allocatable;
  const u128 range = (u128)u.bound * 2;
  const unsigned long long hi = (unsigned long long)(range >> 64), lo = (unsigned long long)range;
  const int bits = hi ? 128 - __clzll((long long)hi) : 64 - __clzll((long long)lo);
  u.shift = 114 - bits;
  return u;
}

// Class-ordered key, smallest first: class 0 by playback buffer ascending, class 1 by ready
// age descending, class 2 by the Eq. 1 utility descending (U scaled by allocatable * P_safe,
// an exact integer with the same order); then the position in the ready set.  Each class's
// value is shifted up as far as its range allows, so that the key's upper half mostly decides
// a comparison by itself.
__device__ u128 request_key(const lv_request& r, int idx, const lv_sched_params& q, const UtilityScale& u,
                            long long* err) {
  long long P = r.play_buffer_us, A = r.ready_age_us, K = r.kv_pages;
  if (P < 0 || P > (1ll << 40) || A < 0 || A > (1ll << 62) || K < 0 || K > (1ll << 24) ||
      r.tokens < 0 || r.kv_needed < 0) {
    sched_error(err, LV_ERR_BOUNDS);
    P = P < 0 ? 0 : (P > (1ll << 40) ? (1ll << 40) : P);
    A = A < 0 ? 0 : (A > (1ll << 62) ? (1ll << 62) : A);
    K = K < 0 ? 0 : (K > (1ll << 24) ? (1ll << 24) : K);
  }
  unsigned cls;
  u128 v;
  if (!r.started) {
    cls = 1;
    v = (u128)((1ll << 62) - A) << 51;
  } else if (P <= q.p_safe_us) {
    cls = 0;
    v = (u128)P << 73;
  } else {
    cls = 2;
    // U' = beta*K*occupied*P_safe - alpha*(P - P_safe)*allocatable
    const i128 gain = (i128)q.beta * K * q.occupied * q.p_safe_us;
    const i128 cost = (i128)q.alpha * (P - q.p_safe_us) * q.allocatable;
    v = (u128)(u.bound - (gain - cost)) << u.shift;
  }
  return ((u128)cls << 126) | (v << 12) | (u128)(unsigned)idx;
}

// The request's fields in 64-bit loads, all in flight at once (48 bytes; the ready set may
// lie in host memory, where a load takes a microsecond or two).
__device__ __forceinline__ lv_request load_request(const lv_request* q) {
  static_assert(sizeof(lv_request) == 48, "six words");
  union {
    lv_request r;
    long long w[6];
  } u;
#pragma unroll
  for (int i = 0; i < 6; ++i)
    asm volatile("ld.global.b64 %0, [%1];" : "=l"(u.w[i]) : "l"(reinterpret_cast<const long long*>(q) + i));
  return u.r;
}

__device__ __forceinline__ u128 make_key(unsigned long long hi, unsigned long long lo) {
  return (u128)hi << 64 | lo;
}

struct SchedShared {
  alignas(16) unsigned long long hi[kChunk];
  unsigned long long lo[kChunk];               // the keys' halves, sorted ascending
  longlong2 before[kChunk + 1]; // costs of the requests before each place
  longlong2 cost[kChunk];       // by request
  longlong2 warp[kWarps];
  int32_t id[kChunk];           // by request
};

// What bounds it: instructions and latency.  3000 requests in host memory: 2.2 us to load
// them and make keys, 3.0 for the 45 exchanges of the sort (35 by shuffle, 10 through shared
// memory), 0.8 for the costs' prefix sums, 0.7 for the cluster barrier, 6.5 for the places.
// A round of 3000 requests takes 14.1 us (6 of them 5.4); as two kernels that compared every key with every
// other and summed 64-bit costs in that loop it took 22.6 (8.2).
template <int kCtas>
__global__ void __launch_bounds__(kChunk)
k_schedule(lv_sched_params q, const lv_request* reqs, int n, int32_t* order, int32_t* batch,
           long long* err) {
  __shared__ SchedShared sh;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cg::cluster_group cluster = cg::this_cluster();
  const int me = kCtas > 1 ? (int)cluster.block_rank() : 0;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int i = me * kChunk + t;
  u128 key = ~(u128)0;          // past every request's
  longlong2 mine = make_longlong2(0, 0);
  if (i < n) {
    const lv_request r = load_request(&reqs[i]);
    sh.id[t] = r.id;
    key = request_key(r, i, q, utility_scale(q), err);
    mine = make_longlong2(r.tokens > 0 ? r.tokens : 0, r.kv_needed > 0 ? r.kv_needed : 0);
  }
  sh.cost[t] = mine;
  // bitonic sort of the CTA's keys, one per thread
#pragma unroll
  for (int k = 2; k <= kChunk; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      unsigned long long lo = (unsigned long long)key, hi = (unsigned long long)(key >> 64);
      if (j >= 32) {
        sh.hi[t] = hi;
        sh.lo[t] = lo;
        __syncthreads();
        hi = sh.hi[t ^ j];
        lo = sh.lo[t ^ j];
        __syncthreads();
      } else {
        lo = __shfl_xor_sync(0xffffffffu, lo, j);
        hi = __shfl_xor_sync(0xffffffffu, hi, j);
      }
      const u128 other = make_key(hi, lo);
      const bool keep_small = ((t & k) == 0) == ((t & j) == 0);
      if ((other < key) == keep_small) key = other;
    }
  }
  const unsigned long long my_hi = (unsigned long long)(key >> 64), my_lo = (unsigned long long)key;
  sh.hi[t] = my_hi;
  sh.lo[t] = my_lo;
  // the sorted request's cost, and the costs before it in this CTA's order
  const bool live = key != ~(u128)0;
  const int own = live ? (int)(key & (u128)(LV_SCHED_MAX_REQUESTS - 1)) - me * kChunk : 0;
  __syncthreads();
  const longlong2 c = live ? sh.cost[own] : make_longlong2(0, 0);
  longlong2 x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long a = __shfl_up_sync(0xffffffffu, x.x, o), b = __shfl_up_sync(0xffffffffu, x.y, o);
    if (lane >= o) {
      x.x += a;
      x.y += b;
    }
  }
  if (lane == 31) sh.warp[wid] = x;
  __syncthreads();
  longlong2 base = make_longlong2(0, 0);
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const longlong2 y = sh.warp[w];
    base.x += w < wid ? y.x : 0;
    base.y += w < wid ? y.y : 0;
  }
  sh.before[t] = make_longlong2(base.x + x.x - c.x, base.y + x.y - c.y);
  if (t == kChunk - 1) sh.before[kChunk] = make_longlong2(base.x + x.x, base.y + x.y);
  int rank = t;
  longlong2 sum = make_longlong2(base.x + x.x, base.y + x.y);     // through this request
  if (kCtas > 1) {
    if (me == 0 && t == 0) *batch = 0;
    cluster.sync();
    // the other CTAs' sorted keys, copied here first: searching in their memory is bound by
    // the traffic between SMs (3000 requests: 9.4 us, against 1.6 for the copy and 4.5-5 for
    // the searches in this CTA's own)
    extern __shared__ __align__(16) unsigned long long peer[];       // [kCtas - 1][2][kChunk]
    constexpr int kPeers = kCtas > 1 ? kCtas - 1 : 1;
#pragma unroll
    for (int o = 0; o < kPeers; ++o) {
      // hi and lo lie one behind the other: 16 bytes a thread
      const ulonglong2* from = reinterpret_cast<const ulonglong2*>(cluster.map_shared_rank(sh.hi, (me + 1 + o) & (kCtas - 1)));
      reinterpret_cast<ulonglong2*>(peer)[o * kChunk + t] = from[t];
    }
    __syncthreads();
    // the place in every other CTA's order: the number of its keys below this one
    int pos[kPeers];
#pragma unroll
    for (int o = 0; o < kPeers; ++o) pos[o] = 2 * o * kChunk;
    auto below = [&](int at) {
      const unsigned long long hi = peer[at];
      const bool tie = hi == my_hi;
      unsigned long long lo = 0;
      if (tie) lo = peer[at + kChunk];
      return (hi < my_hi) | (tie & (lo < my_lo));
    };
#pragma unroll
    for (int step = kChunk / 2; step > 0; step >>= 1) {
#pragma unroll
      for (int o = 0; o < kPeers; ++o) {
        pos[o] += below(pos[o] + step - 1) ? step : 0;
      }
    }
    // kChunk - 1 keys were looked at: the last one decides between that many and one more
#pragma unroll
    for (int o = 0; o < kPeers; ++o) {
      pos[o] += (below(pos[o]) ? 1 : 0) - 2 * o * kChunk;
      const longlong2 b = cluster.map_shared_rank(sh.before, (me + 1 + o) & (kCtas - 1))[pos[o]];
      rank += pos[o];
      sum.x += b.x;
      sum.y += b.y;
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");   // done with the others' memory
  }
  if (live) order[rank] = sh.id[own];
  const bool fits = live && sum.x <= q.token_budget && sum.y <= q.kv_budget;
  const int admitted = __syncthreads_count(fits);
  if (kCtas > 1) {
    if (t == 0 && admitted) atomicAdd(batch, admitted);
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");     // nobody reads this CTA's memory any more
  } else if (t == 0) {
    *batch = admitted;
  }
}

}  // namespace

cudaError_t configure_schedule() {
  cudaError_t e = cudaSuccess;
  const int chunk = 2 * (int)sizeof(unsigned long long) * kChunk;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_schedule<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 3 * chunk);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_schedule<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 7 * chunk);
  return e;
}

cudaError_t launch_schedule(const lv_sched_params& q, const lv_request* reqs, int n, int32_t* order,
                            int32_t* batch, long long* ctl, cudaStream_t s) {
  // as few CTAs as hold the requests, a power of two of them
  unsigned ctas = 1;
  while ((int)ctas * kChunk < n) ctas *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kChunk);
  cfg.dynamicSmemBytes = (ctas - 1) * 2 * sizeof(unsigned long long) * kChunk;
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
  auto* kernel = ctas == 1 ? k_schedule<1> : ctas == 2 ? k_schedule<2> : ctas == 4 ? k_schedule<4> : k_schedule<8>;
  return cudaLaunchKernelEx(&cfg, kernel, q, reqs, n, order, batch, ctl);
}

}  // namespace lv
