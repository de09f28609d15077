// hx_kernels.cu -- the kernels of the batched HexGen-Flow scheduler simulation
// (arXiv 2505.05286, Sec. 4.1-4.3) for sm_103a.
//
// Every result is integer arithmetic: times are int64 microseconds, scores and
// keys int64 fixed point, divisions truncate.  Single precision only bounds a
// score or estimates a quotient, and what it leaves open is decided exactly.
// Nothing here is a dense contraction, so there are no tensor-core paths; the
// simulation kernel is bound by its chain of dependent instructions and, on a
// full GPU, by the integer pipe, the preparation kernel by HBM.
#include <climits>

#include "hx_device.cuh"

namespace hx {

// ------------------------------------------------------------------ helpers
__device__ __forceinline__ int64_t ceil_div_pos(int64_t a, int64_t b) { return (a + b - 1) / b; }

constexpr uint64_t kDigestMul = 0x9E3779B97F4A7C15ull;  // golden-ratio increment of splitmix64
constexpr uint64_t kMixA = 0xBF58476D1CE4E5B9ull;       // splitmix64 output-function multipliers
constexpr uint64_t kMixB = 0x94D049BB133111EBull;       // (Steele, Lea & Flood, OOPSLA 2014)

// Digest terms: the splitmix64 output function (two xor-shift-multiply rounds
// and a final xor-shift) of (time * phi) xor (id << 8 | tag); every step is a
// bijection, so a change of any one call's instance or start (or any query's
// end) changes the sum.
__device__ __forceinline__ uint64_t digest_term(uint64_t t, uint64_t idtag) {
  uint64_t z = (t * kDigestMul) ^ idtag;
  z = (z ^ (z >> 30)) * kMixA;
  z = (z ^ (z >> 27)) * kMixB;
  return z ^ (z >> 31);
}

// Id tags: a call's start is (rid << 8 | instance), a query's end (qid << 8 | 0xFF).
__device__ __forceinline__ uint32_t call_tag(int32_t rid, int inst) { return ((uint32_t)rid << 8) | (uint32_t)inst; }
__device__ __forceinline__ uint32_t query_tag(int32_t qid) { return ((uint32_t)qid << 8) | 0xFFu; }

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
  uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
  uint32_t mh = __reduce_min_sync(kFull, hi);
  uint32_t ml = __reduce_min_sync(kFull, hi == mh ? lo : 0xffffffffu);
  return ((uint64_t)mh << 32) | ml;
}

// Highest signed score, ties to the lowest index; every lane gets the index.
__device__ __forceinline__ int warp_argmax_s64(int64_t s, int idx) {
  uint64_t u = (uint64_t)s ^ 0x8000000000000000ull;
  uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
  uint32_t mh = __reduce_max_sync(kFull, hi);
  bool c1 = hi == mh;
  uint32_t ml = __reduce_max_sync(kFull, c1 ? lo : 0u);
  bool c2 = c1 && lo == ml;
  return (int)__reduce_min_sync(kFull, c2 ? (uint32_t)idx : 0xffffffffu);
}

// floor(n / d) for 0 <= n < 2^63 and 1 <= d < 2^54.  Trial-quotient method
// (Knuth, TAOCP vol. 2, 4.3.1): a quotient estimate from a single-precision
// reciprocal, refined once on the exact int64 remainder, then corrected by at
// most one step each way.  The estimate's relative error is below 2^-21 (two
// conversions, the approximate reciprocal, one product), so below 2^30 the
// remainder's quotient is below 2^9 and the refined estimate within one of n/d.
// Quotients of 2^30 or more take the exact integer path.
__device__ __forceinline__ uint64_t udiv_refine(uint64_t n, uint64_t d, float rd, float qf) {
  uint64_t q = (uint32_t)qf;
  q += (int64_t)(int32_t)((float)(int64_t)(n - q * d) * rd);
  const int64_t r = (int64_t)(n - q * d);
  return q - (r < 0 ? 1 : 0) + (r >= (int64_t)d ? 1 : 0);
}

__device__ __forceinline__ uint64_t udiv_trial(uint64_t n, uint64_t d) {
  float rd;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"((float)d));
  const float qf = (float)n * rd;
  return qf >= 1073741824.0f ? n / d : udiv_refine(n, d, rd, qf);
}

// Workload-balanced reward term of Eq. (score): beta / max(t_queue, 1), capped.
__device__ __forceinline__ int64_t reward_of(int64_t beta, int64_t q) {
  int64_t r = beta / (q > 1 ? q : 1);
  return r < kRewardCap ? r : kRewardCap;
}

__device__ __forceinline__ float warp_max_f32(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// Bounds of the score (1 - alpha) * min(floor(beta / max(q, 1)), cap) - alpha * e
// in single precision, f = ((1 - alpha) beta, (1 - alpha) cap, 2 (1 - alpha)):
// with t the reward term, u the cost term and w = t + u, the conversions of q
// and e, the approximate reciprocal (1 ulp), the rounded constants and the
// products leave t within 5 * 2^-24 and u within 2^-23 of their values without
// the floor, the difference adds 2^-24 w and the bounds' own rounding 2^-23 w,
// less than 2^-20 w together; the floor lowers the score by less than 1 - alpha.
// So lo - (1 - alpha) <= score <= hi - (1 - alpha), and an instance whose hi is
// below the largest lo loses.  neg_a = -inf (no instance): lo = -inf, hi = NaN,
// below everything.  One 32-bit reduction and no division in place of a 64-bit
// division pass per changed queue and a three-step 64-bit argmax: an event is a
// chain of dependent instructions, and these were the longest part of it (19
// traces x 5003 queries x 512 points on 32 instances 159.2 -> 127.3 ms, 8 x
// 20000 x 1024 on 64 instances 566.0 -> 529.4 ms).
struct ScoreRange {
  float lo, hi;
};

__device__ __forceinline__ ScoreRange score_range(int64_t q, int e, float4 f, float neg_a) {
  float rq;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rq) : "f"((float)(q > 1 ? q : 1)));
  const float t = fminf(f.x * rq, f.y), nu = neg_a * (float)e;
  const float s = t + nu, w = t - nu;
  constexpr float kErr = 1.0f / (1 << 20);
  return {fmaf(w, -kErr, s), fmaf(w, kErr, s + f.z)};
}

// (num * tb) / d truncated toward zero, for |num| < 2^41 and 1 <= tb <= d < 2^33:
// splitting num = q1 * d + r1 keeps every product below 2^63.
__device__ __forceinline__ int64_t scaled_div(int64_t num, int64_t tb, int64_t d) {
  if (num < (int64_t(1) << 32) && num > -(int64_t(1) << 32)) return (num * tb) / d;
  int64_t q1 = num / d, r1 = num % d;
  return q1 * tb + (r1 * tb) / d;
}

__device__ __forceinline__ int64_t cost_on_type(const ClusterK& c, int t, int64_t prompt, int64_t out) {
  return ceil_div_pos(prompt * kUsPerS, c.prefill[t]) + out * (int64_t)c.decode[t];
}

// Rest of a request's own path after it (the budget denominator minus its own
// mean cost), by CallRec::fcode: stage reference costs, i.e. means over instances
// of Eq. (comp) at the stage's reference tokens, for G, min(rho, R - u)
// corrections and E.
__device__ __forceinline__ int64_t rest_of_path(const ClusterK& c, int64_t rho, int row) {
  int64_t cref[4];
  for (int s = 0; s < 4; ++s) {
    int64_t sum = 0;
    for (int ty = 0; ty < c.n_types; ++ty) sum += cost_on_type(c, ty, c.ref_prompt[s], c.ref_out[s]) * c.cnt[ty];
    cref[s] = sum / c.n_inst;
  }
  const int64_t rmax = c.rmax;
  if (row == 0) return cref[HX_STAGE_G] + (rho < rmax ? rho : rmax) * cref[HX_STAGE_C] + cref[HX_STAGE_E];
  if (row == kFRows - 1) return 0;
  const int64_t left = rmax - (row - 1);
  return (rho < left ? rho : left) * cref[HX_STAGE_C] + cref[HX_STAGE_E];
}

// ------------------------------------------------------------- prep kernel
// One thread per query: Eq. (comp) per call and type, tbar, chain successor
// links and the deadline arrival + slo_mult * L0 (L0 = S + slowest
// candidate chain + E on the reference type).
__global__ void __launch_bounds__(256) hx_prep_kernel(PrepArgs a, ClusterK c) {
  int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g == 0) *a.work_counter = 0ull;
  // a run over a subset: the simulations outside it report HX_SKIPPED
  for (int64_t i = g; i < a.n_skip; i += (int64_t)gridDim.x * blockDim.x) {
    hx_result r;
    r.p95_us = -1;
    r.makespan_us = 0;
    r.events = 0;
    r.digest = 0;
    r.slo_met = 0;
    r.n_done = 0;
    r.status = HX_SKIPPED;
    r.cycles_k = 0;
    a.skip_results[i] = r;
    if (a.skip_extras) {
      hx_extra x;
      for (int t = 0; t < HX_MAX_TENANTS; ++t) {
        x.slo_met[t] = 0;
        x.n_done[t] = 0;
        x.p95_us[t] = -1;
      }
      x.reissued = 0;
      x.pad = 0;
      a.skip_extras[i] = x;
    }
  }
  if (g >= a.n_queries) return;
  int lo = 0, hi = a.n_traces;  // trace of query g: q_off[t] <= g < q_off[t+1]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (a.q_off[mid] <= g) lo = mid; else hi = mid;
  }
  const int t = lo;
  const int64_t cbase = a.c_off[t];
  const int32_t qid = (int32_t)(g - a.q_off[t]);
  const int64_t b = a.qcall[g], e = a.qcall[g + 1];
  const int k = a.kq[g];
  const int64_t arr = a.arrival[g];
  const int T = c.n_types;

  // pass 1: first correction of every chain and the exclusive latency L0
  int32_t first_corr[HX_MAX_K];
  int64_t chain[HX_MAX_K];
#pragma unroll
  for (int i = 0; i < HX_MAX_K; ++i) { first_corr[i] = -1; chain[i] = 0; }
  int64_t l_s = 0, l_e = 0;
  for (int64_t j = b; j < e; ++j) {
    const int st = a.stage[j];
    const int64_t s_ref = cost_on_type(c, c.ref_type, a.prompt[j], a.out[j]);
    if (st == HX_STAGE_S) {
      l_s += s_ref;
    } else if (st == HX_STAGE_E) {
      l_e += s_ref;
    } else {
      const int cd = a.cand[j];
      chain[cd] += s_ref;
      if (st == HX_STAGE_C && a.retry[j] == 1) first_corr[cd] = (int32_t)(j - cbase);
    }
  }
  int64_t longest = 0;
  for (int i = 0; i < k; ++i) longest = chain[i] > longest ? chain[i] : longest;
  const int tenant = a.tenant ? a.tenant[g] : 0;
  const int64_t mult = c.n_tenants > 1 ? c.tenant_mult[tenant] : c.slo_mult_fp;
  const int64_t t_slo = (mult * (l_s + longest + l_e)) / kScale;
  const int64_t deadline = arr + t_slo;
  const int32_t e_rid = (int32_t)(e - 1 - cbase);

  // pass 2: one 64-byte record per call
  for (int64_t j = b; j < e; ++j) {
    const int64_t p = a.prompt[j], o = a.out[j], oe = a.out_est[j];
    const int st = a.stage[j];
    CallRec r;
    int64_t sum = 0;
#pragma unroll
    for (int ty = 0; ty < HX_MAX_TYPES; ++ty) {
      if (ty < T) {
        const int64_t pre = ceil_div_pos(p * kUsPerS, c.prefill[ty]);
        const int64_t es = pre + oe * (int64_t)c.decode[ty];
        r.ev[ty] = make_int2((int32_t)es, (int32_t)(pre + o * (int64_t)c.decode[ty]));
        sum += es * c.cnt[ty];
      } else {
        r.ev[ty] = make_int2(0, 0);
      }
    }
    r.tbar = (int32_t)(sum / c.n_inst);
    r.deadline = deadline;
    r.arrival = arr;
    r.qid = qid;
    if (st == HX_STAGE_S) {
      r.u = 0;
      r.fcode = 0;
      r.done = kDoneRelease;
      r.next = (int32_t)(j + 1 - cbase);
      r.k = (uint8_t)k;
    } else if (st == HX_STAGE_E) {
      r.u = (uint8_t)tenant;
      r.fcode = kFRows - 1;
      r.done = kDoneQuery;
      r.next = 0;
      r.k = 0;
    } else {
      const int cd = a.cand[j];
      int32_t nx;
      if (st == HX_STAGE_G) {
        r.u = 0;
        nx = first_corr[cd];
      } else {
        r.u = a.retry[j];
        nx = (j + 1 < e - 1 && a.stage[j + 1] == HX_STAGE_C && a.cand[j + 1] == cd) ? (int32_t)(j + 1 - cbase) : -1;
      }
      r.done = nx >= 0 ? kDoneRelease : kDoneChain;
      r.next = nx >= 0 ? nx : e_rid;
      r.k = (uint8_t)(nx >= 0 ? 1 : k);
      r.fcode = (uint8_t)(1 + r.u);
    }
    const int4* src = reinterpret_cast<const int4*>(&r);
    int4* dst = reinterpret_cast<int4*>(a.rec + j);
    dst[0] = src[0];
    dst[1] = src[1];
    dst[2] = src[2];
    dst[3] = src[3];
  }
}

// -------------------------------------------------------- simulation kernel
namespace {

// Event times of one simulation are relative to a base.  While no attempt can
// take 2^25 us (on any type, stretched by fault windows and timeouts), they are
// 32-bit, the base moves up every 2^25 us, and an instance's next completion is
// time << 6 | instance: one 32-bit warp minimum gives the next event's time and
// instance (a dispatch's least cost << 6 | instance likewise), without the ballot
// and the bit search that lengthened the event's chain (8 x 2000 queries x 64
// points 6.80 -> 6.29 ms, 8 x 20000 x 1024 on 64 instances 431 -> 399 ms; fault
// windows on 24 x 2000 x 64 15.5 -> 13.8 ms).  Longer attempts have 64-bit times,
// base 0, in a family that carries policies, tenants and faults too: one such
// attempt in a grid that needs none of these costs half as much again (8 x 2000 x 64
// 6.3 -> 9.3 ms, 64 x 2000 x 64 14.1 -> 21.3, 8 x 4000 x 1024 on 64 instances 74 -> 112).
template <bool kWide>
struct Times {
  using T = uint32_t;
  using Slot = Slot32;
};
template <>
struct Times<true> {
  using T = uint64_t;
  using Slot = Slot64;
};
constexpr int kInstBits = 6;                          // of a key: HX_MAX_INST instances
constexpr uint64_t kInstMask = (1 << kInstBits) - 1;

// Running calls complete by (end, request id); a tag is request id << 8 |
// kFailBit if the attempt times out | slot.
__device__ __forceinline__ bool before(uint32_t e0, uint32_t tag0, uint32_t e1, uint32_t tag1) {
  return ((uint64_t)e0 << 32 | tag0) < ((uint64_t)e1 << 32 | tag1);
}
__device__ __forceinline__ bool before(uint64_t e0, uint32_t tag0, uint64_t e1, uint32_t tag1) {
  return (e0 < e1) | ((e0 == e1) & (tag0 < tag1));
}

// A value that every lane holds alike, broadcast so that the compiler knows it:
// branches on such values need no reconvergence code, and warp-wide operations
// behind them no check that the warp is whole.
// Every branch of the event loop that leads to a warp-wide operation is on a
// broadcast or voted value: 195 -> 171 warp-instructions per event (no BRA.DIV,
// a tenth of the BSSY / BSYNC), 8 x 2000 queries x 64 points 7.6 -> 6.8 ms,
// alpha = 1 on 64 instances 3226 -> 2788 cycles per event.
template <class T>
__device__ __forceinline__ T uniform(T v) {
  return __shfl_sync(kFull, v, 0);
}

__device__ __forceinline__ uint32_t warp_min(uint32_t v) { return __reduce_min_sync(kFull, v); }
__device__ __forceinline__ uint64_t warp_min(uint64_t v) { return warp_min_u64(v); }

// The digest is a sum of terms, so they are hashed a batch at a time: every
// lane calls with the same (t, tag) and stores the same pair; a full batch is
// hashed one term per lane and summed into W->digest.
template <bool kWide>
__device__ __noinline__ void digest_flush(WarpShared* W, int n, int lane) {
  __syncwarp();
  uint64_t t, tag;
  if (kWide) {
    const ulonglong2 e = reinterpret_cast<const ulonglong2*>(W->dterm)[lane < n ? lane : 0];
    t = e.x;
    tag = e.y;
  } else {
    const uint2 e = reinterpret_cast<const uint2*>(W->dterm)[lane < n ? lane : 0];
    t = (uint64_t)W->base + e.x;
    tag = e.y;
  }
  uint64_t y = lane < n ? digest_term(t, tag) : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(kFull, y, o);
  if (lane == 0) W->digest += y;
  __syncwarp();
}

template <bool kWide, class T>
__device__ __forceinline__ void digest_push(WarpShared* W, int& dn, T t, uint32_t tag, int lane) {
  constexpr int kBatch = kWide ? 16 : 32;
  if (kWide)
    reinterpret_cast<ulonglong2*>(W->dterm)[dn] = make_ulonglong2(t, tag);
  else
    reinterpret_cast<uint2*>(W->dterm)[dn] = make_uint2((uint32_t)t, tag);
  if (++dn == kBatch) {
    digest_flush<kWide>(W, kBatch, lane);
    dn = 0;
  }
}

__device__ __forceinline__ bool ent_better(const HeapEnt& a, const HeapEnt& b) {
  return (a.key > b.key) | ((a.key == b.key) & (a.rid < b.rid));
}

// A heap entry in one 16-byte access.
__device__ __forceinline__ HeapEnt ent_load(const HeapEnt* p) {
  HeapEnt e;
  uint32_t lo, hi;
  asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(lo), "=r"(hi), "=r"(e.rid), "=r"(e.svc)
               : "l"(p)
               : "memory");
  e.key = (unsigned long long)hi << 32 | lo;
  return e;
}

// The same under a predicate and not a branch; without it the key is 0, below
// every key (rid and svc are whatever they were).
__device__ __forceinline__ HeapEnt ent_load(const HeapEnt* p, bool on) {
  HeapEnt e;
  uint32_t lo = 0, hi = 0;
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.s32 p, %5, 0;\n @p ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n}"
      : "+r"(lo), "+r"(hi), "=r"(e.rid), "=r"(e.svc)
      : "l"(p), "r"((int)on)
      : "memory");
  e.key = (unsigned long long)hi << 32 | lo;
  return e;
}

__device__ __forceinline__ void ent_store(HeapEnt* p, const HeapEnt& e, bool on) {
  asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %5, 0;\n @p st.global.v4.b32 [%4], {%0, %1, %2, %3};\n}" ::"r"(
                   (uint32_t)e.key),
               "r"((uint32_t)(e.key >> 32)), "r"(e.rid), "r"(e.svc), "l"(p), "r"((int)on)
               : "memory");
}

// Local queues are 32-ary max-heaps on (key desc, rid asc) in the warp's
// arena: node i has children 32 i + 1 .. 32 i + 32, so 40k waiting requests
// sit four levels deep.  New requests rarely climb past their parent, so an
// event's join at once unless one does; pop and replace sift down with the whole
// warp, one lane per child.  At alpha = 1 every call passes through one queue and
// the event's chain sets a run's end: with the root's children read before the
// key or the start needs them, the children compared by their keys' high words
// and entries moved by predicated 16-byte accesses, 8 traces x 20000 queries x
// 1024 points took 463 -> 430 ms, 3000 queries on 64 instances 40.3 -> 38.4 ms.
__device__ __forceinline__ void heap_push(HeapEnt* h, int n, HeapEnt e) {
  int i = n;
  while (i > 0) {
    const int par = (i - 1) >> 5;
    const HeapEnt pe = ent_load(h + par);
    if (!ent_better(e, pe)) break;
    ent_store(h + i, pe, true);
    i = par;
  }
  ent_store(h + i, e, true);
}

// This lane's child of node i in a heap of m entries; past its end an entry
// that goes after every other.
__device__ __forceinline__ HeapEnt heap_child(const HeapEnt* h, int i, int m, int lane) {
  const int child = 32 * i + 1 + lane;
  return ent_load(h + child, child < m);
}

// One level of a sift: all lanes call with the same arguments but c, their child
// of node i.  Unless `sink` goes before every child, the best one moves up to
// node i, which becomes the node it came from, c its children there; else false.
__device__ __forceinline__ bool heap_step(HeapEnt* h, int m, const HeapEnt& sink, int& i, HeapEnt& c, int lane) {
  if (32 * i + 1 >= m) return false;
  const uint32_t sink_hi = (uint32_t)(sink.key >> 32);
  // the first child by (key desc, rid asc): the keys' high words decide, the
  // low words and the rids among equals only
  const uint32_t hi = (uint32_t)(c.key >> 32);
  const uint32_t mh = __reduce_max_sync(kFull, hi);
  if (mh < sink_hi) return false;
  unsigned best = __ballot_sync(kFull, hi == mh);
  if (((best & (best - 1)) != 0) | (mh == sink_hi)) {
    const uint32_t lo = (uint32_t)c.key, ml = __reduce_max_sync(kFull, hi == mh ? lo : 0u);
    best = __ballot_sync(kFull, (hi == mh) & (lo == ml));
    const bool tie = (best >> lane) & 1u;
    const uint32_t mr = __reduce_min_sync(kFull, tie ? (uint32_t)c.rid : 0xffffffffu);
    best = __ballot_sync(kFull, tie & ((uint32_t)c.rid == mr));
    if (__ballot_sync(kFull, ent_better(c, sink)) == 0) return false;
  }
  const int b = 31 - __clz(best);
  ent_store(h + i, c, lane == b);  // the best child moves up
  i = 32 * i + 1 + b;
  c = heap_child(h, i, m, lane);
  return true;
}

// All lanes call with the same arguments but c, their child of node i, whose entry
// has left.  `sink` takes its place, sinking to its level; the heap then holds m
// entries (m = n - 1 and sink = the last entry: a pop; m = n and sink = a new
// entry: a replace).
__device__ __forceinline__ void heap_sift_warp(HeapEnt* h, int m, HeapEnt sink, int i, HeapEnt c, int lane) {
  while (heap_step(h, m, sink, i, c, lane)) {
  }
  ent_store(h + i, sink, (lane == 0) & (m > 0));
  __syncwarp();
}

// Min-heap of the K largest latencies seen so far, 32-ary like the local
// queues; its root is the K-th largest latency, i.e. the nearest-rank P95
// when K = n - ceil(0.95 n) + 1.  All lanes call with the same v: lane 0
// writes the heap, every lane writes the same size (*size) and root (*root)
// copies in shared memory.
__device__ __noinline__ void topk_insert_warp(int64_t* h, int32_t* size, int kcap, int64_t* root_out, int64_t v,
                                              int lane) {
  __builtin_assume(__isGlobal(h));
  const int n = uniform(*size);
  kcap = uniform(kcap);
  if (n < kcap) {
    // filling: sift up on lane 0 (few levels)
    if (lane == 0) {
      int i = n;
      while (i > 0) {
        const int par = (i - 1) >> 5;
        const int64_t pv = h[par];
        if (pv <= v) break;
        h[i] = pv;
        i = par;
      }
      h[i] = v;
    }
    __syncwarp();
    *size = n + 1;
    if (n + 1 == kcap) *root_out = h[0];
  } else if (__any_sync(kFull, v > *root_out)) {
    // v replaces the root and sinks; one lane per child (latencies are >= 0)
    int i = 0;
    int64_t root = v;
    for (;;) {
      const int first = 32 * i + 1;
      if (first >= n) break;
      const int ch = first + lane;
      const uint64_t cv = ch < n ? (uint64_t)h[ch] : ~0ull;
      const uint64_t mn = warp_min_u64(cv);
      if (__any_sync(kFull, mn >= (uint64_t)v)) break;
      const int b = __ffs(__ballot_sync(kFull, cv == mn)) - 1;
      if (i == 0) root = (int64_t)mn;
      if (lane == 0) h[i] = (int64_t)mn;
      i = first + b;
    }
    if (lane == 0) h[i] = v;
    __syncwarp();
    *root_out = root;
  }
}

__device__ __noinline__ int64_t budget_wide(int64_t num, int64_t tb, int64_t d) { return scaled_div(num, tb, d); }

// t_slo of Eq. (budget): (deadline - now) * tbar / (tbar + F), truncated
// toward zero; |num| < 2^34 keeps |num| * tbar below 2^63.
__device__ __forceinline__ int64_t slo_budget(int64_t num, int64_t tb, int64_t dd) {
  if (num > -(int64_t(1) << 34) && num < (int64_t(1) << 34)) {
    const uint64_t res = udiv_trial((uint64_t)(num < 0 ? -num : num) * (uint64_t)tb, (uint64_t)dd);
    return num < 0 ? -(int64_t)res : (int64_t)res;
  }
  return budget_wide(num, tb, dd);
}

__device__ __noinline__ int64_t budget_exact(int64_t num, int64_t tb, int64_t dd) { return slo_budget(num, tb, dd); }

// Local-queue key, higher first, of a request dispatched now: Eq. (priority)
// with the budget at send time (now) and the common now dropped; FCFS: earliest
// enqueue; LLF: least deadline - now - remaining work, again with the common
// now dropped.  est is its Eq. (comp) on the instance.  All lanes call,
// so that its branches are uniform; a lane without a request (mine: false, with some
// other's record) stays out of the vote between them (record 0's deadline, once it is
// 2^34 us past, sent every lane to the exact divisions: 1.2 to 1.4 times the cycles).
__device__ __forceinline__ unsigned long long queue_key(const WarpShared* W, const CallRec* r, int est, int64_t now, int lpol,
                                                        bool mine) {
  const int64_t dl = r->deadline;
  const int4 tail = *reinterpret_cast<const int4*>(&r->tbar);
  const int64_t tb = tail.x;
  const int64_t dd = tb + W->frest[(tail.w >> 16) & 0xff];
  int64_t key;
  if (lpol == HX_LOCAL_PQ) {
    // slo_budget with one uniform branch: |num| * tbar below 2^62 and a quotient
    // below 2^30 on every lane, or all lanes take the exact divisions
    const int64_t num = mine ? dl - now : 0;
    const uint64_t n = (uint64_t)(num < 0 ? -num : num);
    float rd;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rd) : "f"((float)dd));
    const float qf = (float)(n * (uint64_t)tb) * rd;
    int64_t budget;
    if (__all_sync(kFull, ((n >> 34) == 0) & (qf < 1073741824.0f))) {
      const uint64_t res = udiv_refine(n * (uint64_t)tb, (uint64_t)dd, rd, qf);
      budget = num < 0 ? -(int64_t)res : (int64_t)res;
    } else {
      budget = budget_exact(num, tb, dd);
    }
    key = kScale * ((int64_t)est - budget) - W->G * now;
  } else {
    key = lpol == HX_LOCAL_FCFS ? -now : dd - dl;
  }
  return (unsigned long long)key ^ 1ull << 63;
}

// The instance's new requests (this lane's: e; on the lanes of pm) join its
// local queue, which moves to a region of twice the size when it is full (8
// requests at most, so once).  All lanes call.  Returns HX_OK or
// HX_ERR_CAPACITY.
__device__ __forceinline__ int push_pending(WarpShared* W, InstState* I, HeapEnt e, unsigned pm, int64_t arena_per_warp,
                                            int lane) {
  HeapEnt* const arena = W->arena;
  __builtin_assume(__isGlobal(arena));
  const int size = uniform(I->hsize), np = __popc(pm);
  const uint32_t heap = uniform(I->heap);
  const int hcl = (int)(heap >> kHeapCodeShift), cap = hcl ? 8 << hcl : 0;
  int hoff = (int)(heap & kHeapOffMask);
  if (size + np > cap) {
    const int ncap = cap ? 2 * cap : 16, bump = uniform(W->bump), off = hoff;
    if ((int64_t)bump + ncap > arena_per_warp) return HX_ERR_CAPACITY;
    hoff = bump;
    for (int i = lane; i < size; i += 32) arena[hoff + i] = arena[off + i];
    __syncwarp();
    W->bump = bump + ncap;  // every lane writes the same values
    I->heap = (uint32_t)hoff | (uint32_t)(hcl + 1) << kHeapCodeShift;
  }
  HeapEnt* const h = arena + hoff;
  const bool mine = (pm >> lane) & 1u;
  const int pos = size + __popc(pm & ((1u << lane) - 1));
  // with a non-empty queue every new entry's parent is an old one: when none
  // climbs past its parent, all are stored at once
  const bool ask = mine & (size > 0);
  const HeapEnt pe = ent_load(h + ((pos - 1) >> 5), ask);
  if (!__any_sync(kFull, (ask & ent_better(e, pe)) | (size == 0))) {
    ent_store(h + pos, e, mine);
  } else {
    for (unsigned left = pm; left; left &= left - 1) {
      if (lane == __ffs(left) - 1) heap_push(h, pos, e);
      __syncwarp();
    }
  }
  I->hsize = size + np;
  __syncwarp();
  return HX_OK;
}

// The dispatch winner from exact scores, for the dispatches whose float bounds
// overlap: highest score, ties to the lowest instance.  All lanes call.
template <int J>
__device__ __noinline__ int exact_winner(const WarpShared* W, int64_t q0, int64_t q1, int e0, int e1, bool ok0, bool ok1,
                                         int lane) {
  const uint64_t beta = (uint64_t)W->beta;
  const int64_t A = W->A, oma = W->one_minus_a;
  const uint64_t r0 = udiv_trial(beta, q0 > 1 ? (uint64_t)q0 : 1ull);
  const int64_t s0 = ok0 ? oma * (int64_t)(r0 < (uint64_t)kRewardCap ? r0 : kRewardCap) - A * e0 : INT64_MIN;
  if (J == 1) return warp_argmax_s64(s0, lane);
  const uint64_t r1 = udiv_trial(beta, q1 > 1 ? (uint64_t)q1 : 1ull);
  const int64_t s1 = ok1 ? oma * (int64_t)(r1 < (uint64_t)kRewardCap ? r1 : kRewardCap) - A * e1 : INT64_MIN;
  const bool take1 = s1 > s0;
  return warp_argmax_s64(take1 ? s1 : s0, take1 ? lane + 32 : lane);
}

// All lanes: a query's evaluation call finished at `now` (Sec. 4.3's metrics).
__device__ __forceinline__ void finish_query(WarpShared* W, int64_t now, int64_t arrival, int64_t deadline, int lane) {
  // every lane reads the counters, then every lane writes the same new values
  const int32_t slo = W->slo_met + (now <= deadline ? 1 : 0), nd = W->n_done + 1;
  __syncwarp();
  W->slo_met = slo;
  W->n_done = nd;
  W->makespan = now;
  // most latencies of a full heap fall below its root and change nothing
  const int64_t v = now - arrival;
  if (__any_sync(kFull, (W->tk < W->kcap) | (v > W->tkmin))) topk_insert_warp(W->topk, &W->tk, W->kcap, &W->tkmin, v, lane);
}

}  // namespace

// Resident blocks per SM the register allocation aims for (4 warps each): 8
// with one instance per lane; with two, 7, whose 72 registers hold the event
// loop's state (8 spill 48 bytes in the event loop: 8 traces x 20000 queries x
// 1024 points 503 ms against 458 ms).  What these forms spill, 0 to 48 bytes by
// family, lies outside the loop: no local load per event is counted.  The form for few
// warps aims at 5 (96 registers, no spills: 64 x 3001 x 16 25.5 -> 23.5 ms; 4 or 6
// blocks 1 to 4 % slower).
#ifndef HX_SIM_MIN_BLOCKS
#define HX_SIM_MIN_BLOCKS(J) ((J) == 1 ? 8 : 7)
#endif
constexpr int kFewMinBlocks = 5;
constexpr int kLongQueue = 128;  // entries (512: 27.0 ms)

// Bounds-checked build (-DHX_CHECKED): before every shared- or global-memory
// access whose index the simulation forms from its own state (instance,
// request id, query id, slot, heap offset and size, top-K size), the
// index is range-checked; a failed check sets the simulation's status to
// HX_ERR_BOUNDS and leaves the loop it is in instead of making the access,
// and the simulation stops after that event.  Every checked value is the
// same on all lanes, so the exit is warp-uniform.  In the normal build the
// checks compile to nothing.
#ifdef HX_CHECKED
#define HX_BOUND(cond)          \
  if (!(cond)) {                \
    status = HX_ERR_BOUNDS;     \
    break;                      \
  }
#define HX_STOP_IF_FAILED() \
  if (status != HX_OK) break;
#else
#define HX_BOUND(cond)
#define HX_STOP_IF_FAILED()
#endif

// The lane with the lowest tag (a call of its own: it is rare, and inlined it
// would run predicated at every completion).
__device__ __noinline__ unsigned lowest_id(uint32_t tag) {
  return __ballot_sync(kFull, tag == __reduce_min_sync(kFull, tag));
}

// One warp, one simulation.  J instances per lane: lane l owns l and, with J = 2,
// l + 32.  kFew: the form for runs of few warps.
//
// An event is a chain of dependent warp instructions.  A lone simulation waits on
// it (171 instructions, 820 cycles per call event with one instance per lane); a
// full GPU, 7 or 8 warps per scheduler, spends 165 instructions, 1730 cycles per
// event and warp, on its half-rate integer pipe (68 % busy) and issue slots (67 %).
// So the state that only scores and the next event need stays in the owner lane's
// registers, where an update is a select; event times are 32-bit, so one warp
// reduction finds the next completion; running calls sit unsorted in their slots
// under a free mask, so a start is one store and one comparison, and a completion
// one reduction over the instance's slots; and up to 32 instances take one lane
// each (half the per-lane work).  Against sorted 64-bit slot keys and per-instance
// arrays in shared memory, when this layout came: 342 -> 178 instructions, 8 x 2000
// queries x 64 points on 8 instances 14.2 -> 10.9 ms, 19 x 5003 x 512 on 32
// instances 127 -> 89 ms, 8 x 20000 x 1024 on 64 instances 529 -> 460 ms.
template <int J, int kFamily, bool kFew>
__device__ __forceinline__ void sim_body(const SimArgs& a, const ClusterK& c) {
  constexpr bool kLog = kFamily >= kSimLog, kGeneric = kFamily >= kSimGeneric;
  constexpr bool kFaults = kFamily >= kSimFaults, kWide = kFamily == kSimWide;
  constexpr bool kSpaced = spaced_slots(J, kWide, kFew);
  using T = typename Times<kWide>::T;
  using Slot = typename Times<kWide>::Slot;
  constexpr T kIdle = ~T(0);                        // no time
  constexpr T kNone = kIdle & ~T(kInstMask);        // keys from here on: no running call, no arrival in range
  constexpr T kFar = kWide ? kNone : T(1) << 31;  // an event with such a key moves the base up first
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = uniform((int)(threadIdx.x >> 5));
  // volatile: read once and kept, not read again wherever it is used
  int lane;
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
  WarpShared* const W = reinterpret_cast<WarpShared*>(smem_raw + warp * c.smem_per_warp);
  InstState* const inst = reinterpret_cast<InstState*>(W + 1);
  Slot* const slots = reinterpret_cast<Slot*>(inst + 32 * J);
  if (lane == 0) {
    // this warp's slices of the scratch arrays (kept in shared memory to spare registers)
    const int64_t gw = (int64_t)blockIdx.x * kWarpsPerBlock + warp;
    W->arena = a.arena + gw * a.arena_per_warp;
    W->chains = a.chains + gw * a.chains_per_warp;
    W->topk = a.topk + gw * a.topk_per_warp;
  }
  __syncwarp();  // every lane clears its part of W->chains before a simulation's first barrier
  const int N = c.n_inst;
  // an instance's slots are read one per lane of the lower half warp
  const int l16 = lane & 15;
  const uint32_t lbit = lane < 16 ? 1u << lane : 0u;
  uint32_t lrec[J];  // byte offset of this lane's type in a call record
#pragma unroll
  for (int j = 0; j < J; ++j) lrec[j] = lane + 32 * j < N ? 8u * c.inst_type[lane + 32 * j] : 0u;

  for (;;) {
    unsigned long long work = 0;
    if (lane == 0) work = atomicAdd(a.work_counter, 1ull);
    const int64_t w = (int64_t)uniform(work);
    if (w >= a.n_work) break;
    // trace-major, so that concurrent simulations share a trace in L2; within a
    // trace the highest point index (highest alpha, the longest queues) first
    // (a subset comes sorted in the same order)
    int t, p;
    if (a.subset) {
      const int64_t s = a.subset[w];
      t = (int)(s / a.n_points);
      p = (int)(s - (int64_t)t * a.n_points);
    } else {
      t = (int)(w / a.n_points);
      p = a.n_points - 1 - (int)(w - (int64_t)t * a.n_points);
    }
    const int64_t sim = (int64_t)t * a.n_points + p;
    const long long clk0 = clock64();
    const int64_t qb = a.q_off[t];
    const int32_t nq = uniform((int32_t)(a.q_off[t + 1] - qb));
    const int64_t cb = a.c_off[t];
    const int32_t nc = uniform((int32_t)(a.c_off[t + 1] - cb));
    const CallRec* const rec = a.rec + cb;
    if (lane == 0) {
      W->qb = qb;
      W->cb = cb;
      W->nq = nq;
      W->nc = nc;
      W->sim = sim;
      W->clk0 = clk0;
    }

    // per-instance state that every lane reads later: written before the
    // barrier below
    auto has_windows = [&](int m) -> bool {
      bool any = false;
      for (int f = 0; f < c.n_faults; ++f) any |= c.faults[f].inst == m;
      return any;
    };
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int m = lane + 32 * j;
      const uint32_t mask = m < N ? (1u << c.inst_slots[m]) - 1 : 0u;
      inst[m] = InstState{mask, 0, 0u, mask | (m < N ? (uint32_t)c.slot_base[m] << 16 : 0u) |
                                           (kFaults && m < N && has_windows(m) ? kWindowsBit : 0u)};
    }
    // no chain of any query has finished
    for (int i = 16 * lane; i < nq; i += 512) *reinterpret_cast<uint4*>(W->chains + i) = make_uint4(0, 0, 0, 0);
    if (lane < kFRows) W->frest[lane] = rest_of_path(c, a.rho[p], lane);
    if (kGeneric && lane < HX_MAX_TENANTS)
      W->tkcap[lane] = a.tenant_kcap ? a.tenant_kcap[(int64_t)t * HX_MAX_TENANTS + lane] : 0;
    if (lane == 0) {
      const int64_t A = a.alpha[p];
      W->A = (int32_t)A;
      W->one_minus_a = (int32_t)(kScale - A);
      W->G = a.gamma[p];
      const int64_t beta = a.beta[p], oma = kScale - A;
      W->beta = beta;
      W->fscore = make_float4((float)((double)oma * (double)beta), (float)oma * (float)kRewardCap, 2.0f * (float)oma, 0.0f);
      // t_queue up to which instances share the greatest reward and beat every
      // other one whatever its cost (below 2^28): all of them when rewards have
      // no weight (alpha = 1); the idle ones (max(t_queue, 1) = 1) when the step
      // from beta to the next reward, at most beta / 2, outweighs any cost
      // difference; else none.  Instances past N hold INT64_MAX.
      const bool idle_top = oma * (reward_of(beta, 1) - reward_of(beta, 2)) > A << 28;
      W->tie = make_longlong2(A == kScale ? INT64_MAX - 1 : idle_top ? 1 : -1, A != 0 ? 0xffffffffll : 0ll);
      W->lpol = a.lpol[p];
      W->kcap = nq - (95 * nq + 99) / 100 + 1;
      W->rr = 0;
      W->bump = 0;
      W->digest = 0;
      W->makespan = 0;
      W->n_done = 0;
      W->slo_met = 0;
      W->tk = 0;
      W->tkmin = 0;
      for (int t = 0; t < HX_MAX_TENANTS; ++t) {
        W->tcount[t] = make_int2(0, 0);
        W->ttk[t] = 0;
        W->ttkmin[t] = 0;
      }
      W->reissued = 0;
      W->excl = -1;
    }
    __syncwarp();

    // What this lane keeps of its instances, in registers: t_queue, the next
    // completion's key (kNone up: nothing runs) and its tag (request id << 8 |
    // slot).  An instance past N has t_queue INT64_MAX and cost weight -inf in the
    // score filter, and never wins.
    int64_t q[J];
    T next_key[J];
    uint32_t next_tag[J];
    float neg_a[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const bool on = lane + 32 * j < N;
      q[j] = on ? 0 : INT64_MAX;
      next_key[j] = kIdle;
      next_tag[j] = 0;
      neg_a[j] = on ? -(float)W->A : -INFINITY;
    }

    // the record slot of a logged simulation, or -1; the dispatch policy
    const int recj = kLog && a.rec_map ? uniform(a.rec_map[sim]) : -1;
    const bool round_robin = kGeneric && uniform((int)a.dpol[p]) == HX_DISPATCH_RR;

    // Eq. (comp) and the service time on this lane's instances of the request
    // that is dispatched next
    int2 cost_of[J];
    auto load_costs = [&](int32_t rid) {
#pragma unroll
      for (int j = 0; j < J; ++j)
        cost_of[j] = *reinterpret_cast<const int2*>(reinterpret_cast<const char*>(rec + rid) + lrec[j]);
    };
    // what a run of few warps has registers to keep
    uint8_t* const chains0 = W->chains;
    const longlong2 tie0 = W->tie;
    const float4 fscore0 = W->fscore;

    // the key of an arrival, after every completion at its time; kNone up: 2^26 us
    // or more past the base
    W->base = 0;
    auto arrival_key = [&](int64_t t_abs) -> T {
      if (kWide) return (T)t_abs << kInstBits | kInstMask;
      const uint64_t d = (uint64_t)(t_abs - W->base);
      return (d >> (32 - kInstBits)) ? kIdle : (T)d << kInstBits | kInstMask;
    };
    auto absolute = [&](T t) -> int64_t { return kWide ? (int64_t)t : W->base + (int64_t)t; };
    W->arrivals = 0;
    W->next_arrival = nq > 0 ? a.arrival[qb] : 0;
    T arr = nq > 0 ? uniform(arrival_key(a.arrival[qb])) : kIdle;
    T now = 0;
    int32_t status = HX_OK, npend = 0;
    // event bound; re-issued attempts add events while fault windows last
    int32_t steps_left = nc + nq + 8 + (kFaults ? 16 * nc + 4096 : 0);
#ifdef HX_CHECKED
    // the warp's scratch slices must hold this trace's chain counters and top-K
    if (!(nq <= a.chains_per_warp && W->kcap <= a.topk_per_warp && (a.tenant_kcap == nullptr ||
          (int64_t)(HX_MAX_TENANTS + 1) * a.tenant_topk_off[0] <= a.topk_per_warp)))
      status = HX_ERR_BOUNDS;
#endif

    auto first_slot = [&](int m, const InstState& I) -> uint32_t { return kSpaced ? 16u * m : (kFaults ? I.cfg & ~kWindowsBit : I.cfg) >> 16; };
    // A request starts that waited in a long queue: its record's second half and
    // the records that follow have left L1 since its query arrived (3000 queries on
    // 64 instances, whose alpha = 1 queue grows past 1000: 29.0 -> 26.4 ms).  Left
    // out with one instance per lane, where it cost the sweeps 1 to 2 %: their
    // queues stayed short.
    auto fetch_after = [&](int32_t rid) {
      const int64_t off = (int64_t)rid * 64 + 32 + 32 * lane;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&W->sink);
      const char* const from = reinterpret_cast<const char*>(rec) + off;
      if (off < (int64_t)nc * 64) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(from) : "memory");
    };
    auto queue_of = [&](uint32_t heap) -> HeapEnt* {
      HeapEnt* const arena = W->arena;
      __builtin_assume(__isGlobal(arena));
      return arena + (heap & kHeapOffMask);
    };
    // an instance without fault windows skips the search for the one that covers
    // now (24 x 2000 queries x 64 points, 3 of 8 instances with windows: 13.5 -> 13.25 ms)
    auto windows_on = [&](const InstState& I) -> bool { return kFaults && (uniform(I.cfg) & kWindowsBit); };
    // Request rid starts on instance m now in the highest of its free slots;
    // svc is its service time on m (on m's lane at least).  The slots stay
    // unsorted: a start is one store and a comparison with the instance's next
    // completion.  Returns the remaining free slots.
    int dn = 0;  // digest terms waiting in W->dterm
    auto start_call = [&](int m, uint32_t free, uint32_t slot_base, bool windows, int rid, int svc) -> uint32_t {
      T run = (T)svc;
      bool fail = false;
      if (kFaults && windows) {
        // the first fault window of m that covers now, and the timeout (Sec. 3.3)
        const int64_t t_abs = absolute(now);
        int64_t r64 = svc;
        bool in_window = false, down = false;
        for (int f = 0; f < c.n_faults; ++f) {
          const FaultK& F = c.faults[f];
          if (F.inst == m && t_abs >= F.t0 && t_abs < F.t1) {
            in_window = true;
            if (F.slow == 0) down = true;
            else r64 = (r64 * F.slow + kScale - 1) / kScale;
            break;
          }
        }
        if (in_window && c.timeout_mult_fp > 0) {
          const int64_t timeout = ((int64_t)rec[rid].ev[c.inst_type[m]].x * c.timeout_mult_fp) / kScale;
          if (down || r64 > timeout) {
            fail = true;
            r64 = timeout;
          }
        }
        run = (T)r64;
      }
      const int s = 31 - __clz(free);
      const uint32_t tag = (uint32_t)rid << 8 | (kFaults && fail ? kFailBit : 0u) | (uint32_t)s;
      const T end = now + run, key = end << kInstBits | (T)m;
      if (lane == (m & 31)) {
        Slot e;
        e.end = end;
        e.tag = tag;
        if constexpr (kWide) e.pad = 0;
        slots[slot_base + s] = e;
        if (kLog && recj >= 0) {
          a.rec_start[(int64_t)recj * a.rec_stride + rid] = absolute(now);
          a.rec_end[(int64_t)recj * a.rec_stride + rid] = absolute(end);
        }
      }
#pragma unroll
      for (int j = 0; j < J; ++j) {
        // the lowest request id completes first among equal ends
        const bool first = (lane + 32 * j == m) & before(key, tag, next_key[j], next_tag[j]);
        next_key[j] = first ? key : next_key[j];
        next_tag[j] = first ? tag : next_tag[j];
      }
      free ^= 1u << s;
      inst[m].free = free;  // every lane stores the same mask
      digest_push<kWide>(W, dn, now, call_tag(rid, m), lane);
      return free;
    };

    for (;;) {
      HX_STOP_IF_FAILED()
      __syncwarp();
      const T mn = warp_min(J == 2 && next_key[J - 1] < next_key[0] ? next_key[J - 1] : next_key[0]);
      if (((mn < arr ? mn : arr) >= kFar) | (steps_left == 0)) {
        // the end, too many events, or nothing within 2^25 us of the base, which
        // then moves to the next event
        const bool more = uniform(W->arrivals) < nq;
        if (mn >= kNone && !more) break;
        if (steps_left-- == 0) {
          status = HX_ERR_STEP_LIMIT;
          break;
        }
        ++steps_left;
        if (!kWide) {
          digest_flush<kWide>(W, dn, lane);
          dn = 0;
          const int64_t base = W->base, at = W->next_arrival;
          int64_t nb = mn >= kNone ? at : base + (int64_t)(mn >> kInstBits);
          if (more && at < nb) nb = at;
          const T shift = (T)(nb - base);
#pragma unroll
          for (int j = 0; j < J; ++j) next_key[j] = next_key[j] >= kNone ? kIdle : next_key[j] - (shift << kInstBits);
          for (int j = lane; j < c.slot_entries; j += 32) slots[j].end -= shift;
          __syncwarp();
          W->base = nb;  // every lane writes the same value
          arr = more ? uniform(arrival_key(at)) : kIdle;
          continue;
        }
      }
      --steps_left;
      npend = 0;
      int cm = -1, waiting = 0;  // the instance whose slot this event frees, and whether requests wait for it
      // requests released by this event: rel_first .. rel_first + rel_count - 1
      int32_t rel_first = 0, rel_count = 0;
      if (mn <= arr) {
        // completion on the lowest instance that has one at mn
        now = mn >> kInstBits;
        const int m = (int)(mn & kInstMask);
        const bool low = J == 1 || m < 32;
        HX_BOUND(m < N)
        const uint32_t tag = __shfl_sync(kFull, low ? next_tag[0] : next_tag[J - 1], m & 31);
        const int32_t rid = (int32_t)(tag >> 8);
        const int hole = (int)(tag & 15u);
        HX_BOUND(rid < nc)
        const CallRec* const r = rec + rid;
        const int4 tail = *reinterpret_cast<const int4*>(&r->tbar);
        const int est = *reinterpret_cast<const int*>(reinterpret_cast<const char*>(r) + (low ? lrec[0] : lrec[J - 1]));
        const InstState I = inst[m];
        const uint32_t slot_base = first_slot(m, I);
        HX_BOUND((int)slot_base + 16 <= c.slot_entries && hole < 16 && ((I.cfg & ~I.free) >> hole & 1u))
        // what the completion does.  A run of few warps reads the query's finished
        // chains and the first released request's costs before they are known to
        // be needed, so that no branch delays the loads.
        const int32_t qid = tail.z;
        HX_BOUND(qid >= 0 && qid < nq && tail.y >= 0 && tail.y < nc)
        const uint32_t tw = uniform((uint32_t)tail.w), what = tw >> kDoneShift;
        uint8_t* const chains = (kFew ? chains0 : W->chains) + qid;
        __builtin_assume(__isGlobal(chains));
        int ended = 0;
        if (kFew || what == kDoneChain) ended = *chains + 1;
        if (kFew) load_costs(tail.y);
        // the slot is free; the next completion is the earliest of those still running
        const uint32_t free = I.free | 1u << (tag & 31u);
        const bool failed = kFaults && (tag & kFailBit) != 0;
        const Slot e = slots[slot_base + l16];
        const bool runs = (I.cfg & ~free & lbit) != 0;
        const T nmin = warp_min(runs ? e.end : kIdle);
        unsigned nb = __ballot_sync(kFull, runs & (e.end == nmin));
        if (nb & (nb - 1)) {
          nb = lowest_id(runs & (e.end == nmin) ? e.tag : 0xffffffffu);  // equal ends
        }
        const uint32_t ntag = __shfl_sync(kFull, e.tag, 31 - __clz(nb));
        inst[m].free = free;  // every lane stores the same mask
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const bool own = lane + 32 * j == m;
          next_key[j] = own ? nmin << kInstBits | (T)m : next_key[j];
          next_tag[j] = own ? ntag : next_tag[j];
          q[j] -= own ? est : 0;
        }
        // whether the last chain ended, if one did, and whether requests wait for
        // the freed slot (only then does it need a batch boundary): one ballot, or
        // on a full GPU, whose busiest unit its bit tests would use, two votes
        // (8 x 20000 x 1024 on 64 instances 394 -> 380 ms; few warps +1 %)
        bool last, wait;
        if (kFew) {
          const unsigned flags = __ballot_sync(kFull, lane == 0 ? ended == (int)(tw & 0xff) : I.hsize > 0);
          last = flags & 1u;
          wait = flags & 2u;
        } else {
          last = __any_sync(kFull, ended == (int)(tw & 0xff));
          wait = __any_sync(kFull, I.hsize > 0);
        }
        cm = m;
        waiting = wait;
        // released: the next calls; at a chain's end the evaluation, if it is the last
        const bool chain = (what == kDoneChain) & !failed;
        rel_first = tail.y;
        rel_count = chain ? (int)last : (int)(tw & 0xff);
        if (chain) *chains = (uint8_t)ended;  // every lane writes the same byte
        if (kFaults && failed) {
          // the attempt timed out: the request goes out again, avoiding m
          const int32_t n = W->reissued + 1;
          __syncwarp();
          W->reissued = n;
          W->excl = c.n_inst > 1 ? m : -1;
          rel_first = rid;
          rel_count = 1;
          if (kFew) load_costs(rid);
        } else if (what == kDoneQuery) {
          const int64_t t_abs = absolute(now), dl = r->deadline, at = r->arrival;
          if (kGeneric) {
            const int ten = (tw >> 8) & 0xff;
            HX_BOUND(ten < HX_MAX_TENANTS)
            // every lane reads and writes the same, and the top-K's capacity is at
            // hand: one lane's branch and a load from global memory took longer
            // (24 traces of 2000 queries with competing requests x 64 points: 14.66 -> 14.31 ms)
            const int2 count = W->tcount[ten];
            const int kc = W->tkcap[ten];
            __syncwarp();
            W->tcount[ten] = make_int2(count.x + 1, count.y + (t_abs <= dl ? 1 : 0));
            if (a.tenant_kcap) {
              // this tenant's own top-K, for its P95 (Sec. 5's per-tenant tail latency)
              HX_BOUND(kc <= a.tenant_topk_off[0])
              const int64_t v = t_abs - at;
              if (__any_sync(kFull, (W->ttk[ten] < kc) | (v > W->ttkmin[ten])))
                topk_insert_warp(W->topk + a.tenant_topk_off[ten], &W->ttk[ten], kc, &W->ttkmin[ten], v, lane);
            }
          }
          digest_push<kWide>(W, dn, now, query_tag(qid), lane);
          finish_query(W, t_abs, at, dl, lane);
        }
        HX_BOUND(rel_first >= 0 && rel_count <= HX_MAX_K && rel_first + rel_count <= nc)
      } else {
        now = arr >> kInstBits;
        const int64_t qbase = W->qb;
        const int32_t qa = uniform(W->arrivals);
        HX_BOUND(qa < nq)
        rel_first = (int32_t)(a.qcall[qbase + qa] - W->cb);
        HX_BOUND(rel_first >= 0 && rel_first < nc)
        if (kFew) load_costs(rel_first);
        rel_count = 1;
        if (kFew) {
          // the query's records into L1, 32 bytes a lane (a copy that nobody reads)
          const char* pa = reinterpret_cast<const char*>(rec + rel_first);
          const char* const pe = reinterpret_cast<const char*>(rec + (a.qcall[qbase + qa + 1] - W->cb));
          const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&W->sink);
          for (pa += 32 * lane; pa < pe; pa += 1024)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(pa) : "memory");
        }
        __syncwarp();
        W->arrivals = qa + 1;  // every lane writes the same values
        const int64_t at = qa + 1 < nq ? a.arrival[qbase + qa + 1] : 0;
        W->next_arrival = at;
        arr = qa + 1 < nq ? uniform(arrival_key(at)) : kIdle;
      }

      // Sec. 4.1 for each released request, in request-id order: score every
      // instance and send it to the winner (its Sec. 4.2 key is formed at the
      // batch boundary below, and only if it has to wait).
      for (int32_t rid = rel_first; rel_count > 0; ++rid, --rel_count) {
        HX_BOUND(rid < nc)
        if (!kFew) load_costs(rid);
        int2 ev[J];
#pragma unroll
        for (int j = 0; j < J; ++j) ev[j] = cost_of[j];
        if (kFew && rel_count > 1) load_costs(rid + 1);
        int m;
        // a re-issued request avoids the instance it timed out on
        const int excl = kFaults ? uniform(W->excl) : -1;
        if (kGeneric && round_robin) {
          m = uniform(W->rr);
          if (m == excl) m = (m + 1 == N) ? 0 : m + 1;
          __syncwarp();
          W->rr = (m + 1 == N) ? 0 : m + 1;  // every lane writes the same value
        } else {
          // instances that tie in their reward and beat all others: the least cost wins
          // (the lowest instance at alpha = 0, where costs have no weight)
          const longlong2 tie = kFew ? tie0 : W->tie;
          T cost[J];  // << 6 | instance
#pragma unroll
          for (int j = 0; j < J; ++j)
            cost[j] = q[j] <= tie.x ? (T)((uint32_t)ev[j].x & (uint32_t)tie.y) << kInstBits | (T)(lane + 32 * j) : kIdle;
          const T least = warp_min(J == 2 && cost[J - 1] < cost[0] ? cost[J - 1] : cost[0]);
          if ((least != kIdle) & (excl < 0)) {
            m = (int)(least & kInstMask);
          } else {
            const float4 f = kFew ? fscore0 : W->fscore;
            ScoreRange s[J];
#pragma unroll
            for (int j = 0; j < J; ++j) s[j] = score_range(q[j], ev[j].x, f, neg_a[j]);
            const float lo = warp_max_f32(J == 2 ? fmaxf(s[0].lo, s[J - 1].lo) : s[0].lo);
            const unsigned b0 = __ballot_sync(kFull, s[0].hi >= lo);
            const unsigned b1 = J == 2 ? __ballot_sync(kFull, s[J - 1].hi >= lo) : 0u;
            // one instance's score can reach the best lower bound: it wins
            if ((((b0 & (b0 - 1)) | (b1 & (b1 - 1))) == 0) & ((b0 == 0) != (b1 == 0)) & (excl < 0)) {
              m = J == 1 || b0 ? __ffs(b0) - 1 : __ffs(b1) + 31;
            } else {
              m = exact_winner<J>(W, q[0], q[J - 1], ev[0].x, ev[J - 1].x, lane < N && lane != excl,
                                  J == 2 && lane + 32 < N && lane + 32 != excl, lane);
            }
          }
        }
        if (kFaults) W->excl = -1;
        HX_BOUND(m >= 0 && m < N)
        const bool low = J == 1 || m < 32;
        // the winner's costs, on its lane
        const int est = low ? ev[0].x : ev[J - 1].x, svc = low ? ev[0].y : ev[J - 1].y;
#pragma unroll
        for (int j = 0; j < J; ++j) q[j] += lane + 32 * j == m ? est : 0;
        if (kLog && recj >= 0) {
          // (the budget at send time follows from these: hx_log_kernel)
          HX_BOUND(rid < a.rec_calls)
          if (lane == 0) {
            a.rec_inst[2 * (int64_t)recj * a.rec_stride + rid] = m;
            a.rec_enq[(int64_t)recj * a.rec_stride + rid] = absolute(now);
          }
        }
        // nothing of this event waits yet, m's queue is empty and m has a free
        // slot for this request and every one still to be dispatched in this
        // event: the batch boundary below would start it now whatever the others
        // do, so it starts at once
        const InstState I = inst[m];
        if (__all_sync(kFull, ((npend | I.hsize) == 0) & (__popc(I.free) >= rel_count))) {
          start_call(m, I.free, first_slot(m, I), windows_on(I), rid, svc);
          continue;
        }
        // the local-queue key is formed only if the request has to wait
        HX_BOUND(npend < HX_MAX_K)
        if (lane == (m & 31)) W->pend[npend] = make_int4(rid, svc, est, m);
        npend++;
      }
      HX_STOP_IF_FAILED()

      // Batch boundary on the instance with a freed slot and requests waiting
      // for it, and on every instance this event's requests wait for: its free
      // slots go to the most urgent of the waiting requests and the new ones.
      if (npend | waiting) {
        const int lpol = kGeneric ? uniform(W->lpol) : HX_LOCAL_PQ;
        int m = cm;
        int4 pe = make_int4(0, 0, 0, -1);  // entry j on lane j
        unsigned left = 0, pm = 0;
        if (npend) {
          __syncwarp();
          if (lane < npend) pe = W->pend[lane];
          left = (1u << npend) - 1;
          if (!waiting) m = __shfl_sync(kFull, pe.w, 0);
        }
        for (;;) {
          HX_BOUND(m >= 0 && m < N)
          const InstState I = inst[m];
          uint32_t free = uniform(I.free);
          const uint32_t slot_base = first_slot(m, I);
          const int hs = uniform(I.hsize);
          HeapEnt* h = queue_of(I.heap);
#ifdef HX_CHECKED
          {
            // m's heap lies inside the warp's arena and holds at most its capacity
            const int hcl = (int)(I.heap >> kHeapCodeShift);
            const int64_t off = I.heap & kHeapOffMask, cap = hcl ? (int64_t)8 << hcl : 0;
            HX_BOUND(off + cap <= a.arena_per_warp && hs >= 0 && hs <= cap && (free & ~I.cfg & 0xffffu) == 0)
          }
#endif
          if (npend) {
            pm = __ballot_sync(kFull, pe.w == m);
            left &= ~pm;
          }
          // kEarly: where requests wait and one slot is free, the queue's top and its
          // root's children are loaded before the new request's key is formed, and
          // the first level of the sift is done before the start, so that the next
          // level's load passes meanwhile (32 x 5000 queries x 256 points on 16
          // instances 119.5 -> 116.1 ms, 19 x 5003 x 512 on 32 81.7 -> 79.4, a lone
          // 3000 queries on 64 26.6 -> 25.95).  The other two forms lose more where
          // no request waits: 8 x 2000 x 64 on 8 instances 6.24 -> 6.32, 8 x 20000 x
          // 1024 on 64 378 -> 385.
          constexpr bool kEarly = kFew == (J == 2);
          const bool single = hs > 0 && m == cm && __popc(pm) < 2;
          HeapEnt kid, top, e;
          if (kEarly && single) {
            kid = heap_child(h, 0, hs, lane);
            top = ent_load(h);
          }
          if (pm) {
            e.key = hs > 0 || __popc(pm) > __popc(free) ? queue_key(W, rec + pe.x, pe.z, absolute(now), lpol, pe.w == m) : 0;
            e.rid = pe.x;
            e.svc = pe.y;
          }
          if (kEarly ? single : hs > 0 && m == cm && __popc(pm) < 2) {
            if (!kEarly) {
              kid = heap_child(h, 0, hs, lane);
              top = ent_load(h);
            }
            // requests wait, so this event freed m's only free slot.  It goes to
            // the queue's top, or to the new request if that is more urgent; the
            // queue's last entry or the new one sinks from the top.
            int n = hs;
            bool fresh = false;
            if (pm) {
              const int j = __ffs(pm) - 1;
              e.key = __shfl_sync(kFull, e.key, j);
              e.rid = __shfl_sync(kFull, e.rid, j);
              e.svc = __shfl_sync(kFull, e.svc, j);
              fresh = __any_sync(kFull, ent_better(e, top));
            } else {
              e = ent_load(h + --n);
              if (lane + 1 >= n) kid.key = 0;  // the last entry is no child any more
              inst[m].hsize = n;  // every lane writes the same size
            }
            const int rid = fresh ? e.rid : top.rid, svc = fresh ? e.svc : top.svc;
            HX_BOUND(rid >= 0 && rid < nc)
            if (kFew && J == 2 && n >= kLongQueue) fetch_after(rid);
            int at = 0;
            bool more = false;
            if (kEarly && !fresh) more = heap_step(h, n, e, at, kid, lane);
            start_call(m, free, slot_base, windows_on(I), rid, svc);
            if (!fresh) {
              if (!kEarly || more) while (heap_step(h, n, e, at, kid, lane)) {}
              ent_store(h + at, e, (lane == 0) & (n > 0));
              __syncwarp();
            }
          } else {
            const bool direct = hs == 0 && __popc(pm) <= __popc(free);
            int n = 0;
            if (!direct) {
              status = push_pending(W, inst + m, e, pm, a.arena_per_warp, lane);
              if (status != HX_OK) break;
              h = queue_of(inst[m].heap);
              n = hs + __popc(pm);
            }
            // free slots: to all of this event's requests (an empty queue with
            // room for them), or to the most urgent
            while (free != 0 && (direct ? pm != 0 : n > 0)) {
              int rid, svc;
              if (direct) {
                const int j = __ffs(pm) - 1;
                pm &= pm - 1;
                rid = __shfl_sync(kFull, pe.x, j);
                svc = __shfl_sync(kFull, pe.y, j);
              } else {
                const HeapEnt top = ent_load(h), last = ent_load(h + --n);
                rid = top.rid;
                svc = top.svc;
                inst[m].hsize = n;  // every lane writes the same size
                heap_sift_warp(h, n, last, 0, heap_child(h, 0, n, lane), lane);
              }
              HX_BOUND(rid >= 0 && rid < nc)
              free = start_call(m, free, slot_base, windows_on(I), rid, svc);
            }
          }
          HX_STOP_IF_FAILED()
          if (left == 0) break;
          m = __shfl_sync(kFull, pe.w, __ffs(left) - 1);
        }
        if (status != HX_OK) break;
      }
      HX_STOP_IF_FAILED()
      if (kGeneric && a.checked) {
        // after every event: no instance keeps a slot free while requests wait
        // in its queue (Sec. 4.2: free slots take waiting requests at every
        // batch boundary) or has slots that are not its own, and t_queue stays
        // non-negative
        __syncwarp();
        bool bad = false;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const InstState I = inst[lane + 32 * j];
          bad |= (I.free != 0 && I.hsize > 0) || (I.free & ~I.cfg) != 0 || q[j] < 0;
        }
        if (__any_sync(kFull, bad)) {
          status = HX_ERR_INVARIANT;
          break;
        }
      }
    }

    digest_flush<kWide>(W, dn, lane);
    // conservation at the end: every dispatched request finished (t_queue back
    // to zero, no running call, no waiting request)
    bool left = false;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const InstState I = inst[lane + 32 * j];
      left |= (lane + 32 * j < N && q[j] != 0) || I.free != (I.cfg & 0xffffu) || I.hsize != 0;
    }
    const bool leftover = __any_sync(kFull, left);
    if (lane == 0) {
      int st = status;
      const int32_t n_done = W->n_done;
      const int32_t steps0 = W->nc + nq + 8 + (kFaults ? 16 * W->nc + 4096 : 0);
      const int64_t events = (steps0 - steps_left) - W->arrivals - (kFaults ? W->reissued : 0);
      // every query and every call completed exactly once
      if (st == HX_OK && (leftover || n_done != nq || events != W->nc)) st = HX_ERR_INVARIANT;
      hx_result res;
      res.p95_us = st == HX_OK ? (nq > 0 ? W->topk[0] : 0) : -1;
      res.makespan_us = W->makespan;
      res.events = events;
      res.digest = W->digest;
      res.slo_met = W->slo_met;
      res.n_done = n_done;
      res.status = st;
      const long long dc = (clock64() - W->clk0) >> 10;
      res.cycles_k = dc < INT32_MAX ? (int32_t)dc : INT32_MAX;
      a.results[W->sim] = res;
      if (kGeneric && a.extras) {
        hx_extra ex;
        for (int t = 0; t < HX_MAX_TENANTS; ++t) {
          ex.slo_met[t] = W->tcount[t].y;
          ex.n_done[t] = W->tcount[t].x;
          if (st != HX_OK) ex.p95_us[t] = -1;
          else if (!a.tenant_kcap) ex.p95_us[t] = t == 0 ? res.p95_us : 0;
          else ex.p95_us[t] = W->ttk[t] > 0 ? W->topk[a.tenant_topk_off[t]] : 0;
        }
        ex.reissued = W->reissued;
        ex.pad = 0;
        a.extras[W->sim] = ex;
      }
    }
    __syncwarp();
  }
  // the last prefetches' copies land before the block's shared memory is given back
  if (kFew) asm volatile("cp.async.wait_all;" ::: "memory");
}

#define HX_SIM_KERNEL(name, family)                                                                   \
  template <int J, bool kFew>                                                                         \
  __global__ void __launch_bounds__(kWarpsPerBlock * 32, kFew ? kFewMinBlocks : HX_SIM_MIN_BLOCKS(J)) \
      name(SimArgs a, ClusterK c) {                                                                   \
    sim_body<J, family, kFew>(a, c);                                                                  \
  }
HX_SIM_KERNEL(hx_sim_kernel_lean, kSimLean)
HX_SIM_KERNEL(hx_sim_kernel_log, kSimLog)
HX_SIM_KERNEL(hx_sim_kernel, kSimGeneric)
HX_SIM_KERNEL(hx_sim_kernel_faults, kSimFaults)
HX_SIM_KERNEL(hx_sim_kernel_wide, kSimWide)
#undef HX_SIM_KERNEL

#define HX_FORMS(name) name<2, false>, name<1, false>, name<2, true>, name<1, true>
const SimKernel kSimKernel[kSimKernels] = {HX_FORMS(hx_sim_kernel_lean), HX_FORMS(hx_sim_kernel_log),
                                           HX_FORMS(hx_sim_kernel), HX_FORMS(hx_sim_kernel_faults),
                                           HX_FORMS(hx_sim_kernel_wide)};
#undef HX_FORMS

// ----------------------------------------------------------- log kernel
// The SLO budget at send time (Sec. 4.2) of every logged dispatch, one thread
// per call of a logged simulation: its division (a hundred instructions) in the
// event loop would lengthen the logged simulation's chain, which one window's
// sweep waits for.
__global__ void __launch_bounds__(256) hx_log_kernel(LogArgs a, ClusterK c) {
  __shared__ int64_t rest[kFRows];
  const int64_t per = (a.rec_calls + 255) / 256;  // blocks of calls per simulation
  for (int64_t b = blockIdx.x; b < per * a.n_record; b += gridDim.x) {
    const int64_t j = b / per;
    const int64_t sim = a.record_sims[j], t = sim / a.n_points;
    __syncthreads();
    if (threadIdx.x < kFRows) rest[threadIdx.x] = rest_of_path(c, a.rho[sim - t * a.n_points], threadIdx.x);
    __syncthreads();
    const int64_t rid = (b - j * per) * 256 + threadIdx.x;
    if (rid < a.c_off[t + 1] - a.c_off[t]) {
      const CallRec* const r = a.rec + a.c_off[t] + rid;
      const int64_t o = j * a.rec_stride + rid, dd = r->tbar + rest[r->fcode];
      a.rec_budget[o] = slo_budget(r->deadline - a.rec_enq[o], r->tbar, dd);
    }
  }
}

// ---------------------------------------------------------- best kernel
namespace {

__device__ __forceinline__ bool cand_better(const BestCand& x, const BestCand& y, int obj) {
  const bool xv = x.flags & 1, yv = y.flags & 1;
  if (xv != yv) return xv;
  if (!xv) return x.p < y.p;
  if (obj == HX_OBJ_P95_SLO95) {
    const bool xf = (x.flags >> 1) & 1, yf = (y.flags >> 1) & 1;
    if (xf != yf) return xf;
    if (!xf && x.slo != y.slo) return x.slo > y.slo;
  }
  if (x.p95 != y.p95) return x.p95 < y.p95;
  return x.p < y.p;
}

__device__ void block_reduce_best(BestCand mine[2], BestCand* out) {
  __shared__ BestCand red[2][256];
  for (int o = 0; o < 2; ++o) red[o][threadIdx.x] = mine[o];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      for (int o = 0; o < 2; ++o)
        if (cand_better(red[o][threadIdx.x + w], red[o][threadIdx.x], o)) red[o][threadIdx.x] = red[o][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = red[0][0];
    out[1] = red[1][0];
  }
}

}  // namespace

// Blocks 0..T-1: best point of trace t; block T: best point of the sums over traces.
__global__ void __launch_bounds__(256) hx_best_kernel(BestArgs a) {
  const int P = a.n_points;
  BestCand mine[2];
  for (int o = 0; o < 2; ++o) {
    mine[o].p95 = 0;
    mine[o].slo = 0;
    mine[o].p = INT32_MAX;
    mine[o].flags = 0;
  }
  if ((int)blockIdx.x < a.n_traces) {
    const int t = blockIdx.x;
    const int64_t nq = a.q_off[t + 1] - a.q_off[t];
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
      const hx_result r = a.results[(int64_t)t * P + p];
      BestCand x;
      x.p95 = r.p95_us;
      x.slo = r.slo_met;
      x.p = p;
      x.flags = (r.status == HX_OK ? 1 : 0) | ((int64_t)r.slo_met * 100 >= 95 * nq ? 2 : 0);
      for (int o = 0; o < 2; ++o)
        if (cand_better(x, mine[o], o)) mine[o] = x;
    }
    block_reduce_best(mine, a.per_trace + 2 * t);
  } else {
    const int64_t nsum = a.q_off[a.n_traces] - a.q_off[0];
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
      BestCand x;
      x.p95 = 0;
      x.slo = 0;
      x.p = p;
      int valid = 1;
      for (int t = 0; t < a.n_traces; ++t) {
        const hx_result r = a.results[(int64_t)t * P + p];
        x.p95 += r.p95_us;
        x.slo += r.slo_met;
        valid &= r.status == HX_OK ? 1 : 0;
      }
      x.flags = valid | (x.slo * 100 >= 95 * nsum ? 2 : 0);
      if (a.point_sums) {
        a.point_sums[3 * p] = x.p95;
        a.point_sums[3 * p + 1] = x.slo;
        a.point_sums[3 * p + 2] = valid ? 0 : 1;
      }
      for (int o = 0; o < 2; ++o)
        if (cand_better(x, mine[o], o)) mine[o] = x;
    }
    block_reduce_best(mine, a.global);
  }
}

// Self-test of udiv_trial against the compiler's division.
__global__ void hx_selftest_div_kernel(const uint64_t* n, const uint64_t* d, uint64_t* q, uint64_t* q_ref,
                                       int64_t count) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) {
    q[i] = udiv_trial(n[i], d[i]);
    q_ref[i] = n[i] / d[i];
  }
}

}  // namespace hx
