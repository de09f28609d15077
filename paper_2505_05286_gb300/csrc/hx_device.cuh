// hx_device.cuh -- device-side data layout and kernels of the batched
// HexGen-Flow scheduler simulation (arXiv 2505.05286, Sec. 4) for sm_103a.
//
//   hx_prep_kernel  : per query, Eq. (comp) per call and instance type, the
//                     mean cost tbar of Sec. 4.2, workflow successor links
//                     (Sec. 2.1) and the query deadline (SLO of Sec. 5.1);
//                     writes one 64-byte record per call.
//   hx_sim_kernel   : persistent; one warp runs one (trace, point) discrete
//                     event simulation of the workload-balanced dispatcher
//                     (Sec. 4.1) and the urgency queues (Sec. 4.2), and
//                     reduces it to P95 / SLO count / digest (Sec. 4.3).
//   hx_log_kernel   : the SLO budgets (Sec. 4.2) of logged simulations' calls.
//   hx_best_kernel  : argmin of the P95 objective per trace and over the grid.
#pragma once

#include <stdint.h>

#include "hxsim.h"

namespace hx {

constexpr int64_t kScale = 1000000;       // fixed point of alpha, gamma, slo_mult
constexpr int64_t kUsPerS = 1000000;      // prefill throughput is per second
constexpr int64_t kRewardCap = (int64_t(1) << 43) - 1;
constexpr int64_t kLongCall = int64_t(1) << 25;  // us; attempts this long need 64-bit event times
constexpr int kWarpsPerBlock = 4;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kFRows = 18;                // S, G/C with 0..15 corrections done, E

// What a completion does: release the k calls from `next` on, end a chain of
// the query (the last of its k chains releases `next`), end the query.
enum { kDoneRelease = 0, kDoneChain = 1, kDoneQuery = 2 };
constexpr int kDoneShift = 24;  // of the last four bytes as one word

// One call as the simulator reads it: 64 bytes, 16-byte aligned.
struct __align__(16) CallRec {
  int2 ev[4];         // per type: Eq. (comp) with the believed output length, and the
                      // same with the true output length (service time)
  int64_t deadline;   // query arrival + T_slo
  int64_t arrival;    // query arrival
  int32_t tbar;       // mean of est over the instances
  int32_t next;       // S: G_0; G/C: the next correction, or E at the end of the chain
  int32_t qid;        // query index within the trace
  uint8_t k, u, fcode, done;  // calls that its completion releases, or at a chain's end the
                              // query's chains; corrections done incl. this call (E: the
                              // query's tenant); row of the rest-of-path table: S 0, G/C 1 + u,
                              // E 17; what its completion does (kDone*)
};
static_assert(sizeof(CallRec) == 64, "CallRec is one 64-byte unit");

// Local-queue entry: priority key + 2^63 (higher first) and request id (lower first).
struct __align__(16) HeapEnt {
  unsigned long long key;
  int rid;
  int svc;   // service time on the queue's instance
};

// A fault window of one instance (see hx_fault).
struct FaultK {
  int64_t t0, t1, slow;
  int32_t inst, pad;
};

// Cluster description passed by value (kernel parameter space).
struct ClusterK {
  int32_t n_inst, n_types, ref_type, rmax;
  int64_t slo_mult_fp;
  int32_t prefill[HX_MAX_TYPES], decode[HX_MAX_TYPES], slots[HX_MAX_TYPES], cnt[HX_MAX_TYPES];
  int32_t ref_prompt[4], ref_out[4];
  int32_t slot_entries;     // slot entries per warp, packed; the kernel's own at launch
  int32_t smem_per_warp;
  uint8_t inst_type[HX_MAX_INST];
  uint8_t inst_slots[HX_MAX_INST];
  uint16_t slot_base[HX_MAX_INST];
  // tenants and faults (only the last two kernel families handle faults)
  int32_t n_tenants, n_faults;
  int64_t tenant_mult[HX_MAX_TENANTS];
  int64_t timeout_mult_fp;
  FaultK faults[HX_MAX_FAULTS];
};

struct PrepArgs {
  const int64_t* arrival;   // [Q]
  const uint8_t* kq;        // [Q]
  const int64_t* qcall;     // [Q + 1] first call (global index) of each query
  const int64_t* q_off;     // [T + 1]
  const int64_t* c_off;     // [T + 1]
  const int32_t* prompt;
  const int32_t* out;
  const int32_t* out_est;
  const uint8_t* stage;
  const uint8_t* cand;
  const uint8_t* retry;
  const uint8_t* tenant;    // [Q] or NULL
  int64_t n_queries;
  int32_t n_traces;
  CallRec* rec;             // [C]
  unsigned long long* work_counter;
  hx_result* skip_results;  // with a subset: every result starts as HX_SKIPPED
  hx_extra* skip_extras;    // and its per-tenant counts at zero (NULL: none kept)
  int64_t n_skip;           // n_sims with a subset, else 0
};

struct SimArgs {
  const CallRec* rec;
  const int64_t* arrival;
  const int64_t* qcall;
  const int64_t* q_off;
  const int64_t* c_off;
  const int64_t* alpha;
  const int64_t* gamma;
  const int32_t* rho;
  const int64_t* beta;
  const uint8_t* lpol;
  const uint8_t* dpol;
  int32_t n_points;
  int32_t n_traces;
  int64_t n_sims;
  hx_result* results;
  unsigned long long* work_counter;
  HeapEnt* arena;           // per resident warp: arena_per_warp entries
  int64_t arena_per_warp;
  uint8_t* chains;          // per resident warp: chains_per_warp bytes (a multiple of 16)
  int64_t chains_per_warp;
  int64_t* topk;            // per resident warp: topk_per_warp latencies
  int64_t topk_per_warp;
  const int32_t* rec_map;   // [n_sims] record slot or -1; NULL when not recording
  int32_t* rec_inst;
  int64_t* rec_enq;
  int64_t* rec_start;
  int64_t* rec_end;
  int64_t rec_calls, rec_stride;  // calls and int64 units per logged simulation
  hx_extra* extras;         // [n_sims] per-tenant counts and re-issues (generic kernel), or NULL
  const int32_t* tenant_kcap;  // [n_traces * 4] top-K size per (trace, tenant) (0: no queries), or
                               // NULL: one tenant
  int64_t tenant_topk_off[HX_MAX_TENANTS];  // tenant t's top-K heap within the warp's topk slice
  const int64_t* subset;    // [n_work] sims to run in work order, or NULL: all n_sims
  int64_t n_work;
  int32_t checked;          // check the scheduler's invariants after every event (generic kernel)
};

// A running call in its batch slot: end time and request id << 8 | kFailBit if the
// attempt times out at its end | slot.
constexpr uint32_t kFailBit = 0x80;
struct __align__(8) Slot32 {
  uint32_t end, tag;
};
struct __align__(16) Slot64 {
  uint64_t end;
  uint32_t tag, pad;
};

// One instance as every lane reads it (one 16-byte load).  Its t_queue and next
// completion are in its owner lane's registers.
struct __align__(16) InstState {
  uint32_t free;                // free batch slots, one bit each
  int32_t hsize;                // local queue: heap size
  uint32_t heap;                // local queue: heap offset in the arena, capacity code << 27
                                // (8 << code entries; 0: none yet)
  uint32_t cfg;                 // its slots' mask, first slot << 16, kWindowsBit: it has fault windows
};
constexpr uint32_t kWindowsBit = 1u << 31;
constexpr int kHeapCodeShift = 27;  // the arena holds at most 4 * 2^24 + 1024 entries
constexpr uint32_t kHeapOffMask = (1u << kHeapCodeShift) - 1;

// Whether every instance has 16 slot entries, so that no load gives the first; if
// not, it has its own slots only, and 16 entries follow the last instance's.  64-bit
// times spaced (8 KB a warp) would let 20 warps reside on an SM where the registers of
// the full GPU's form let 32: there they are packed (64 traces x 2000 queries x 64
// points on 8 instances 29.4 -> 21.5 ms, 32 x 2000 x 256 on 16 81.4 -> 69.4), and spaced
// in the form for few warps (packed, 8 x 2000 x 64 takes 9.53 ms against 9.33).
__host__ __device__ constexpr bool spaced_slots(int instances_per_lane, bool wide, bool few) {
  return instances_per_lane == 1 && (!wide || few);
}

// Per-warp shared memory of one simulation: per-simulation constants and
// warp-uniform state, then an InstState per lane and instance of it and the
// slot entries, which are read 16 at a time (spaced_slots()).
struct __align__(16) WarpShared {
  int4 pend[HX_MAX_K];          // this event's waiting dispatches: request id, service time and
                                // Eq. (comp) on the instance, instance
  uint4 dterm[16];              // digest terms waiting to be hashed: 32 of (relative time, id
                                // tag), with 64-bit times 16
  longlong2 tie;                // t_queue up to which the least cost alone decides a dispatch; cost mask
  float4 fscore;                // the score filter's constants (score_range)
  // per-simulation constants
  int64_t G, beta;
  int64_t frest[kFRows];        // rest-of-path cost of the budget denominator by fcode
  int32_t A, one_minus_a;       // alpha and 1 - alpha, fixed point
  int32_t lpol, kcap, rr, bump;
  // this warp's scratch slices and the current trace's offsets
  HeapEnt* arena;
  uint8_t* chains;              // finished chains per query
  int64_t* topk;
  int64_t qb, cb;
  int32_t nq, nc;
  int64_t sim, clk0;            // result index and start clock of the simulation
  int64_t base;                 // what the 32-bit event times are relative to (written alike by every lane)
  int64_t next_arrival;         // time of the next arrival (likewise)
  int32_t arrivals;             // arrivals taken so far (likewise)
  uint64_t digest;
  int64_t makespan;
  int32_t n_done, slo_met, sink, tk;  // sink: where prefetched records are copied to
  int64_t tkmin;                // root of the full top-K heap (written alike by every lane)
  int2 tcount[HX_MAX_TENANTS];  // per tenant: completed queries, SLO hits (generic kernel)
  int32_t tkcap[HX_MAX_TENANTS], ttk[HX_MAX_TENANTS];  // per-tenant top-K heaps: capacities, entries
  int64_t ttkmin[HX_MAX_TENANTS];  //                 and roots once full
  int32_t reissued, excl;       // timed-out attempts; the instance a re-issue avoids (-1: none)
};
static_assert(sizeof(WarpShared) % 16 == 0, "InstState follows");

struct BestCand {
  int64_t p95;
  int64_t slo;
  int32_t p;
  int32_t flags;  // bit0 valid, bit1 feasible
};

struct LogArgs {
  const CallRec* rec;
  const int64_t* c_off;
  const int32_t* rho;
  const int32_t* record_sims;  // [n_record]
  int32_t n_record, n_points;
  const int64_t* rec_enq;
  int64_t* rec_budget;
  int64_t rec_calls, rec_stride;
};

struct BestArgs {
  const hx_result* results;
  const int64_t* q_off;
  int32_t n_traces;
  int32_t n_points;
  BestCand* per_trace;      // [T * 2]
  BestCand* global;         // [2]
  int64_t* point_sums;      // [P * 3] (sum P95, sum SLO hits, failed sims) or NULL
};

__global__ void hx_prep_kernel(PrepArgs a, ClusterK c);
// The instantiations of the simulation kernel.  hx_sim_kernel_lean: every point
// workload-balanced with the urgency queue, nothing logged; hx_sim_kernel_log:
// with per-call logs; hx_sim_kernel: those and any mix of dispatch and
// local-queue policies, tenants and event checks; hx_sim_kernel_faults: all of
// it with fault windows; hx_sim_kernel_wide: all of it with attempts of kLongCall
// us and more (64-bit times).  Each for clusters of up to 64 instances, two a lane,
// and of up to 32, one a lane, and both for a full GPU and for a run of few
// warps: kernel 4 * family + 2 * few + (one a lane).
enum { kSimLean = 0, kSimLog = 1, kSimGeneric = 2, kSimFaults = 3, kSimWide = 4 };
using SimKernel = void (*)(SimArgs, ClusterK);
constexpr int kSimKernels = 20;
extern const SimKernel kSimKernel[kSimKernels];
__global__ void hx_log_kernel(LogArgs a, ClusterK c);
__global__ void hx_best_kernel(BestArgs a);
__global__ void hx_selftest_div_kernel(const uint64_t* n, const uint64_t* d, uint64_t* q, uint64_t* q_ref,
                                       int64_t count);

}  // namespace hx
