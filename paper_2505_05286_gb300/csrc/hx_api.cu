// hx_api.cu -- the C ABI (include/hxsim.h): input validation, flattening of
// the traces into device arrays, per-warp scratch sizing and the launches of
// the preparation, simulation and best-point kernels on the caller's stream.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstddef>
#include <cstring>
#include <exception>
#include <memory>
#include <mutex>
#include <stdexcept>
#include <system_error>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "hx_device.cuh"

namespace {

thread_local std::string g_err;

// NVTX range over one ABI call (host side: validation, copies, launches), for
// profilers that group kernels by range (e.g. ncu --nvtx).
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

// Host-side C++ exceptions (an allocation that fails) become a status
// here instead of crossing the C ABI.
template <class F>
int guarded(F&& f) noexcept {
  const char* msg = "unexpected host exception";
  int code = HX_ERR_STATE;
  try {
    return f();
  } catch (const std::bad_alloc&) {
    msg = "host allocation failed";
    code = HX_ERR_OOM;
  } catch (const std::length_error&) {
    msg = "host allocation failed";
    code = HX_ERR_OOM;
  } catch (...) {
  }
  try {
    g_err = msg;
  } catch (...) {
  }
  return code;
}

#define HX_CUDA(x)                                                                   \
  do {                                                                               \
    cudaError_t e_ = (x);                                                            \
    if (e_ != cudaSuccess)                                                           \
      return fail(e_ == cudaErrorMemoryAllocation ? HX_ERR_OOM : HX_ERR_CUDA,        \
                  std::string(#x) + ": " + cudaGetErrorString(e_));                  \
  } while (0)

constexpr int64_t kTokMax = int64_t(1) << 20;     // prompt / output tokens per call
constexpr int64_t kCostMax = int64_t(1) << 28;    // any per-call cost bound, us
constexpr int64_t kHorizonMax = int64_t(1) << 39; // last arrival + all service, us

int64_t align_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

// The dynamic shared-memory limit of a kernel (cudaFuncAttributeMax-
// DynamicSharedMemorySize) is one setting per function and device, shared by
// every handle in the process.  It is set, under a mutex, to the largest size
// any launch of that kernel on that device has asked for, so a later handle
// or static call with a smaller cluster never lowers it below what an earlier
// handle launches with.  Called before every launch; it sets the attribute
// each time (a host-side call), so a device reset cannot leave it lower than
// the record says.
constexpr int kMaxDevices = 64;
std::mutex g_smem_mu;
int g_smem_limit[kMaxDevices][hx::kSimKernels] = {};  // [device][kernel]

// The instantiation of the simulation kernel for a cluster; few: a run of few
// warps.  That one fetches a query's records into L1 as it arrives (an event
// reads two sectors of them that would come from L2 otherwise, about a fifth of
// its latency) and may use twice the registers.
int sim_kernel_of(int family, const hx::ClusterK& ck, bool few) {
  return 4 * family + (few ? 2 : 0) + (ck.n_inst <= 32 ? 1 : 0);
}

// Few warps: up to the 20 per SM that those kernels' registers let reside.  Against
// the full GPU's form: 1216 to 3040 warps 6 to 22 % faster (36 traces x 2000
// queries x 64 points 11.5 -> 8.9 ms, 2560 warps on 64 instances 80 -> 75 ms); runs
// of several waves are faster in the full form (8192 simulations on 16 instances
// 119 ms against 137).
bool few_warps(int64_t warps, int sms) { return warps <= 20 * (int64_t)sms; }

int ensure_dyn_smem(int kernel, int bytes) {
  int dev = 0;
  HX_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return fail(HX_ERR_INVALID, "device index out of range");
  std::lock_guard<std::mutex> lock(g_smem_mu);
  int& cur = g_smem_limit[dev][kernel];
  const int want = std::max(cur, bytes);
  if (cudaFuncSetAttribute((const void*)hx::kSimKernel[kernel], cudaFuncAttributeMaxDynamicSharedMemorySize, want) != cudaSuccess) {
    cudaGetLastError();
    return fail(HX_ERR_CUDA, "cannot reserve " + std::to_string(want) +
                                 " bytes of shared memory for the simulation kernel");
  }
  cur = want;
  return HX_OK;
}

// The family of the simulation kernel that serves a run: the lean one serves
// grids that are all workload-balanced dispatch with the urgency queue, log
// nothing, check nothing, count one tenant and have no fault windows.  (The wide
// one serves any run of traces with an attempt of kLongCall us or more.)
int sim_family(const hx_grid* grid, const hx::ClusterK& ck, bool record, bool force, bool checked) {
  if (ck.n_faults > 0) return hx::kSimFaults;
  bool generic = force || checked || ck.n_tenants > 1;
  for (int p = 0; p < grid->n_points; ++p)
    generic |= grid->local_policy[p] != HX_LOCAL_PQ || grid->dispatch_policy[p] != HX_DISPATCH_WB;
  return generic ? hx::kSimGeneric : record ? hx::kSimLog : hx::kSimLean;
}

}  // namespace

struct hx_sim {
  int32_t n_traces = 0, n_points = 0;
  int64_t n_sims = 0, n_q = 0, n_c = 0;
  int32_t max_nq = 0, max_nc = 0, max_kcap = 1;
  hx::ClusterK ck{};
  int32_t n_tenants = 0;          // as given in hx_cluster (validation of later uploads)
  std::vector<hx_fault> faults;
  std::vector<int32_t> h_nq, h_nc;
  std::vector<int64_t> q_off, c_off;  // [n_traces + 1]
  // device: inputs
  int64_t* d_arrival = nullptr;
  int64_t* d_qcall = nullptr;
  int64_t* d_q_off = nullptr;
  int64_t* d_c_off = nullptr;
  uint8_t* d_k = nullptr;
  uint8_t* d_tenant = nullptr;
  int32_t* d_prompt = nullptr;
  int32_t* d_out = nullptr;
  int32_t* d_out_est = nullptr;
  uint8_t* d_stage = nullptr;
  uint8_t* d_cand = nullptr;
  uint8_t* d_retry = nullptr;
  int64_t* d_alpha = nullptr;
  int64_t* d_gamma = nullptr;
  int64_t* d_beta = nullptr;
  int32_t* d_rho = nullptr;
  uint8_t* d_lp = nullptr;
  uint8_t* d_dp = nullptr;
  // device: derived and outputs
  hx::CallRec* d_rec = nullptr;
  hx_result* d_results = nullptr;
  hx_extra* d_extras = nullptr;  // generic families only
  unsigned long long* d_counter = nullptr;
  hx::BestCand* d_best_trace = nullptr;
  hx::BestCand* d_best_global = nullptr;
  int64_t* d_point_sums = nullptr;
  // per-tenant top-K heaps (generic kernel with several tenants)
  int32_t* d_tenant_kcap = nullptr;
  int64_t tenant_topk_off[HX_MAX_TENANTS] = {0, 0, 0, 0};
  // device: scratch
  hx::HeapEnt* d_arena = nullptr;
  uint8_t* d_chains = nullptr;
  int64_t* d_topk = nullptr;
  int64_t arena_per_warp = 0, chains_per_warp = 0, topk_per_warp = 0;
  // device: records
  int32_t n_record = 0;
  int64_t rec_calls = 0, rec_stride = 0;  // calls and int64 units per logged simulation
  int64_t* d_rec_log = nullptr;
  int32_t* d_rec_map = nullptr;
  int32_t* d_rec_sims = nullptr;
  // run only these simulations, in work order (NULL: all of them)
  int64_t* d_subset = nullptr;  // the work order when not the kernel's own (see work_order)
  int64_t n_work = 0;
  int32_t work_order = 0;       // hx_info.work_order
  bool checked = false;
  std::vector<int32_t> record_sims;
  // the simulation kernel's family and launch for the traces as they are: [0] with
  // short calls only, [1] with an attempt of kLongCall us or more
  struct Launch {
    int family = hx::kSimWide, kernel = 0, blocks = 0, smem_per_block = 0, slot_entries = 0;
  } launch[2];
  bool long_calls = false;
  int32_t* d_long = nullptr;    // the same on the device, for captured runs
  const Launch& shape() const { return launch[long_calls ? 1 : 0]; }
  int64_t scratch_bytes = 0, device_bytes = 0;
  cudaStream_t last_stream = nullptr;
  bool ran = false;
  bool timing = false;
  // with timing: four events per run (before prep, before and after the
  // simulations, after the best point) for the last kTimedRuns runs
  static constexpr int kTimedRuns = 64;
  std::vector<cudaEvent_t> ev;
  int64_t runs = 0;
  cudaEvent_t* run_ev(int64_t r) { return ev.data() + 4 * (r % kTimedRuns); }
  // Everything the handle holds on the device is one block, laid out by place()
  // and allocated by commit() (28 allocations and as many frees took 260 us of a
  // fresh 2.8 ms window sweep; one of each takes 65).
  unsigned char* block = nullptr;
  std::vector<std::pair<void**, int64_t>> placed;
  // The inputs lead it: the per-query arrays, the constants of cluster and grid and
  // the per-call arrays.  `stage` is the same on the host, so that an upload is one
  // copy (64 traces' 384 copies took 2.5 ms).  The per-call arrays are staged while
  // that is cheaper than six copies a trace from the caller's (see stage_calls_of);
  // otherwise they are copied from there and no stage is kept.
  std::unique_ptr<unsigned char[]> stage;
  int64_t query_bytes = 0, const_bytes = 0, input_bytes = 0;  // ends of the three parts
  bool stage_calls = false;

  template <class T>
  void place(T** p, int64_t count) {
    placed.emplace_back(reinterpret_cast<void**>(p), device_bytes);
    device_bytes += align_up(std::max<int64_t>(count, 1) * (int64_t)sizeof(T), 256);
  }
  int commit() {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, (size_t)device_bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(HX_ERR_OOM, "cudaMalloc of " + std::to_string(device_bytes) + " bytes: " + cudaGetErrorString(e));
    }
    block = static_cast<unsigned char*>(q);
    for (const auto& p : placed) *p.first = block + p.second;
    return HX_OK;
  }
  // where the host copy of a device input is
  template <class T>
  T* staged(T* d) const {
    return reinterpret_cast<T*>(stage.get() + (reinterpret_cast<unsigned char*>(d) - block));
  }

  ~hx_sim() {
    cudaFree(block);
    for (auto e : ev)
      if (e) cudaEventDestroy(e);
  }
};

namespace {

int validate_cluster(const hx_cluster* c, int64_t* min_prefill, int64_t* max_decode) {
  if (!c) return fail(HX_ERR_INVALID, "cluster is NULL");
  if (c->n_types < 1 || c->n_types > HX_MAX_TYPES) return fail(HX_ERR_INVALID, "n_types must be 1..4");
  if (c->n_inst < 1 || c->n_inst > HX_MAX_INST) return fail(HX_ERR_INVALID, "n_inst must be 1..64");
  if (!c->prefill_tok_s || !c->decode_us_tok || !c->slots || !c->inst_type || !c->stage_ref_prompt ||
      !c->stage_ref_out)
    return fail(HX_ERR_INVALID, "cluster array is NULL");
  int64_t mp = INT64_MAX, md = 0;
  for (int t = 0; t < c->n_types; ++t) {
    if (c->prefill_tok_s[t] < 1) return fail(HX_ERR_INVALID, "prefill_tok_s must be >= 1");
    if (c->decode_us_tok[t] < 0) return fail(HX_ERR_INVALID, "decode_us_tok must be >= 0");
    if (c->slots[t] < 1 || c->slots[t] > HX_MAX_SLOTS) return fail(HX_ERR_INVALID, "slots must be 1..16");
    mp = std::min<int64_t>(mp, c->prefill_tok_s[t]);
    md = std::max<int64_t>(md, c->decode_us_tok[t]);
  }
  for (int m = 0; m < c->n_inst; ++m)
    if (c->inst_type[m] >= c->n_types) return fail(HX_ERR_INVALID, "inst_type out of range");
  if (c->ref_type < 0 || c->ref_type >= c->n_types) return fail(HX_ERR_INVALID, "ref_type out of range");
  if (c->slo_mult_fp < 0 || c->slo_mult_fp > 16 * HX_SCALE) return fail(HX_ERR_INVALID, "slo_mult_fp must be 0..16*SCALE");
  if (c->rmax < 0 || c->rmax > HX_MAX_RETRY) return fail(HX_ERR_INVALID, "rmax must be 0..15");
  for (int s = 0; s < 4; ++s) {
    const int64_t p = c->stage_ref_prompt[s], o = c->stage_ref_out[s];
    if (p < 0 || p > kTokMax || o < 0 || o > kTokMax) return fail(HX_ERR_INVALID, "stage reference tokens out of range");
    if ((p * 1000000 + mp - 1) / mp + o * md >= kCostMax) return fail(HX_ERR_INVALID, "stage reference cost too large");
  }
  if (c->n_tenants < 0 || c->n_tenants > HX_MAX_TENANTS) return fail(HX_ERR_INVALID, "n_tenants must be 0..4");
  if (c->tenant_slo_mult_fp)
    for (int t = 0; t < std::max(c->n_tenants, 1); ++t)
      if (c->tenant_slo_mult_fp[t] < 0 || c->tenant_slo_mult_fp[t] > 16 * HX_SCALE)
        return fail(HX_ERR_INVALID, "tenant_slo_mult_fp must be 0..16*SCALE");
  if (c->timeout_mult_fp != 0 && (c->timeout_mult_fp < HX_SCALE || c->timeout_mult_fp > 100 * HX_SCALE))
    return fail(HX_ERR_INVALID, "timeout_mult_fp must be 0 or SCALE..100*SCALE");
  if (c->n_faults < 0 || c->n_faults > HX_MAX_FAULTS) return fail(HX_ERR_INVALID, "n_faults must be 0..16");
  if (c->n_faults > 0 && !c->faults) return fail(HX_ERR_INVALID, "faults is NULL");
  for (int f = 0; f < c->n_faults; ++f) {
    const hx_fault& F = c->faults[f];
    if (F.inst < 0 || F.inst >= c->n_inst) return fail(HX_ERR_INVALID, "fault instance out of range");
    if (F.t0_us < 0 || F.t1_us < F.t0_us || F.t1_us > (int64_t(1) << 38))
      return fail(HX_ERR_INVALID, "fault window must satisfy 0 <= t0 <= t1 <= 2^38");
    if (F.slow_fp != 0 && (F.slow_fp < HX_SCALE / 100 || F.slow_fp > 100 * HX_SCALE))
      return fail(HX_ERR_INVALID, "fault slow_fp must be 0 or SCALE/100..100*SCALE");
    if (F.slow_fp == 0 && c->timeout_mult_fp == 0)
      return fail(HX_ERR_INVALID, "a stopped instance (slow_fp = 0) needs a timeout");
  }
  *min_prefill = mp;
  *max_decode = md;
  return HX_OK;
}

int validate_grid(const hx_grid* g) {
  if (!g) return fail(HX_ERR_INVALID, "grid is NULL");
  if (g->n_points < 1) return fail(HX_ERR_INVALID, "n_points must be >= 1");
  if (!g->alpha_fp || !g->gamma_fp || !g->rho || !g->beta_us2 || !g->local_policy || !g->dispatch_policy)
    return fail(HX_ERR_INVALID, "grid array is NULL");
  for (int p = 0; p < g->n_points; ++p) {
    if (g->alpha_fp[p] < 0 || g->alpha_fp[p] > HX_SCALE) return fail(HX_ERR_INVALID, "alpha_fp must be 0..SCALE");
    if (g->gamma_fp[p] < 0 || g->gamma_fp[p] > 4 * HX_SCALE) return fail(HX_ERR_INVALID, "gamma_fp must be 0..4*SCALE");
    if (g->rho[p] < 0 || g->rho[p] > HX_MAX_RETRY) return fail(HX_ERR_INVALID, "rho must be 0..15");
    if (g->beta_us2[p] < 0 || g->beta_us2[p] > (int64_t(1) << 62)) return fail(HX_ERR_INVALID, "beta_us2 out of range");
    if (g->local_policy[p] > 2 || g->dispatch_policy[p] > 1) return fail(HX_ERR_INVALID, "unknown policy");
  }
  return HX_OK;
}

// Counts that no valid trace has (a query has at least one call): nothing may be
// read or sized by them.
bool bad_counts(const hx_trace& tr) {
  return tr.n_queries < 0 || tr.n_calls < 0 || tr.n_calls >= (1 << 24) || tr.n_queries > tr.n_calls;
}

// *long_call: whether an attempt may take kLongCall us or more on some type.
int validate_trace(const hx_trace* tr, int ti, const hx_cluster* c, int64_t min_prefill, int64_t max_decode,
                   bool* long_call) {
  // fault windows stretch attempts (slow-down or timeout) and delay the rest
  int64_t stretch = HX_SCALE;
  for (int f = 0; f < c->n_faults; ++f)
    stretch = std::max(stretch, std::max<int64_t>(c->faults[f].slow_fp, c->timeout_mult_fp));
  const int64_t long_cost = (hx::kLongCall - 1) * HX_SCALE / stretch + 1;  // stretched, kLongCall or more
  const std::string where = "trace " + std::to_string(ti) + ": ";
  if (bad_counts(*tr)) return fail(HX_ERR_INVALID, where + "n_queries/n_calls out of range");
  if (tr->n_queries > 0 && (!tr->arrival_us || !tr->k || !tr->prompt || !tr->out || !tr->out_est || !tr->stage ||
                            !tr->cand || !tr->retry))
    return fail(HX_ERR_INVALID, where + "array is NULL");
  if (!tr->call_base) return fail(HX_ERR_INVALID, where + "call_base is NULL");
  if (tr->call_base[0] != 0 || tr->call_base[tr->n_queries] != tr->n_calls)
    return fail(HX_ERR_INVALID, where + "call_base must run from 0 to n_calls");
  // the time horizon: the last arrival plus every call's cost bound
  // ceil(prompt * 10^6 / min_prefill) + max(out, out_est) * max_decode;
  // summed here as sum(prompt) and sum(decode part), the sum of the ceilings
  // lying within n_calls above the ceiling of the sum
  int64_t tok_sum = 0, dec_sum = 0, most = 0;
  for (int32_t i = 0; i < tr->n_queries; ++i) {
    if (tr->arrival_us[i] < 0 || (i > 0 && tr->arrival_us[i] < tr->arrival_us[i - 1]))
      return fail(HX_ERR_INVALID, where + "arrivals must be non-negative and sorted");
    const int32_t b = tr->call_base[i], e = tr->call_base[i + 1];
    const int k = tr->k[i];
    if (tr->tenant && tr->tenant[i] >= std::max(c->n_tenants, 1))
      return fail(HX_ERR_INVALID, where + "tenant out of range");
    if (k == 0) {
      // a single-shot request: one evaluation-stage call
      if (e - b != 1 || b < 0 || e > tr->n_calls || tr->stage[b] != HX_STAGE_E)
        return fail(HX_ERR_INVALID, where + "a k = 0 query must be a single E call");
    } else {
      if (k > HX_MAX_K) return fail(HX_ERR_INVALID, where + "k must be 0..8");
      if (e - b < 2 + k || b < 0 || e > tr->n_calls) return fail(HX_ERR_INVALID, where + "bad call_base");
      if (tr->stage[b] != HX_STAGE_S || tr->stage[e - 1] != HX_STAGE_E)
        return fail(HX_ERR_INVALID, where + "a query must start with S and end with E");
      for (int cd = 0; cd < k; ++cd)
        if (tr->stage[b + 1 + cd] != HX_STAGE_G || tr->cand[b + 1 + cd] != cd)
          return fail(HX_ERR_INVALID, where + "S must be followed by G_0..G_{k-1}");
      int prev_c = -1, prev_r = 0;
      for (int32_t j = b + 1 + k; j < e - 1; ++j) {
        const int cd = tr->cand[j], r = tr->retry[j];
        if (tr->stage[j] != HX_STAGE_C || cd >= k || r < 1 || r > c->rmax)
          return fail(HX_ERR_INVALID, where + "corrections must be C calls of a candidate with 1 <= retry <= rmax");
        if (cd == prev_c ? r != prev_r + 1 : (cd < prev_c || r != 1))
          return fail(HX_ERR_INVALID, where + "corrections must be ordered by (candidate, retry)");
        prev_c = cd;
        prev_r = r;
      }
    }
    for (int32_t j = b; j < e; ++j) {
      const int64_t p = tr->prompt[j], o = tr->out[j], oe = tr->out_est[j];
      if (p < 1 || p > kTokMax || o < 0 || o > kTokMax || oe < 0 || oe > kTokMax)
        return fail(HX_ERR_INVALID, where + "token counts out of range");
      // ceil(p * 10^6 / min_prefill) + dec >= 2^28, decided without a division:
      // ceil(x / d) + y >= m exactly when x + y * d > (m - 1) * d (below 2^60 here);
      // whether the longest call is a long one, likewise, once for the trace (per call
      // it was a tenth of the time that a trace of 756k calls takes to upload)
      const int64_t dec = std::max(o, oe) * max_decode, scaled = p * 1000000 + dec * min_prefill;
      if (dec >= kCostMax || scaled > (kCostMax - 1) * min_prefill)
        return fail(HX_ERR_INVALID, where + "a call's cost exceeds 2^28 us");
      most = std::max(most, scaled);
      tok_sum += p;
      dec_sum += dec;
    }
  }
  *long_call = most > (long_cost - 1) * min_prefill;
  int64_t last = tr->n_queries > 0 ? tr->arrival_us[tr->n_queries - 1] : 0;
  for (int f = 0; f < c->n_faults; ++f) last = std::max(last, c->faults[f].t1_us);
  const int64_t widen = 1 + (stretch + HX_SCALE - 1) / HX_SCALE, halve = c->n_faults > 0 ? 1 : 2;
  const __int128 tok_us = (__int128)tok_sum * 1000000;
  const int64_t lower = (int64_t)((tok_us + min_prefill - 1) / min_prefill) + dec_sum;
  const int64_t upper = lower + tr->n_calls;
  if (upper <= kHorizonMax && upper * widen / halve + last <= kHorizonMax) return HX_OK;
  // near the limit: the exact sum of the per-call bounds decides
  int64_t horizon = 0;
  for (int32_t j = 0; j < tr->n_calls; ++j)
    horizon += (tr->prompt[j] * int64_t(1000000) + min_prefill - 1) / min_prefill +
               std::max<int64_t>(tr->out[j], tr->out_est[j]) * max_decode;
  if (horizon > kHorizonMax) return fail(HX_ERR_INVALID, where + "time horizon exceeds 2^39 us");
  horizon = horizon * widen / halve + last;
  if (horizon > kHorizonMax) return fail(HX_ERR_INVALID, where + "time horizon exceeds 2^39 us");
  return HX_OK;
}

// Host threads that work on so many traces and calls: up to 16, when the calls pay
// for them.
int host_threads(int32_t n_traces, int64_t calls) {
  const int64_t hw = std::max<int64_t>(1, std::thread::hardware_concurrency());
  return (int)std::min<int64_t>({16, hw, (int64_t)n_traces, calls / 200000 + 1});
}

// Whether to stage the per-call arrays of so many traces: up to 64 MiB of inputs,
// and 1.25 MiB a trace for every thread that stages them.  A thread stages about 19
// GB/s and a trace's own six copies cost about 66 us, their bytes next to nothing:
// an upload of one trace of 45k calls takes 0.24 ms staged, 0.27 not; one of 151k
// 0.05 ms longer staged, one of 756k 0.35 ms (of 2.7); four of 151k (four threads)
// 0.1 ms less (of 0.9), 64 of 23k 2.4 ms instead of 4.9.
constexpr int64_t kStageMost = int64_t(64) << 20, kStagePerThread = int64_t(1280) << 10;
bool stage_calls_of(int32_t n_traces, int64_t calls, int64_t input_bytes, int64_t call_bytes) {
  return input_bytes <= kStageMost && call_bytes <= kStagePerThread * n_traces * host_threads(n_traces, calls);
}

// fn(t) for t = 0 .. n_traces - 1 on host_threads(), one trace at a time each.
template <class F>
void for_each_trace(const hx_trace* traces, int32_t n_traces, F fn) {
  int64_t calls = 0;
  for (int32_t t = 0; t < n_traces; ++t) calls += traces[t].n_calls;
  const int nt = host_threads(n_traces, calls);
  if (nt <= 1) {
    for (int32_t t = 0; t < n_traces; ++t) fn(t);
    return;
  }
  std::atomic<int32_t> next{0};
  std::mutex m;
  std::exception_ptr first;  // the first exception a worker met, thrown again below
  auto work = [&]() {
    try {
      for (int32_t t; (t = next.fetch_add(1)) < n_traces;) fn(t);
    } catch (...) {
      std::lock_guard<std::mutex> lock(m);
      if (!first) first = std::current_exception();
      next = n_traces;  // the others stop at their next trace
    }
  };
  std::vector<std::thread> pool;
  pool.reserve((size_t)nt - 1);  // any allocation failure comes before a thread starts
  for (int i = 1; i < nt; ++i) {
    try {
      pool.emplace_back(work);
    } catch (const std::system_error&) {
      break;  // fewer threads than asked for: those started and this one share the traces
    }
  }
  work();
  for (std::thread& th : pool) th.join();
  if (first) std::rethrow_exception(first);
}

// validate_trace over every trace, in parallel, and then pack(t); the
// lowest-numbered failing trace's status and message are reported, as a loop in
// order would.
template <class F>
int validate_traces(const hx_trace* traces, int32_t n_traces, const hx_cluster* c, int64_t min_prefill,
                    int64_t max_decode, bool* long_calls, F pack) {
  std::vector<int> rc((size_t)n_traces, HX_OK);
  std::atomic<bool> any_long{false};
  std::vector<std::string> msg((size_t)n_traces);
  for_each_trace(traces, n_traces, [&](int32_t t) {
    bool is_long = false;
    rc[t] = validate_trace(&traces[t], t, c, min_prefill, max_decode, &is_long);
    if (is_long) any_long = true;
    if (rc[t] != HX_OK) msg[t] = g_err;  // this thread's message
    else pack(t);
  });
  for (int32_t t = 0; t < n_traces; ++t)
    if (rc[t] != HX_OK) return fail(rc[t], msg[t]);
  *long_calls = any_long;
  return HX_OK;
}

template <class T>
int upload(T* dst, const T* src, int64_t count, cudaStream_t s) {
  if (count <= 0) return HX_OK;
  HX_CUDA(cudaMemcpyAsync(dst, src, (size_t)count * sizeof(T), cudaMemcpyHostToDevice, s));
  return HX_OK;
}

// A validated trace's part of the staged inputs.
void pack_trace(hx_sim* h, const hx_trace& tr, int32_t t) {
  const int64_t qo = h->q_off[t], co = h->c_off[t], nq = tr.n_queries, nc = tr.n_calls;
  int64_t* const qcall = h->staged(h->d_qcall) + qo;
  for (int64_t i = 0; i < nq; ++i) qcall[i] = co + tr.call_base[i];
  if (t == h->n_traces - 1) qcall[nq] = h->n_c;
  if (nq > 0) {
    std::memcpy(h->staged(h->d_arrival) + qo, tr.arrival_us, (size_t)nq * sizeof(int64_t));
    std::memcpy(h->staged(h->d_k) + qo, tr.k, (size_t)nq);
    if (tr.tenant) std::memcpy(h->staged(h->d_tenant) + qo, tr.tenant, (size_t)nq);
    else std::memset(h->staged(h->d_tenant) + qo, 0, (size_t)nq);
  }
  if (h->d_tenant_kcap) {
    // top-K size of each tenant for its P95: n_t - ceil(0.95 n_t) + 1 over its n_t
    // queries (0 without queries); at most the trace's own K
    int32_t n[HX_MAX_TENANTS] = {0, 0, 0, 0};
    for (int64_t i = 0; i < nq; ++i) n[tr.tenant ? tr.tenant[i] : 0]++;
    int32_t* const kcap = h->staged(h->d_tenant_kcap) + (int64_t)t * HX_MAX_TENANTS;
    for (int u = 0; u < HX_MAX_TENANTS; ++u) kcap[u] = n[u] ? n[u] - (95 * n[u] + 99) / 100 + 1 : 0;
  }
  if (h->stage_calls && nc > 0) {
    std::memcpy(h->staged(h->d_prompt) + co, tr.prompt, (size_t)nc * sizeof(int32_t));
    std::memcpy(h->staged(h->d_out) + co, tr.out, (size_t)nc * sizeof(int32_t));
    std::memcpy(h->staged(h->d_out_est) + co, tr.out_est, (size_t)nc * sizeof(int32_t));
    std::memcpy(h->staged(h->d_stage) + co, tr.stage, (size_t)nc);
    std::memcpy(h->staged(h->d_cand) + co, tr.cand, (size_t)nc);
    std::memcpy(h->staged(h->d_retry) + co, tr.retry, (size_t)nc);
  }
}

// Copies the first `bytes` of the staged inputs to the device, and the per-call
// arrays that are not staged.
int upload_inputs(hx_sim* h, const hx_trace* traces, int64_t bytes, cudaStream_t s) {
  int rc;
  if ((rc = upload(h->block, h->stage.get(), bytes, s))) return rc;
  for (int t = 0; t < h->n_traces && !h->stage_calls; ++t) {
    const hx_trace& tr = traces[t];
    const int64_t co = h->c_off[t];
    if ((rc = upload(h->d_prompt + co, tr.prompt, tr.n_calls, s)) || (rc = upload(h->d_out + co, tr.out, tr.n_calls, s)) ||
        (rc = upload(h->d_out_est + co, tr.out_est, tr.n_calls, s)) ||
        (rc = upload(h->d_stage + co, tr.stage, tr.n_calls, s)) || (rc = upload(h->d_cand + co, tr.cand, tr.n_calls, s)) ||
        (rc = upload(h->d_retry + co, tr.retry, tr.n_calls, s)))
      return rc;
  }
  HX_CUDA(cudaStreamSynchronize(s));
  if (!h->stage_calls) h->stage.reset();
  return HX_OK;
}

// WarpShared and the instance states and slot entries that follow it.
int per_warp_smem(const hx::ClusterK& ck, int family, int slot_entries) {
  const int64_t slot = family == hx::kSimWide ? sizeof(hx::Slot64) : sizeof(hx::Slot32);
  return (int)align_up((int64_t)sizeof(hx::WarpShared) + (ck.n_inst <= 32 ? 32 : 64) * (int64_t)sizeof(hx::InstState) +
                       slot * slot_entries, 16);
}

// The launch of a kernel family for a cluster, of up to `want` blocks: the kernel
// and the blocks that are resident at once.
int launch_shape(int family, const hx::ClusterK& ck, const cudaDeviceProp& prop, int64_t want, hx_sim::Launch* out) {
  want = std::max<int64_t>(want, 1);
  out->family = family;
  const bool few = few_warps(want * hx::kWarpsPerBlock, prop.multiProcessorCount);
  out->kernel = sim_kernel_of(family, ck, few);
  out->slot_entries = ck.n_inst <= 32 && hx::spaced_slots(1, family == hx::kSimWide, few) ? 16 * 32 : ck.slot_entries;
  out->smem_per_block = hx::kWarpsPerBlock * per_warp_smem(ck, family, out->slot_entries);
  if (int rc = ensure_dyn_smem(out->kernel, out->smem_per_block)) return rc;
  int bps = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, (const void*)hx::kSimKernel[out->kernel],
                                                    hx::kWarpsPerBlock * 32, out->smem_per_block) != cudaSuccess ||
      bps < 1) {
    cudaGetLastError();
    return fail(HX_ERR_CUDA, "simulation kernel does not fit on an SM");
  }
  out->blocks = (int)std::min<int64_t>(want, (int64_t)bps * prop.multiProcessorCount);
  return HX_OK;
}

// Whether s is being captured (if that cannot be told, the launches say so).
bool capturing(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return cap != cudaStreamCaptureStatusNone;
}

// Gives the simulation kernel that follows all of the work, or none of it.
__global__ void hx_gate_kernel(const int32_t* long_calls, int32_t want, unsigned long long n_work,
                               unsigned long long* work_counter) {
  *work_counter = (*long_calls != 0) == (want != 0) ? 0ull : n_work;
}

int launch_sim(const hx_sim::Launch& l, const hx::SimArgs& sa, hx::ClusterK ck, cudaStream_t s) {
  ck.smem_per_warp = l.smem_per_block / hx::kWarpsPerBlock;
  ck.slot_entries = l.slot_entries;
  if (int rc = ensure_dyn_smem(l.kernel, l.smem_per_block)) return rc;
  hx::kSimKernel[l.kernel]<<<(unsigned)l.blocks, hx::kWarpsPerBlock * 32, l.smem_per_block, s>>>(sa, ck);
  HX_CUDA(cudaGetLastError());
  return HX_OK;
}

// Kernel-parameter copy of a validated cluster.
void fill_cluster(const hx_cluster* cluster, hx::ClusterK& ck) {
  ck = hx::ClusterK{};
  ck.n_inst = cluster->n_inst;
  ck.n_types = cluster->n_types;
  ck.ref_type = cluster->ref_type;
  ck.rmax = cluster->rmax;
  ck.slo_mult_fp = cluster->slo_mult_fp;
  for (int t = 0; t < HX_MAX_TYPES; ++t) {
    const bool on = t < cluster->n_types;
    ck.prefill[t] = on ? cluster->prefill_tok_s[t] : 1;
    ck.decode[t] = on ? cluster->decode_us_tok[t] : 0;
    ck.slots[t] = on ? cluster->slots[t] : 0;
    ck.cnt[t] = 0;
  }
  for (int s = 0; s < 4; ++s) {
    ck.ref_prompt[s] = cluster->stage_ref_prompt[s];
    ck.ref_out[s] = cluster->stage_ref_out[s];
  }
  int base = 0;
  for (int m = 0; m < HX_MAX_INST; ++m) {
    const bool on = m < cluster->n_inst;
    const int ty = on ? cluster->inst_type[m] : 0;
    ck.inst_type[m] = (uint8_t)ty;
    ck.inst_slots[m] = on ? (uint8_t)cluster->slots[ty] : 0;
    ck.slot_base[m] = (uint16_t)base;
    if (on) {
      base += cluster->slots[ty];
      ck.cnt[ty]++;
    }
  }
  ck.slot_entries = base + 16;
  // per-tenant SLO multipliers replace slo_mult_fp when given
  ck.n_tenants = std::max(cluster->n_tenants, 1);
  for (int t = 0; t < HX_MAX_TENANTS; ++t)
    ck.tenant_mult[t] = (cluster->tenant_slo_mult_fp && t < ck.n_tenants) ? cluster->tenant_slo_mult_fp[t]
                                                                          : cluster->slo_mult_fp;
  ck.timeout_mult_fp = cluster->timeout_mult_fp;
  ck.n_faults = cluster->n_faults;
  for (int f = 0; f < cluster->n_faults; ++f) {
    const hx_fault& F = cluster->faults[f];
    ck.faults[f].t0 = F.t0_us;
    ck.faults[f].t1 = F.t1_us;
    ck.faults[f].slow = F.slow_fp;
    ck.faults[f].inst = F.inst;
    ck.faults[f].pad = 0;
  }
  ck.smem_per_warp = 0;  // by kernel family, at launch
}

// The simulations of opt->sim_subset, checked (in range, distinct) and sorted
// into the kernel's work order: trace-major, highest point first.
int order_subset(const hx_options* opt, int32_t n_traces, int32_t n_points, std::vector<int64_t>* out) {
  out->clear();
  if (!opt || opt->n_subset == 0) return HX_OK;
  if (opt->n_subset < 0) return fail(HX_ERR_INVALID, "n_subset < 0");
  if (!opt->sim_subset) return fail(HX_ERR_INVALID, "sim_subset is NULL");
  const int64_t n_sims = (int64_t)n_traces * n_points;
  std::vector<int64_t> w((size_t)opt->n_subset);
  for (int32_t i = 0; i < opt->n_subset; ++i) {
    const int64_t s = opt->sim_subset[i];
    if (s < 0 || s >= n_sims)
      return fail(HX_ERR_INVALID, "sim_subset[" + std::to_string(i) + "] = " + std::to_string(s) + " is out of range");
    const int64_t t = s / n_points, p = s - t * n_points;
    w[i] = t * n_points + (n_points - 1 - p);
  }
  std::sort(w.begin(), w.end());
  for (size_t i = 1; i < w.size(); ++i)
    if (w[i] == w[i - 1]) return fail(HX_ERR_INVALID, "sim_subset lists a simulation twice");
  out->resize(w.size());
  for (size_t i = 0; i < w.size(); ++i) {
    const int64_t t = w[i] / n_points;
    (*out)[i] = t * n_points + (n_points - 1 - (w[i] - t * n_points));
  }
  return HX_OK;
}

// Work order for a whole grid when it pays to change the default one.  The
// kernel takes simulations trace-major (the warps on one trace share its
// records in L2), highest point first within a trace.  A simulation whose
// points dispatch workload-balanced at alpha = 1 sends every request to the
// fastest instance and builds the longest local queue, so it costs more per
// event than any other point, and trace-major order starts the last traces'
// such simulations in the last wave, where they set the end of the run.  If
// the run is at most four waves of warps deep and every trace's records fit
// in L2 together, all traces' alpha = 1 points go first (hx_info.work_order
// 2); otherwise the traces of about the last two waves take theirs first,
// the others staying trace-major (3).  *order is left empty, and 0 returned,
// when the default stands.  Results do not depend on the order.
int costliest_first(const hx_grid* grid, int32_t n_traces, int64_t n_calls, int64_t l2_bytes,
                    int64_t resident_warps, std::vector<int64_t>* order) {
  order->clear();
  const int32_t P = grid->n_points;
  const int64_t n_sims = (int64_t)n_traces * P;
  // a list longer than 2^24 entries (128 MiB) is not worth its device memory
  if (n_sims <= resident_warps || n_sims > (int64_t(1) << 24)) return 0;
  std::vector<int32_t> hot, cold;
  for (int32_t p = P - 1; p >= 0; --p)
    (grid->alpha_fp[p] == hx::kScale && grid->dispatch_policy[p] == HX_DISPATCH_WB ? hot : cold).push_back(p);
  if (hot.empty() || cold.empty()) return 0;
  int32_t t0 = 0;  // traces before t0 keep the default order
  if (n_sims > 4 * resident_warps || n_calls * (int64_t)sizeof(hx::CallRec) > l2_bytes) {
    const int64_t k = (2 * resident_warps + P - 1) / P;
    if (k >= n_traces) return 0;
    t0 = n_traces - (int32_t)k;
  }
  order->reserve((size_t)n_sims);
  for (int32_t t = 0; t < t0; ++t)
    for (int32_t p = P - 1; p >= 0; --p) order->push_back((int64_t)t * P + p);
  for (const std::vector<int32_t>* part : {&hot, &cold})
    for (int32_t t = t0; t < n_traces; ++t)
      for (int32_t p : *part) order->push_back((int64_t)t * P + p);
  return t0 == 0 ? 2 : 3;
}

}  // namespace

extern "C" {

const char* hx_last_error(void) { return g_err.c_str(); }

static int hx_sim_create_impl(const hx_trace* traces, int32_t n_traces, const hx_cluster* cluster, const hx_grid* grid,
                              const hx_options* opt, hx_sim** out) {
  NvtxRange range("hx_sim_create");
  if (!out) return fail(HX_ERR_INVALID, "out is NULL");
  *out = nullptr;
  g_err.clear();
  if (!traces || n_traces < 1) return fail(HX_ERR_INVALID, "need at least one trace");
  int64_t min_prefill = 0, max_decode = 0;
  int rc;
  if ((rc = validate_cluster(cluster, &min_prefill, &max_decode))) return rc;
  if ((rc = validate_grid(grid))) return rc;
  auto validate = [&](bool* long_calls, auto pack) {
    return validate_traces(traces, n_traces, cluster, min_prefill, max_decode, long_calls, pack);
  };
  int64_t n_calls = 0;
  bool refuse = false, long_calls = false;
  for (int32_t i = 0; i < n_traces; ++i) {
    refuse |= bad_counts(traces[i]);
    n_calls += traces[i].n_calls;
  }
  if (refuse || n_calls >= (int64_t(1) << 31)) {
    if ((rc = validate(&long_calls, [](int32_t) {}))) return rc;
    return fail(HX_ERR_INVALID, "more than 2^31 calls in total");
  }
  // the handle is freed on every early return (and exception) until it is handed out
  std::unique_ptr<hx_sim> owner(new (std::nothrow) hx_sim());
  hx_sim* h = owner.get();
  if (!h) return fail(HX_ERR_OOM, "host allocation failed");
  auto bail = [](int code) { return code; };
  h->n_traces = n_traces;
  h->n_points = grid->n_points;
  h->n_sims = (int64_t)n_traces * grid->n_points;
  std::vector<int64_t>&q_off = h->q_off, &c_off = h->c_off;
  q_off.assign((size_t)n_traces + 1, 0);
  c_off.assign((size_t)n_traces + 1, 0);
  for (int t = 0; t < n_traces; ++t) {
    const int32_t nq = traces[t].n_queries, nc = traces[t].n_calls;
    h->h_nq.push_back(nq);
    h->h_nc.push_back(nc);
    q_off[t + 1] = q_off[t] + nq;
    c_off[t + 1] = c_off[t] + nc;
    h->max_nq = std::max(h->max_nq, nq);
    h->max_nc = std::max(h->max_nc, nc);
    h->max_kcap = std::max(h->max_kcap, nq - (95 * nq + 99) / 100 + 1);
  }
  h->n_q = q_off[n_traces];
  h->n_c = c_off[n_traces];
  // cluster constants (kernel parameter)
  hx::ClusterK& ck = h->ck;
  fill_cluster(cluster, ck);
  h->n_tenants = cluster->n_tenants;
  h->faults.assign(cluster->faults, cluster->faults + cluster->n_faults);

  // the inputs: per-query arrays and constants, then the per-call arrays
  const bool tenants = ck.n_tenants > 1;
  h->place(&h->d_arrival, h->n_q);
  h->place(&h->d_qcall, h->n_q + 1);
  h->place(&h->d_k, h->n_q);
  h->place(&h->d_tenant, h->n_q);
  if (tenants) h->place(&h->d_tenant_kcap, (int64_t)n_traces * HX_MAX_TENANTS);
  h->place(&h->d_long, 1);
  h->query_bytes = h->device_bytes;
  h->place(&h->d_q_off, n_traces + 1);
  h->place(&h->d_c_off, n_traces + 1);
  h->place(&h->d_alpha, h->n_points);
  h->place(&h->d_gamma, h->n_points);
  h->place(&h->d_beta, h->n_points);
  h->place(&h->d_rho, h->n_points);
  h->place(&h->d_lp, h->n_points);
  h->place(&h->d_dp, h->n_points);
  h->const_bytes = h->device_bytes;
  h->place(&h->d_prompt, h->n_c);
  h->place(&h->d_out, h->n_c);
  h->place(&h->d_out_est, h->n_c);
  h->place(&h->d_stage, h->n_c);
  h->place(&h->d_cand, h->n_c);
  h->place(&h->d_retry, h->n_c);
  h->input_bytes = h->device_bytes;
  h->stage_calls = stage_calls_of(n_traces, h->n_c, h->input_bytes, h->input_bytes - h->const_bytes);
  const int64_t staged_bytes = h->stage_calls ? h->input_bytes : h->const_bytes;
  h->stage.reset(new unsigned char[(size_t)staged_bytes]);
  // staged() needs the offsets only: the block is allocated when its size is known
  for (const auto& p : h->placed) *p.first = h->block + p.second;
  if ((rc = validate(&long_calls, [&](int32_t i) { pack_trace(h, traces[i], i); }))) return bail(rc);
  *h->staged(h->d_long) = long_calls;
  if (opt && opt->n_record < 0) return bail(fail(HX_ERR_INVALID, "n_record < 0"));
  if (opt && opt->n_record > 0) {
    if (!opt->record_sims) return bail(fail(HX_ERR_INVALID, "record_sims is NULL"));
    std::vector<int32_t> sorted(opt->record_sims, opt->record_sims + opt->n_record);
    std::sort(sorted.begin(), sorted.end());
    const int64_t n_sims = (int64_t)n_traces * grid->n_points;
    for (size_t j = 0; j < sorted.size(); ++j)
      if (sorted[j] < 0 || sorted[j] >= n_sims || (j > 0 && sorted[j] == sorted[j - 1]))
        return bail(fail(HX_ERR_INVALID, "record_sims must be distinct valid sim indices"));
  }
  if (opt && opt->checked != 0 && opt->checked != 1) return bail(fail(HX_ERR_INVALID, "checked must be 0 or 1"));
  if (opt && opt->arena_entries < 0) return bail(fail(HX_ERR_INVALID, "arena_entries < 0"));
  std::vector<int64_t> subset;
  if ((rc = order_subset(opt, n_traces, grid->n_points, &subset))) return bail(rc);

  h->n_work = subset.empty() ? h->n_sims : (int64_t)subset.size();
  h->checked = opt && opt->checked == 1;
  std::copy(q_off.begin(), q_off.end(), h->staged(h->d_q_off));
  std::copy(c_off.begin(), c_off.end(), h->staged(h->d_c_off));
  std::copy_n(grid->alpha_fp, h->n_points, h->staged(h->d_alpha));
  std::copy_n(grid->gamma_fp, h->n_points, h->staged(h->d_gamma));
  std::copy_n(grid->beta_us2, h->n_points, h->staged(h->d_beta));
  std::copy_n(grid->rho, h->n_points, h->staged(h->d_rho));
  std::copy_n(grid->local_policy, h->n_points, h->staged(h->d_lp));
  std::copy_n(grid->dispatch_policy, h->n_points, h->staged(h->d_dp));
  int dev = 0;
  cudaDeviceProp prop;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess) {
    cudaGetLastError();
    return bail(fail(HX_ERR_CUDA, "no CUDA device"));
  }
  // derived and outputs
  h->place(&h->d_rec, h->n_c);
  h->place(&h->d_results, h->n_sims);
  h->place(&h->d_counter, 1);
  h->place(&h->d_best_trace, 2 * (int64_t)n_traces);
  h->place(&h->d_best_global, 2);
  h->place(&h->d_point_sums, 3 * (int64_t)h->n_points);

  // launch shapes of the simulation kernel, for the simulations that run; later
  // uploads may bring longer calls
  int64_t blocks = (h->n_work + hx::kWarpsPerBlock - 1) / hx::kWarpsPerBlock;
  if (opt && opt->max_resident_warps > 0)
    blocks = std::min<int64_t>(blocks, std::max<int64_t>(1, opt->max_resident_warps / hx::kWarpsPerBlock));
  const int family = sim_family(grid, ck, opt && opt->n_record > 0, opt && opt->force_generic, h->checked);
  if ((rc = launch_shape(family, ck, prop, blocks, &h->launch[0])) ||
      (rc = launch_shape(hx::kSimWide, ck, prop, blocks, &h->launch[1])))
    return bail(rc);
  h->long_calls = long_calls;
  const int64_t resident_warps = hx::kWarpsPerBlock * (int64_t)h->shape().blocks;
  // the simulations' order: the caller's subset, else possibly the costliest first
  h->work_order = subset.empty()
                      ? costliest_first(grid, n_traces, h->n_c, (int64_t)prop.l2CacheSize, resident_warps, &subset)
                      : 1;
  if (!subset.empty()) h->place(&h->d_subset, (int64_t)subset.size());
  // heap arena: doubling regions of 16, 32, ... entries per instance total at
  // most 4 * (requests ever queued) + 16 * instances
  h->arena_per_warp = 4 * (int64_t)h->max_nc + 16 * HX_MAX_INST;
  // (no more than a queue's offset can reach: a queue past it is HX_ERR_CAPACITY)
  if (opt && opt->arena_entries > 0)
    h->arena_per_warp = std::min<int64_t>(opt->arena_entries, int64_t(hx::kHeapOffMask) + 1);
  h->chains_per_warp = align_up(std::max(h->max_nq, 1), 256);
  h->topk_per_warp = align_up(h->max_kcap, 32);
  if (tenants) {
    // one more heap per tenant after the simulation's own, each sized for a
    // whole trace (a tenant's K never exceeds its trace's), so uploads of new
    // tenant assignments need no reallocation
    for (int t = 0; t < HX_MAX_TENANTS; ++t) h->tenant_topk_off[t] = h->topk_per_warp * (1 + t);
    h->topk_per_warp *= 1 + HX_MAX_TENANTS;
  }
  const int64_t w = hx::kWarpsPerBlock * (int64_t)std::max(h->launch[0].blocks, h->launch[1].blocks);
  h->place(&h->d_arena, w * h->arena_per_warp);
  h->place(&h->d_chains, w * h->chains_per_warp);
  h->place(&h->d_topk, w * h->topk_per_warp);
  if (family >= hx::kSimGeneric) h->place(&h->d_extras, h->n_sims);
  h->scratch_bytes = w * (h->arena_per_warp * (int64_t)sizeof(hx::HeapEnt) + h->chains_per_warp +
                          h->topk_per_warp * (int64_t)sizeof(int64_t));

  // per-call logs of selected simulations: enq, budget, start, end (int64) and inst
  // (int32) of one simulation side by side, so that they are read back in one copy
  std::vector<int32_t> map;
  if (opt && opt->n_record > 0) {
    h->n_record = opt->n_record;
    h->rec_calls = std::max(h->max_nc, 1);
    h->rec_stride = 4 * h->rec_calls + (h->rec_calls + 1) / 2;
    map.assign((size_t)h->n_sims, -1);
    for (int j = 0; j < opt->n_record; ++j) {
      const int32_t sim = opt->record_sims[j];  // checked above: distinct, in range
      map[sim] = j;
      h->record_sims.push_back(sim);
    }
    h->place(&h->d_rec_map, h->n_sims);
    h->place(&h->d_rec_sims, h->n_record);
    h->place(&h->d_rec_log, h->n_record * h->rec_stride);
  }
  if ((rc = h->commit())) return bail(rc);
  cudaStream_t s0 = nullptr;
  if ((rc = upload_inputs(h, traces, staged_bytes, s0)) || (rc = upload(h->d_subset, subset.data(), (int64_t)subset.size(), s0)) ||
      (rc = upload(h->d_rec_map, map.data(), (int64_t)map.size(), s0)) ||
      (rc = upload(h->d_rec_sims, h->record_sims.data(), h->n_record, s0)))
    return bail(rc);
  if (opt && opt->timing) {
    h->timing = true;
    h->ev.assign(4 * hx_sim::kTimedRuns, nullptr);
    for (auto& e : h->ev)
      if (cudaEventCreate(&e) != cudaSuccess) return bail(fail(HX_ERR_CUDA, "cudaEventCreate failed"));
  }
  if (cudaDeviceSynchronize() != cudaSuccess) return bail(fail(HX_ERR_CUDA, "upload failed"));
  *out = owner.release();
  return HX_OK;
}

static int hx_sim_upload_impl(hx_sim* h, const hx_trace* traces, int32_t n_traces, void* stream) {
  NvtxRange range("hx_sim_upload");
  if (!h || !traces) return fail(HX_ERR_INVALID, "NULL argument");
  if (n_traces != h->n_traces) return fail(HX_ERR_INVALID, "trace count differs from the handle's");
  for (int t = 0; t < n_traces; ++t)
    if (traces[t].n_queries != h->h_nq[t] || traces[t].n_calls != h->h_nc[t])
      return fail(HX_ERR_INVALID, "trace shapes differ from the handle's");
  // same validation as create, against the handle's cluster bounds
  int64_t min_prefill = INT64_MAX, max_decode = 0;
  for (int t = 0; t < h->ck.n_types; ++t) {
    min_prefill = std::min<int64_t>(min_prefill, h->ck.prefill[t]);
    max_decode = std::max<int64_t>(max_decode, h->ck.decode[t]);
  }
  hx_cluster c{};
  c.rmax = h->ck.rmax;
  c.n_inst = h->ck.n_inst;
  c.n_tenants = h->n_tenants;
  c.timeout_mult_fp = h->ck.timeout_mult_fp;
  c.n_faults = (int32_t)h->faults.size();
  c.faults = h->faults.data();
  bool long_calls = false;
  if (!h->stage) h->stage.reset(new unsigned char[(size_t)h->query_bytes]);
  int rc = validate_traces(traces, n_traces, &c, min_prefill, max_decode, &long_calls,
                           [&](int32_t t) { pack_trace(h, traces[t], t); });
  if (rc) return rc;
  // set first: a copy that fails half-way may leave long calls behind
  const bool had_long = h->long_calls;
  h->long_calls = had_long || long_calls;
  *h->staged(h->d_long) = long_calls;
  if ((rc = upload_inputs(h, traces, h->stage_calls ? h->input_bytes : h->query_bytes,
                          static_cast<cudaStream_t>(stream))))
    return rc;
  h->long_calls = long_calls;
  return HX_OK;
}

static int hx_sim_run_impl(hx_sim* h, void* stream) {
  NvtxRange range("hx_sim_run");
  if (!h) return fail(HX_ERR_INVALID, "handle is NULL");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  hx::PrepArgs pa;
  pa.arrival = h->d_arrival;
  pa.kq = h->d_k;
  pa.qcall = h->d_qcall;
  pa.q_off = h->d_q_off;
  pa.c_off = h->d_c_off;
  pa.prompt = h->d_prompt;
  pa.out = h->d_out;
  pa.out_est = h->d_out_est;
  pa.stage = h->d_stage;
  pa.cand = h->d_cand;
  pa.retry = h->d_retry;
  pa.tenant = h->d_tenant;
  pa.n_queries = h->n_q;
  pa.n_traces = h->n_traces;
  pa.rec = h->d_rec;
  pa.work_counter = h->d_counter;
  pa.skip_results = h->d_results;
  pa.skip_extras = h->d_extras;
  pa.n_skip = h->n_work < h->n_sims ? h->n_sims : 0;

  hx::SimArgs sa;
  sa.rec = h->d_rec;
  sa.arrival = h->d_arrival;
  sa.qcall = h->d_qcall;
  sa.q_off = h->d_q_off;
  sa.c_off = h->d_c_off;
  sa.alpha = h->d_alpha;
  sa.gamma = h->d_gamma;
  sa.rho = h->d_rho;
  sa.beta = h->d_beta;
  sa.lpol = h->d_lp;
  sa.dpol = h->d_dp;
  sa.n_points = h->n_points;
  sa.n_traces = h->n_traces;
  sa.n_sims = h->n_sims;
  sa.results = h->d_results;
  sa.work_counter = h->d_counter;
  sa.arena = h->d_arena;
  sa.arena_per_warp = h->arena_per_warp;
  sa.chains = h->d_chains;
  sa.chains_per_warp = h->chains_per_warp;
  sa.topk = h->d_topk;
  sa.topk_per_warp = h->topk_per_warp;
  sa.rec_map = h->d_rec_map;
  sa.rec_inst = reinterpret_cast<int32_t*>(h->d_rec_log + 4 * h->rec_calls);
  sa.rec_enq = h->d_rec_log;
  sa.rec_start = h->d_rec_log + 2 * h->rec_calls;
  sa.rec_end = h->d_rec_log + 3 * h->rec_calls;
  sa.rec_calls = h->rec_calls;
  sa.rec_stride = h->rec_stride;
  sa.extras = h->d_extras;
  sa.tenant_kcap = h->d_tenant_kcap;
  for (int t = 0; t < HX_MAX_TENANTS; ++t) sa.tenant_topk_off[t] = h->tenant_topk_off[t];
  sa.subset = h->d_subset;
  sa.n_work = h->n_work;
  sa.checked = h->checked ? 1 : 0;

  hx::BestArgs ba;
  ba.results = h->d_results;
  ba.q_off = h->d_q_off;
  ba.n_traces = h->n_traces;
  ba.n_points = h->n_points;
  ba.per_trace = h->d_best_trace;
  ba.global = h->d_best_global;
  ba.point_sums = h->d_point_sums;

  const int prep_blocks = (int)std::max<int64_t>(1, (h->n_q + 255) / 256);
  cudaEvent_t* ev = h->timing ? h->run_ev(h->runs) : nullptr;
  if (ev) HX_CUDA(cudaEventRecord(ev[0], s));
  hx::hx_prep_kernel<<<prep_blocks, 256, 0, s>>>(pa, h->ck);
  HX_CUDA(cudaGetLastError());
  if (ev) HX_CUDA(cudaEventRecord(ev[1], s));
  if (capturing(s)) {
    // traces uploaded before a replay may need the other family: both are
    // captured, and the one that does not serve them finds no work left
    for (int f = 0; f < 2; ++f) {
      hx_gate_kernel<<<1, 1, 0, s>>>(h->d_long, f, (unsigned long long)h->n_work, h->d_counter);
      HX_CUDA(cudaGetLastError());
      if (int rc = launch_sim(h->launch[f], sa, h->ck, s)) return rc;
    }
  } else if (int rc = launch_sim(h->shape(), sa, h->ck, s)) {
    return rc;
  }
  if (h->n_record > 0) {
    hx::LogArgs la;
    la.rec = h->d_rec;
    la.c_off = h->d_c_off;
    la.rho = h->d_rho;
    la.record_sims = h->d_rec_sims;
    la.n_record = h->n_record;
    la.n_points = h->n_points;
    la.rec_enq = h->d_rec_log;
    la.rec_budget = h->d_rec_log + h->rec_calls;
    la.rec_calls = h->rec_calls;
    la.rec_stride = h->rec_stride;
    const int64_t log_blocks = (h->rec_calls + 255) / 256 * h->n_record;
    hx::hx_log_kernel<<<(unsigned)std::min<int64_t>(log_blocks, 1 << 16), 256, 0, s>>>(la, h->ck);
    HX_CUDA(cudaGetLastError());
  }
  if (ev) HX_CUDA(cudaEventRecord(ev[2], s));
  hx::hx_best_kernel<<<h->n_traces + 1, 256, 0, s>>>(ba);
  HX_CUDA(cudaGetLastError());
  if (ev) HX_CUDA(cudaEventRecord(ev[3], s));
  h->last_stream = s;
  h->ran = true;
  h->runs++;
  return HX_OK;
}

static int hx_sim_results_impl(hx_sim* h, hx_result* host_out, size_t n) {
  NvtxRange range("hx_sim_results");
  if (!h || !host_out) return fail(HX_ERR_INVALID, "NULL argument");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  if ((int64_t)n > h->n_sims) return fail(HX_ERR_INVALID, "n exceeds the number of simulations");
  HX_CUDA(cudaStreamSynchronize(h->last_stream));
  HX_CUDA(cudaMemcpy(host_out, h->d_results, n * sizeof(hx_result), cudaMemcpyDeviceToHost));
  return HX_OK;
}

static int hx_sim_extras_impl(hx_sim* h, hx_extra* host_out, size_t n) {
  if (!h || !host_out) return fail(HX_ERR_INVALID, "NULL argument");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  if ((int64_t)n > h->n_sims) return fail(HX_ERR_INVALID, "n exceeds the number of simulations");
  HX_CUDA(cudaStreamSynchronize(h->last_stream));
  if (n == 0) return HX_OK;
  if (h->d_extras) {
    HX_CUDA(cudaMemcpy(host_out, h->d_extras, n * sizeof(hx_extra), cudaMemcpyDeviceToHost));
    return HX_OK;
  }
  // the lean and logging families serve one tenant without faults: everything is tenant 0
  std::vector<hx_result> res(n);
  HX_CUDA(cudaMemcpy(res.data(), h->d_results, n * sizeof(hx_result), cudaMemcpyDeviceToHost));
  for (size_t i = 0; i < n; ++i) {
    hx_extra e{};
    e.slo_met[0] = res[i].slo_met;
    e.n_done[0] = res[i].n_done;
    for (int t = 0; t < HX_MAX_TENANTS; ++t) e.p95_us[t] = res[i].status != HX_OK ? -1 : t == 0 ? res[i].p95_us : 0;
    host_out[i] = e;
  }
  return HX_OK;
}

static int hx_sim_best_impl(hx_sim* h, int32_t objective, hx_best* out) {
  if (!h || !out) return fail(HX_ERR_INVALID, "NULL argument");
  if (objective != HX_OBJ_P95 && objective != HX_OBJ_P95_SLO95) return fail(HX_ERR_INVALID, "unknown objective");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  HX_CUDA(cudaStreamSynchronize(h->last_stream));
  hx::BestCand g[2];
  HX_CUDA(cudaMemcpy(g, h->d_best_global, sizeof(g), cudaMemcpyDeviceToHost));
  const bool gv = g[objective].flags & 1;
  out->global_point = gv ? g[objective].p : -1;
  out->pad = 0;
  out->global_sum_p95 = gv ? g[objective].p95 : -1;
  out->global_slo_met = gv ? g[objective].slo : -1;
  if (out->per_trace_point) {
    std::vector<hx::BestCand> pt((size_t)2 * h->n_traces);
    HX_CUDA(cudaMemcpy(pt.data(), h->d_best_trace, pt.size() * sizeof(hx::BestCand), cudaMemcpyDeviceToHost));
    for (int t = 0; t < h->n_traces; ++t) {
      const hx::BestCand& b = pt[(size_t)2 * t + objective];
      out->per_trace_point[t] = (b.flags & 1) ? b.p : -1;
    }
  }
  return HX_OK;
}

static int hx_sim_point_sums_impl(hx_sim* h, int64_t* sum_p95, int64_t* sum_slo_met, int32_t* n_failed,
                                  size_t n_points) {
  if (!h || !sum_p95 || !sum_slo_met || !n_failed) return fail(HX_ERR_INVALID, "NULL argument");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  if ((int64_t)n_points != h->n_points) return fail(HX_ERR_INVALID, "n_points differs from the handle's");
  HX_CUDA(cudaStreamSynchronize(h->last_stream));
  std::vector<int64_t> v(3 * n_points);
  HX_CUDA(cudaMemcpy(v.data(), h->d_point_sums, v.size() * sizeof(int64_t), cudaMemcpyDeviceToHost));
  for (size_t p = 0; p < n_points; ++p) {
    sum_p95[p] = v[3 * p];
    sum_slo_met[p] = v[3 * p + 1];
    n_failed[p] = (int32_t)v[3 * p + 2];
  }
  return HX_OK;
}

static int hx_best_of_sums_impl(const int64_t* sum_p95, const int64_t* sum_slo_met, const int32_t* n_failed,
                                int32_t n_points, int64_t n_queries_total, int32_t objective, hx_best* out) {
  if (!sum_p95 || !sum_slo_met || !n_failed || !out) return fail(HX_ERR_INVALID, "NULL argument");
  if (n_points < 1 || n_queries_total < 0) return fail(HX_ERR_INVALID, "bad sizes");
  if (objective != HX_OBJ_P95 && objective != HX_OBJ_P95_SLO95) return fail(HX_ERR_INVALID, "unknown objective");
  // the summed table as one pseudo-trace, reduced by the same best-point kernel
  std::vector<hx_result> table((size_t)n_points);
  for (int32_t p = 0; p < n_points; ++p) {
    if (sum_slo_met[p] < 0 || sum_slo_met[p] > INT32_MAX) return fail(HX_ERR_INVALID, "SLO sums out of range");
    hx_result r{};
    r.p95_us = sum_p95[p];
    r.slo_met = (int32_t)sum_slo_met[p];
    r.status = n_failed[p] ? HX_ERR_CAPACITY : HX_OK;
    table[p] = r;
  }
  const int64_t qoff[2] = {0, n_queries_total};
  void* buf = nullptr;
  const size_t bytes = table.size() * sizeof(hx_result) + 2 * sizeof(int64_t) + 4 * sizeof(hx::BestCand);
  HX_CUDA(cudaMalloc(&buf, bytes));
  auto run = [&]() -> int {
    unsigned char* b = static_cast<unsigned char*>(buf);
    hx_result* d_res = reinterpret_cast<hx_result*>(b);
    int64_t* d_qoff = reinterpret_cast<int64_t*>(b + table.size() * sizeof(hx_result));
    hx::BestCand* d_cand = reinterpret_cast<hx::BestCand*>(d_qoff + 2);
    HX_CUDA(cudaMemcpy(d_res, table.data(), table.size() * sizeof(hx_result), cudaMemcpyHostToDevice));
    HX_CUDA(cudaMemcpy(d_qoff, qoff, sizeof(qoff), cudaMemcpyHostToDevice));
    hx::BestArgs ba;
    ba.results = d_res;
    ba.q_off = d_qoff;
    ba.n_traces = 1;
    ba.n_points = n_points;
    ba.per_trace = d_cand;
    ba.global = d_cand + 2;
    ba.point_sums = nullptr;
    hx::hx_best_kernel<<<2, 256>>>(ba);
    HX_CUDA(cudaGetLastError());
    hx::BestCand g[2];
    HX_CUDA(cudaMemcpy(g, d_cand + 2, sizeof(g), cudaMemcpyDeviceToHost));
    const bool v = g[objective].flags & 1;
    out->global_point = v ? g[objective].p : -1;
    out->pad = 0;
    out->global_sum_p95 = v ? g[objective].p95 : -1;
    out->global_slo_met = v ? g[objective].slo : -1;
    return HX_OK;
  };
  const int rc = run();
  cudaFree(buf);
  return rc;
}

static int hx_sim_records_impl(hx_sim* h, int32_t rec_index, int32_t* inst, int64_t* enq_us, int64_t* budget_us,
                               int64_t* start_us, int64_t* end_us, size_t n_calls) {
  if (!h) return fail(HX_ERR_INVALID, "handle is NULL");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  if (rec_index < 0 || rec_index >= h->n_record) return fail(HX_ERR_INVALID, "rec_index out of range");
  const int t = (int)(h->record_sims[rec_index] / h->n_points);
  if ((int64_t)n_calls != h->h_nc[t]) return fail(HX_ERR_INVALID, "n_calls differs from the trace's");
  HX_CUDA(cudaStreamSynchronize(h->last_stream));
  if (n_calls == 0) return HX_OK;
  // A short log is read in one copy; from a longer one each column asked for goes
  // straight to the caller: a copy's fixed cost is about 11 us, one through this
  // function's own buffer about 2.4 us per 1000 calls (all columns of 7.5k calls: 64
  // us by column, 44 in one; of 151k calls 89 and 410).
  const int64_t* const d = h->d_rec_log + (int64_t)rec_index * h->rec_stride;
  void* const cols[5] = {enq_us, budget_us, start_us, end_us, inst};
  const int n_cols = 5 - (int)std::count(cols, cols + 5, nullptr);
  std::unique_ptr<int64_t[]> log;
  if ((int64_t)n_calls <= 3000 * (int64_t)(n_cols - 1)) {
    log.reset(new int64_t[(size_t)h->rec_stride]);
    HX_CUDA(cudaMemcpy(log.get(), d, (size_t)h->rec_stride * sizeof(int64_t), cudaMemcpyDeviceToHost));
  }
  for (int i = 0; i < 5; ++i) {
    const size_t bytes = n_calls * (i < 4 ? sizeof(int64_t) : sizeof(int32_t));
    if (!cols[i]) continue;
    if (log) std::memcpy(cols[i], log.get() + i * h->rec_calls, bytes);
    else HX_CUDA(cudaMemcpy(cols[i], d + i * h->rec_calls, bytes, cudaMemcpyDeviceToHost));
  }
  return HX_OK;
}

static int hx_sim_prep_impl(hx_sim* h, int32_t trace_index, int32_t* est, int32_t* svc, int32_t* tbar,
                            int64_t* deadline_us, size_t n_calls) {
  if (!h) return fail(HX_ERR_INVALID, "handle is NULL");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  if (trace_index < 0 || trace_index >= h->n_traces) return fail(HX_ERR_INVALID, "trace_index out of range");
  if ((int64_t)n_calls != h->h_nc[trace_index]) return fail(HX_ERR_INVALID, "n_calls differs from the trace's");
  HX_CUDA(cudaStreamSynchronize(h->last_stream));
  if (n_calls == 0) return HX_OK;
  int64_t off = 0;
  for (int t = 0; t < trace_index; ++t) off += h->h_nc[t];
  std::vector<hx::CallRec> recs(n_calls);
  HX_CUDA(cudaMemcpy(recs.data(), h->d_rec + off, n_calls * sizeof(hx::CallRec), cudaMemcpyDeviceToHost));
  for (size_t j = 0; j < n_calls; ++j) {
    for (int ty = 0; ty < 4; ++ty) {
      if (est) est[4 * j + ty] = recs[j].ev[ty].x;
      if (svc) svc[4 * j + ty] = recs[j].ev[ty].y;
    }
    if (tbar) tbar[j] = recs[j].tbar;
    if (deadline_us) deadline_us[j] = recs[j].deadline;
  }
  return HX_OK;
}

int hx_sim_timings(hx_sim* h, float* prep_ms, float* sim_ms, float* best_ms) {
  return hx_sim_timings_back(h, 0, prep_ms, sim_ms, best_ms);
}

int hx_sim_timings_back(hx_sim* h, int32_t back, float* prep_ms, float* sim_ms, float* best_ms) {
  if (!h) return fail(HX_ERR_INVALID, "handle is NULL");
  if (!h->timing) return fail(HX_ERR_STATE, "created without opt.timing");
  if (!h->ran) return fail(HX_ERR_STATE, "hx_sim_run has not been called");
  if (back < 0 || back >= hx_sim::kTimedRuns || back >= h->runs)
    return fail(HX_ERR_INVALID, "back must be 0 .. min(runs, " + std::to_string(hx_sim::kTimedRuns) + ") - 1");
  cudaEvent_t* ev = h->run_ev(h->runs - 1 - back);
  HX_CUDA(cudaEventSynchronize(ev[3]));
  float a = 0, b = 0, c = 0;
  HX_CUDA(cudaEventElapsedTime(&a, ev[0], ev[1]));
  HX_CUDA(cudaEventElapsedTime(&b, ev[1], ev[2]));
  HX_CUDA(cudaEventElapsedTime(&c, ev[2], ev[3]));
  if (prep_ms) *prep_ms = a;
  if (sim_ms) *sim_ms = b;
  if (best_ms) *best_ms = c;
  return HX_OK;
}

int hx_selftest_div(const uint64_t* n, const uint64_t* d, uint64_t* q, uint64_t* q_ref, size_t count) {
  if (!n || !d || !q || !q_ref) return fail(HX_ERR_INVALID, "NULL argument");
  for (size_t i = 0; i < count; ++i)
    if (n[i] >= (uint64_t(1) << 63) || d[i] < 1 || d[i] >= (uint64_t(1) << 54))
      return fail(HX_ERR_INVALID, "operands must satisfy n < 2^63 and 1 <= d < 2^54");
  if (count == 0) return HX_OK;
  uint64_t* buf = nullptr;
  HX_CUDA(cudaMalloc(&buf, 4 * count * sizeof(uint64_t)));
  auto run = [&]() -> int {
    HX_CUDA(cudaMemcpy(buf, n, count * 8, cudaMemcpyHostToDevice));
    HX_CUDA(cudaMemcpy(buf + count, d, count * 8, cudaMemcpyHostToDevice));
    hx::hx_selftest_div_kernel<<<(unsigned)((count + 255) / 256), 256>>>(buf, buf + count, buf + 2 * count,
                                                                         buf + 3 * count, (int64_t)count);
    HX_CUDA(cudaGetLastError());
    HX_CUDA(cudaMemcpy(q, buf + 2 * count, count * 8, cudaMemcpyDeviceToHost));
    HX_CUDA(cudaMemcpy(q_ref, buf + 3 * count, count * 8, cudaMemcpyDeviceToHost));
    return HX_OK;
  };
  const int rc = run();
  cudaFree(buf);
  return rc;
}

int hx_sim_info(hx_sim* h, hx_info* out) {
  if (!h || !out) return fail(HX_ERR_INVALID, "NULL argument");
  out->n_sims = h->n_sims;
  out->n_calls_total = h->n_c;
  out->n_queries_total = h->n_q;
  out->scratch_bytes = h->scratch_bytes;
  out->device_bytes = h->device_bytes;
  out->resident_warps = hx::kWarpsPerBlock * h->shape().blocks;
  out->warps_per_block = hx::kWarpsPerBlock;
  out->blocks = h->shape().blocks;
  out->smem_per_block = h->shape().smem_per_block;
  out->generic_kernel = h->shape().family != hx::kSimLean ? 1 : 0;
  out->work_order = h->work_order;
  return HX_OK;
}

int hx_sim_destroy(hx_sim* h) {
  if (!h) return HX_OK;
  if (h->ran && h->last_stream) cudaStreamSynchronize(h->last_stream);
  cudaDeviceSynchronize();
  delete h;
  return HX_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// hx_sim_run_static: the whole path for one trace without allocating memory.
//
// For callers that may not allocate device memory -- code running where
// cudaMalloc is forbidden or unavailable (a host process that only owns
// pre-arranged memory, a plugin whose host application controls every
// allocation, a latency-critical loop that must not hit the allocator) -- this
// entry point runs the same preparation, simulation and best-point kernels as
// hx_sim_run, but every intermediate buffer (the copied inputs, the per-call
// records, the per-warp heap arenas, the results) is carved from one
// file-scope device array of HX_STATIC_SCRATCH_BYTES.  That array exists on
// every GPU that loads this library, for as long as the library stays loaded.
namespace {

__device__ __align__(256) unsigned char hx_static_scratch[HX_STATIC_SCRATCH_BYTES];

std::mutex g_static_mu;
unsigned char* g_static_base[kMaxDevices] = {};

// Device address of hx_static_scratch on the current device (the host-side
// symbol is only a stand-in and must never be passed to a kernel).  It is
// looked up again on every call made while `s` is not capturing, so a
// device reset between calls cannot leave a stale address behind; a call
// made during stream capture uses the address of the last earlier call on
// this device, and fails if there was none.
int static_base(cudaStream_t s, unsigned char** out) {
  int dev = 0;
  HX_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return fail(HX_ERR_INVALID, "device index out of range");
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  HX_CUDA(cudaStreamIsCapturing(s, &cap));
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (cap == cudaStreamCaptureStatusNone) {
    void* p = nullptr;
    HX_CUDA(cudaGetSymbolAddress(&p, hx_static_scratch));
    g_static_base[dev] = static_cast<unsigned char*>(p);
  } else if (!g_static_base[dev]) {
    return fail(HX_ERR_STATE, "the first hx_sim_run_static call on a device must come before any stream capture");
  }
  *out = g_static_base[dev];
  return HX_OK;
}

__global__ void hx_widen_kernel(const int32_t* src, int64_t* dst, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[i];
}

// Bump carving of the static array; offsets are 256-byte aligned.
struct Carve {
  int64_t used = 0;
  template <class T>
  int64_t take(int64_t count) {
    const int64_t off = used;
    used = align_up(used + std::max<int64_t>(count, 1) * (int64_t)sizeof(T), 256);
    return off;
  }
};

}  // namespace

static int hx_sim_run_static_impl(const hx_trace* trace, const hx_cluster* cluster, const hx_grid* grid,
                                  int32_t objective, hx_result* results, hx_best* best, void* stream) {
  g_err.clear();
  if (!trace || !results) return fail(HX_ERR_INVALID, "trace and results must not be NULL");
  if (objective != HX_OBJ_P95 && objective != HX_OBJ_P95_SLO95) return fail(HX_ERR_INVALID, "unknown objective");
  int64_t min_prefill = 0, max_decode = 0;
  int rc;
  if ((rc = validate_cluster(cluster, &min_prefill, &max_decode))) return rc;
  if ((rc = validate_grid(grid))) return rc;
  bool long_calls = false;
  if ((rc = validate_trace(trace, 0, cluster, min_prefill, max_decode, &long_calls))) return rc;
  const int64_t nq = trace->n_queries, nc = trace->n_calls, P = grid->n_points;
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  hx::ClusterK ck;
  fill_cluster(cluster, ck);

  // layout of the static array: inputs, records, results, then per-warp scratch
  Carve cv;
  const int64_t o_qoff = cv.take<int64_t>(2), o_coff = cv.take<int64_t>(2), o_ctr = cv.take<unsigned long long>(1);
  const int64_t o_arr = cv.take<int64_t>(nq), o_k = cv.take<uint8_t>(nq), o_cb32 = cv.take<int32_t>(nq + 1);
  const int64_t o_ten = cv.take<uint8_t>(nq);
  const int64_t o_qcall = cv.take<int64_t>(nq + 1);
  const int64_t o_prompt = cv.take<int32_t>(nc), o_out = cv.take<int32_t>(nc), o_oest = cv.take<int32_t>(nc);
  const int64_t o_stage = cv.take<uint8_t>(nc), o_cand = cv.take<uint8_t>(nc), o_retry = cv.take<uint8_t>(nc);
  const int64_t o_alpha = cv.take<int64_t>(P), o_gamma = cv.take<int64_t>(P), o_beta = cv.take<int64_t>(P);
  const int64_t o_rho = cv.take<int32_t>(P), o_lp = cv.take<uint8_t>(P), o_dp = cv.take<uint8_t>(P);
  const int64_t o_rec = cv.take<hx::CallRec>(nc), o_res = cv.take<hx_result>(P);
  const int64_t o_bt = cv.take<hx::BestCand>(2), o_bg = cv.take<hx::BestCand>(2);
  const int64_t fixed = cv.used;
  const int32_t kcap = (int32_t)(nq - (95 * nq + 99) / 100 + 1);
  const int64_t arena_per_warp = 4 * nc + 16 * HX_MAX_INST;
  const int64_t chains_per_warp = align_up(std::max<int64_t>(nq, 1), 256);
  const int64_t topk_per_warp = align_up(std::max<int32_t>(kcap, 1), 32);
  const int64_t per_warp = align_up(arena_per_warp * (int64_t)sizeof(hx::HeapEnt), 256) + chains_per_warp +
                           align_up(topk_per_warp * 8, 256);
  const int64_t room = (int64_t)HX_STATIC_SCRATCH_BYTES - fixed;
  const int64_t fit_warps = room > 0 ? room / per_warp : 0;
  if (fit_warps < hx::kWarpsPerBlock)
    return fail(HX_ERR_INVALID, "trace too large for the static scratch: it needs " +
                                    std::to_string(fixed + hx::kWarpsPerBlock * per_warp) + " bytes, the array holds " +
                                    std::to_string((int64_t)HX_STATIC_SCRATCH_BYTES));

  int dev = 0;
  cudaDeviceProp prop;
  HX_CUDA(cudaGetDevice(&dev));
  HX_CUDA(cudaGetDeviceProperties(&prop, dev));
  const int family = long_calls ? hx::kSimWide : sim_family(grid, ck, false, false, false);
  hx_sim::Launch launch;
  if ((rc = launch_shape(family, ck, prop, std::min<int64_t>(fit_warps / hx::kWarpsPerBlock, (P + hx::kWarpsPerBlock - 1) / hx::kWarpsPerBlock), &launch)))
    return rc;
  const int64_t blocks = launch.blocks;
  const int64_t warps = blocks * hx::kWarpsPerBlock;
  const int64_t o_arena = fixed;
  const int64_t o_chains = o_arena + warps * align_up(arena_per_warp * (int64_t)sizeof(hx::HeapEnt), 256);
  const int64_t o_topk = o_chains + warps * chains_per_warp;

  unsigned char* sb = nullptr;
  if ((rc = static_base(s, &sb))) return rc;
  auto at = [&](int64_t off) { return static_cast<void*>(sb + off); };
  const int64_t offs[4] = {0, nq, 0, nc};
  HX_CUDA(cudaMemcpyAsync(at(o_qoff), offs, 2 * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  HX_CUDA(cudaMemcpyAsync(at(o_coff), offs + 2, 2 * sizeof(int64_t), cudaMemcpyHostToDevice, s));
  struct Up {
    int64_t off;
    const void* src;
    int64_t bytes;
  } ups[] = {{o_arr, trace->arrival_us, nq * 8},     {o_k, trace->k, nq},
             {o_ten, trace->tenant, trace->tenant ? nq : 0},
             {o_cb32, trace->call_base, (nq + 1) * 4}, {o_prompt, trace->prompt, nc * 4},
             {o_out, trace->out, nc * 4},             {o_oest, trace->out_est, nc * 4},
             {o_stage, trace->stage, nc},             {o_cand, trace->cand, nc},
             {o_retry, trace->retry, nc},             {o_alpha, grid->alpha_fp, P * 8},
             {o_gamma, grid->gamma_fp, P * 8},        {o_beta, grid->beta_us2, P * 8},
             {o_rho, grid->rho, P * 4},               {o_lp, grid->local_policy, P},
             {o_dp, grid->dispatch_policy, P}};
  for (const Up& u : ups)
    if (u.bytes > 0) HX_CUDA(cudaMemcpyAsync(at(u.off), u.src, (size_t)u.bytes, cudaMemcpyHostToDevice, s));
  hx_widen_kernel<<<(unsigned)std::max<int64_t>(1, (nq + 1 + 255) / 256), 256, 0, s>>>(
      static_cast<const int32_t*>(at(o_cb32)), static_cast<int64_t*>(at(o_qcall)), nq + 1);
  HX_CUDA(cudaGetLastError());

  hx::PrepArgs pa;
  pa.arrival = static_cast<const int64_t*>(at(o_arr));
  pa.kq = static_cast<const uint8_t*>(at(o_k));
  pa.qcall = static_cast<const int64_t*>(at(o_qcall));
  pa.q_off = static_cast<const int64_t*>(at(o_qoff));
  pa.c_off = static_cast<const int64_t*>(at(o_coff));
  pa.prompt = static_cast<const int32_t*>(at(o_prompt));
  pa.out = static_cast<const int32_t*>(at(o_out));
  pa.out_est = static_cast<const int32_t*>(at(o_oest));
  pa.stage = static_cast<const uint8_t*>(at(o_stage));
  pa.cand = static_cast<const uint8_t*>(at(o_cand));
  pa.retry = static_cast<const uint8_t*>(at(o_retry));
  pa.tenant = trace->tenant ? static_cast<const uint8_t*>(at(o_ten)) : nullptr;
  pa.n_queries = nq;
  pa.n_traces = 1;
  pa.rec = static_cast<hx::CallRec*>(at(o_rec));
  pa.work_counter = static_cast<unsigned long long*>(at(o_ctr));  // zeroed by the prep kernel
  pa.skip_results = nullptr;
  pa.skip_extras = nullptr;
  pa.n_skip = 0;

  hx::SimArgs sa;
  sa.rec = pa.rec;
  sa.arrival = pa.arrival;
  sa.qcall = pa.qcall;
  sa.q_off = pa.q_off;
  sa.c_off = pa.c_off;
  sa.alpha = static_cast<const int64_t*>(at(o_alpha));
  sa.gamma = static_cast<const int64_t*>(at(o_gamma));
  sa.rho = static_cast<const int32_t*>(at(o_rho));
  sa.beta = static_cast<const int64_t*>(at(o_beta));
  sa.lpol = static_cast<const uint8_t*>(at(o_lp));
  sa.dpol = static_cast<const uint8_t*>(at(o_dp));
  sa.n_points = (int32_t)P;
  sa.n_traces = 1;
  sa.n_sims = P;
  sa.results = static_cast<hx_result*>(at(o_res));
  sa.work_counter = pa.work_counter;
  sa.arena = static_cast<hx::HeapEnt*>(at(o_arena));
  sa.arena_per_warp = align_up(arena_per_warp * (int64_t)sizeof(hx::HeapEnt), 256) / (int64_t)sizeof(hx::HeapEnt);
  sa.chains = static_cast<uint8_t*>(at(o_chains));
  sa.chains_per_warp = chains_per_warp;
  sa.topk = static_cast<int64_t*>(at(o_topk));
  sa.topk_per_warp = align_up(topk_per_warp * 8, 256) / 8;
  sa.rec_map = nullptr;
  sa.rec_inst = nullptr;
  sa.rec_enq = nullptr;
  sa.rec_start = nullptr;
  sa.rec_end = nullptr;
  sa.rec_calls = 0;
  sa.rec_stride = 0;
  sa.extras = nullptr;
  sa.tenant_kcap = nullptr;
  for (int t = 0; t < HX_MAX_TENANTS; ++t) sa.tenant_topk_off[t] = 0;
  sa.subset = nullptr;
  sa.n_work = P;
  sa.checked = 0;

  hx::BestArgs ba;
  ba.results = sa.results;
  ba.q_off = pa.q_off;
  ba.n_traces = 1;
  ba.n_points = (int32_t)P;
  ba.per_trace = static_cast<hx::BestCand*>(at(o_bt));
  ba.global = static_cast<hx::BestCand*>(at(o_bg));
  ba.point_sums = nullptr;

  hx::hx_prep_kernel<<<(unsigned)std::max<int64_t>(1, (nq + 255) / 256), 256, 0, s>>>(pa, ck);
  HX_CUDA(cudaGetLastError());
  if ((rc = launch_sim(launch, sa, ck, s))) return rc;
  hx::hx_best_kernel<<<2, 256, 0, s>>>(ba);
  HX_CUDA(cudaGetLastError());
  HX_CUDA(cudaMemcpyAsync(results, at(o_res), (size_t)P * sizeof(hx_result), cudaMemcpyDeviceToHost, s));
  hx::BestCand bg[2];
  HX_CUDA(cudaMemcpyAsync(bg, at(o_bg), sizeof(bg), cudaMemcpyDeviceToHost, s));
  HX_CUDA(cudaStreamSynchronize(s));
  if (best) {
    const bool v = bg[objective].flags & 1;
    best->global_point = v ? bg[objective].p : -1;
    best->pad = 0;
    best->global_sum_p95 = v ? bg[objective].p95 : -1;
    best->global_slo_met = v ? bg[objective].slo : -1;
    if (best->per_trace_point) best->per_trace_point[0] = best->global_point;
  }
  return HX_OK;
}

// The C entry points: each runs its implementation above under guarded(), so
// that no C++ exception crosses the ABI.
extern "C" {

int hx_sim_create(const hx_trace* traces, int32_t n_traces, const hx_cluster* cluster, const hx_grid* grid,
                  const hx_options* opt, hx_sim** out) {
  return guarded([&] { return hx_sim_create_impl(traces, n_traces, cluster, grid, opt, out); });
}

int hx_sim_upload(hx_sim* h, const hx_trace* traces, int32_t n_traces, void* stream) {
  return guarded([&] { return hx_sim_upload_impl(h, traces, n_traces, stream); });
}

int hx_sim_run(hx_sim* h, void* stream) {
  return guarded([&] { return hx_sim_run_impl(h, stream); });
}

int hx_sim_results(hx_sim* h, hx_result* host_out, size_t n) {
  return guarded([&] { return hx_sim_results_impl(h, host_out, n); });
}

int hx_sim_extras(hx_sim* h, hx_extra* host_out, size_t n) {
  return guarded([&] { return hx_sim_extras_impl(h, host_out, n); });
}

int hx_sim_best(hx_sim* h, int32_t objective, hx_best* out) {
  return guarded([&] { return hx_sim_best_impl(h, objective, out); });
}

int hx_sim_point_sums(hx_sim* h, int64_t* sum_p95, int64_t* sum_slo_met, int32_t* n_failed, size_t n_points) {
  return guarded([&] { return hx_sim_point_sums_impl(h, sum_p95, sum_slo_met, n_failed, n_points); });
}

int hx_best_of_sums(const int64_t* sum_p95, const int64_t* sum_slo_met, const int32_t* n_failed, int32_t n_points,
                    int64_t n_queries_total, int32_t objective, hx_best* out) {
  return guarded(
      [&] { return hx_best_of_sums_impl(sum_p95, sum_slo_met, n_failed, n_points, n_queries_total, objective, out); });
}

int hx_sim_records(hx_sim* h, int32_t rec_index, int32_t* inst, int64_t* enq_us, int64_t* budget_us,
                   int64_t* start_us, int64_t* end_us, size_t n_calls) {
  return guarded(
      [&] { return hx_sim_records_impl(h, rec_index, inst, enq_us, budget_us, start_us, end_us, n_calls); });
}

int hx_sim_prep(hx_sim* h, int32_t trace_index, int32_t* est, int32_t* svc, int32_t* tbar, int64_t* deadline_us,
                size_t n_calls) {
  return guarded([&] { return hx_sim_prep_impl(h, trace_index, est, svc, tbar, deadline_us, n_calls); });
}

int hx_sim_run_static(const hx_trace* trace, const hx_cluster* cluster, const hx_grid* grid,
                      int32_t objective, hx_result* results, hx_best* best, void* stream) {
  return guarded([&] { return hx_sim_run_static_impl(trace, cluster, grid, objective, results, best, stream); });
}

}  // extern "C"
