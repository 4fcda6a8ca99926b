// C ABI: plans, heads, slice contraction, amplitudes, sampling.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "buffers.h"
#include "handles.h"
#include "kernels.h"
#include "planner.h"
#include "tn_gb300.h"

namespace {

thread_local std::string g_err;

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

#define CUDA_TRY(x)                                                                          \
  do {                                                                                       \
    cudaError_t e_ = (x);                                                                    \
    if (e_ != cudaSuccess) return fail(TN_ERR_CUDA, std::string(#x) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// NVTX range around a scope: a profiler (nsys, or ncu with --nvtx) sees each
// pass and each step's launch by name; without a tool attached the calls do
// nothing.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

const char* step_range_name(int kind) {
  switch (kind) {
    case tn::ST_SMALL: return "tn small_operand";
    case tn::ST_PERMUTE: return "tn permute";
    case tn::ST_BPREP_TC: return "tn bprep_tc";
    case tn::ST_GEMM_TC: return "tn gemm_tc";
    case tn::ST_BPREP_C: return "tn bprep_simt";
    case tn::ST_GEMM_SIMT: return "tn gemm_simt";
    case tn::ST_ABSMAX: return "tn operand_max";
    default: return "tn step";
  }
}

}  // namespace

static const char* kVersion = "tn_gb300 0.1 (sm_103a)";

namespace tn {
// Lets other translation units of the library report through tn_last_error.
void set_last_error(const std::string& msg) { g_err = msg; }
}  // namespace tn

namespace tn {
// Host-side fault injection: TN_FAULT_INJECT is read on every check, so a
// test can arm and disarm a fault between calls.
static std::string fault_env() {
  const char* e = std::getenv("TN_FAULT_INJECT");
  return e ? std::string(e) : std::string();
}
bool fault_alloc() { return fault_env() == "alloc"; }
bool fault_slice(int64_t s, int64_t t) {
  const std::string f = fault_env();
  if (f.rfind("slice:", 0) != 0) return false;
  long long S = -1, T = 0;
  if (std::sscanf(f.c_str() + 6, "%lld:%lld", &S, &T) < 1) return false;
  return s == S && t == T;
}
bool fault_status() { return fault_env() == "status"; }
size_t fault_scratch() {
  const std::string f = fault_env();
  return f.rfind("scratch:", 0) == 0 ? (size_t)std::strtoull(f.c_str() + 8, nullptr, 10) : (size_t)-1;
}

// After the caller's stream is synchronised: a nonzero device status word of
// the plan means a bounded wait of a tensor-core GEMM gave up in some
// contraction of this plan since the last check.  The word is cleared, the
// head marked invalid and TN_ERR_TIMEOUT returned.
static int report_status(tn_head_t* h, unsigned int word, cudaStream_t st) {
  if (!word) return TN_OK;
  cudaMemsetAsync(h->plan->d_status, 0, sizeof(unsigned int), st);
  cudaStreamSynchronize(st);
  h->invalid = true;
  return fail(TN_ERR_TIMEOUT,
              "a bounded device wait in a contraction of this plan gave up (status " + std::to_string(word) +
                  "); the head is invalid until tn_head_reset");
}
}  // namespace tn

extern "C" const char* tn_last_error(void) { return g_err.c_str(); }
extern "C" const char* tn_version(void) { return kVersion; }

// Per-call scratch: a report in mapped host memory and the partial sums of a
// reduction on the device, plus a device and a pinned host buffer that grow on
// demand (prefix sums, GEMM operands, pattern maps).  Each call takes one for
// its duration, so calls from several threads and streams share none.  Between
// calls at most kMost are kept, with at most kKeepBytes of buffers among them;
// all of it is given back when a device allocation of the library fails.
// Every call that takes one synchronises its stream, which CUDA refuses while any
// stream is captured in global mode (and which ends that capture); beside a
// thread-local capture of another thread it may allocate and free.
struct CallScratch {
  tn::HeadReport* rep = nullptr;
  double* part = nullptr;
  void* buf = nullptr;
  size_t bytes = 0;
  void* host = nullptr;
  size_t host_bytes = 0;
  int device = -1;
};

static std::mutex g_scratch_mu;
static std::vector<CallScratch> g_scratch;

static void free_scratch(CallScratch& c) {
  cudaFreeHost(c.rep);
  cudaFreeHost(c.host);
  cudaFree(c.part);
  cudaFree(c.buf);
  c = CallScratch();
}

namespace tn {
void trim_scratch() {
  std::vector<CallScratch> kept;
  {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    kept.swap(g_scratch);
  }
  for (CallScratch& c : kept) free_scratch(c);
}

cudaError_t device_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    trim_scratch();
    e = cudaMalloc(p, bytes);
  }
  return e;
}
}  // namespace tn

struct ScratchLease {
  static constexpr size_t kMost = 32, kKeepBytes = (size_t)2 << 30;
  CallScratch c;
  cudaStream_t stream;
  bool in_flight = false;
  explicit ScratchLease(cudaStream_t st) : stream(st) {}
  ScratchLease(const ScratchLease&) = delete;
  ScratchLease& operator=(const ScratchLease&) = delete;
  ~ScratchLease() {
    if (!c.rep) return;
    if (in_flight) cudaStreamSynchronize(stream);   // the call failed after a launch
    {
      std::lock_guard<std::mutex> lock(g_scratch_mu);
      size_t kept = c.bytes + c.host_bytes;
      for (const CallScratch& o : g_scratch) kept += o.bytes + o.host_bytes;
      if (g_scratch.size() < kMost && kept <= kKeepBytes) {
        g_scratch.push_back(c);
        return;
      }
    }
    free_scratch(c);
  }
  // The report, once the stream is synchronised.
  tn::HeadReport done() {
    in_flight = false;
    return *c.rep;
  }
  // Call before the launches; the report starts as "nothing missing, no status".
  int take(size_t bytes, size_t host_bytes = 0) {
    int dev = -1;
    CUDA_TRY(cudaGetDevice(&dev));
    if (!c.rep) {   // (one that a failed attempt has taken is used again)
      // the kept one with the smallest buffer that is large enough, else the largest
      std::lock_guard<std::mutex> lock(g_scratch_mu);
      g_scratch.reserve(kMost);
      size_t at = g_scratch.size();
      for (size_t i = 0; i < g_scratch.size(); ++i) {
        if (g_scratch[i].device != dev) continue;
        if (at == g_scratch.size()) { at = i; continue; }
        const size_t x = g_scratch[i].bytes, y = g_scratch[at].bytes;
        if (x >= bytes ? (y < bytes || x < y) : (y < bytes && x > y)) at = i;
      }
      if (at < g_scratch.size()) {
        c = g_scratch[at];
        g_scratch.erase(g_scratch.begin() + (std::ptrdiff_t)at);
      }
    }
    if (!c.rep) {
      c.device = dev;
      void* h = nullptr;
      if (cudaHostAlloc(&h, sizeof(tn::HeadReport), cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess ||
          tn::device_malloc((void**)&c.part, 2 * tn::kHeadParts * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        if (h) cudaFreeHost(h);
        return fail(TN_ERR_OOM, "scratch allocation failed");
      }
      c.rep = (tn::HeadReport*)h;   // one address on host and device (unified addressing)
    }
    if (bytes > tn::fault_scratch())
      return fail(TN_ERR_OOM, "scratch allocation failed (injected: TN_FAULT_INJECT=scratch)");
    if (c.bytes < bytes) {
      cudaFree(c.buf);
      c.buf = nullptr;
      c.bytes = 0;
      if (tn::device_malloc(&c.buf, bytes) != cudaSuccess) {
        cudaGetLastError();
        return fail(TN_ERR_OOM, "scratch allocation failed");
      }
      c.bytes = bytes;
    }
    if (c.host_bytes < host_bytes) {
      cudaFreeHost(c.host);
      c.host = nullptr;
      c.host_bytes = 0;
      if (cudaHostAlloc(&c.host, host_bytes, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) {
        cudaGetLastError();
        return fail(TN_ERR_OOM, "scratch allocation failed");
      }
      c.host_bytes = host_bytes;
    }
    *c.rep = tn::HeadReport{~0ULL, 0u, {0.0, 0.0}};
    in_flight = true;
    return TN_OK;
  }
};

static void plan_release(tn_plan_t* p) {
  if (!p) return;
  if (p->on_device) {
    int cur = -1;
    cudaGetDevice(&cur);
    if (p->device >= 0) cudaSetDevice(p->device);
    cudaFree(p->d_leaves);
    cudaFree(p->d_meta);
    cudaFree(p->d_arena);
    cudaFree(p->d_keys);
    cudaFree(p->d_key_groups);
    cudaFree(p->d_tails);
    cudaFree(p->d_open);
    cudaFree(p->d_status);
    cudaFree(p->d_scale);
    for (auto& g : p->graphs) cudaGraphExecDestroy(g.exec);
    for (auto& e : p->prof_events) cudaEventDestroy(e);
    for (auto& e : p->side_fork) if (e) cudaEventDestroy(e);
    for (auto& e : p->side_join) if (e) cudaEventDestroy(e);
    if (p->side_stream) cudaStreamDestroy(p->side_stream);
    if (cur >= 0) cudaSetDevice(cur);
  }
  delete p;
}

extern "C" void tn_plan_free(tn_plan_t* plan) { plan_release(plan); }

static int plan_upload(tn_plan_t* p) {
  tn::Plan& P = p->P;
  if (tn::fault_alloc()) return fail(TN_ERR_OOM, "device allocation failed (injected: TN_FAULT_INJECT=alloc)");
  CUDA_TRY(cudaGetDevice(&p->device));
  CUDA_TRY(tn::prepare_gemm_tc());
  CUDA_TRY(tn::prepare_direct());
  std::vector<float2> leaves(P.leaf_arena.size());
  for (size_t i = 0; i < leaves.size(); ++i)
    leaves[i] = make_float2((float)P.leaf_arena[i].real(), (float)P.leaf_arena[i].imag());
  p->on_device = true;
  CUDA_TRY(tn::device_malloc((void**)&p->d_leaves, std::max<size_t>(leaves.size(), 1) * sizeof(float2)));
  if (!leaves.empty())
    CUDA_TRY(cudaMemcpy(p->d_leaves, leaves.data(), leaves.size() * sizeof(float2), cudaMemcpyHostToDevice));
  CUDA_TRY(tn::device_malloc((void**)&p->d_meta, std::max<size_t>(P.meta.size(), 1) * sizeof(uint32_t)));
  if (!P.meta.empty())
    CUDA_TRY(cudaMemcpy(p->d_meta, P.meta.data(), P.meta.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
  if (P.workspace_bytes > 0) {
    cudaError_t e = tn::device_malloc((void**)&p->d_arena, (size_t)P.workspace_bytes);
    if (e == cudaErrorMemoryAllocation && P.batch_max > 1) {
      // without the copies of the batched steps (up to 64 MB): every pass runs its whole launch list
      cudaGetLastError();
      P.workspace_bytes -= (P.batch_max - 1) * P.batch_stride;
      P.batch_max = 1;
      e = tn::device_malloc((void**)&p->d_arena, (size_t)P.workspace_bytes);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      return fail(TN_ERR_OOM, "workspace of " + std::to_string(P.workspace_bytes) + " bytes: " + cudaGetErrorString(e));
    }
  }
  // amplitude lookup table
  const size_t L = P.tails_raw.size();
  std::vector<std::pair<uint64_t, uint32_t>> kv(L);
  for (size_t g = 0; g < L; ++g) kv[g] = {P.tails_raw[g] & P.tail_mask, (uint32_t)g};
  std::sort(kv.begin(), kv.end());
  std::vector<uint64_t> keys(L);
  std::vector<uint32_t> grp(L);
  for (size_t i = 0; i < L; ++i) { keys[i] = kv[i].first; grp[i] = kv[i].second; }
  p->n_keys = (int64_t)L;
  CUDA_TRY(tn::device_malloc((void**)&p->d_keys, L * sizeof(uint64_t)));
  CUDA_TRY(tn::device_malloc((void**)&p->d_key_groups, L * sizeof(uint32_t)));
  CUDA_TRY(tn::device_malloc((void**)&p->d_tails, L * sizeof(uint64_t)));
  CUDA_TRY(cudaMemcpy(p->d_keys, keys.data(), L * sizeof(uint64_t), cudaMemcpyHostToDevice));
  CUDA_TRY(cudaMemcpy(p->d_key_groups, grp.data(), L * sizeof(uint32_t), cudaMemcpyHostToDevice));
  CUDA_TRY(cudaMemcpy(p->d_tails, P.tails_raw.data(), L * sizeof(uint64_t), cudaMemcpyHostToDevice));
  const size_t h = P.open_qubits.size();
  CUDA_TRY(tn::device_malloc((void**)&p->d_open, std::max<size_t>(h, 1) * sizeof(int)));
  if (h) CUDA_TRY(cudaMemcpy(p->d_open, P.open_qubits.data(), h * sizeof(int), cudaMemcpyHostToDevice));
  CUDA_TRY(tn::device_malloc((void**)&p->d_status, sizeof(unsigned int)));
  CUDA_TRY(cudaMemset(p->d_status, 0, sizeof(unsigned int)));
  const size_t n_static = P.scale_static.size(), n_slots = n_static + (size_t)P.n_scale_slots * P.batch_max;
  if (n_slots > 0) {
    CUDA_TRY(tn::device_malloc((void**)&p->d_scale, n_slots * sizeof(unsigned int)));
    CUDA_TRY(cudaMemset(p->d_scale, 0, n_slots * sizeof(unsigned int)));
    if (n_static)
      CUDA_TRY(cudaMemcpy(p->d_scale, P.scale_static.data(), n_static * sizeof(unsigned int), cudaMemcpyHostToDevice));
  }
  if (P.n_side_bprep > 0) {
    const size_t ns = P.steps.size();
    p->side_fork.assign(ns, nullptr);
    p->side_join.assign(ns, nullptr);
    p->forks_at.assign(ns, {});
    CUDA_TRY(cudaStreamCreateWithFlags(&p->side_stream, cudaStreamNonBlocking));
    for (size_t i = 0; i < ns; ++i) {
      const int f = P.steps[i].fork;
      if (f < 0) continue;
      if (f >= (int)i) return fail(TN_ERR_INVALID, "internal: side step forks after itself");
      p->forks_at[f].push_back((int)i);
      if (!p->side_fork[f]) CUDA_TRY(cudaEventCreateWithFlags(&p->side_fork[f], cudaEventDisableTiming));
      CUDA_TRY(cudaEventCreateWithFlags(&p->side_join[i], cudaEventDisableTiming));
    }
  }
  return TN_OK;
}

extern "C" int tn_plan(const tn_circuit* circuit, const tn_open_spec* open_spec, const tn_edge* sliced_edges,
                       int n_edges, const int32_t* order, int64_t n_pairs, const tn_plan_opts* opts,
                       tn_plan_t** out) {
  if (!out) return fail(TN_ERR_INVALID, "out is NULL");
  *out = nullptr;
  if (!circuit || !open_spec) return fail(TN_ERR_INVALID, "circuit or open_spec is NULL");
  if (circuit->n_gates > 0 && !circuit->gates) return fail(TN_ERR_INVALID, "gates is NULL");
  if (open_spec->n_open < 0 || (open_spec->n_open > 0 && !open_spec->open_qubits))
    return fail(TN_ERR_INVALID, "bad open qubit list");
  if (open_spec->n_tails < 1 || !open_spec->tails) return fail(TN_ERR_INVALID, "need at least one tail");
  if (n_edges < 0 || (n_edges > 0 && !sliced_edges)) return fail(TN_ERR_INVALID, "bad edge list");
  if (order && n_pairs < 0) return fail(TN_ERR_INVALID, "n_pairs < 0");
  tn::PlanInput in;
  in.n_qubits = circuit->n_qubits;
  in.n_gates = circuit->n_gates;
  std::vector<int> ar(circuit->n_gates), q0(circuit->n_gates), q1(circuit->n_gates);
  std::vector<tn::cd> mats((size_t)circuit->n_gates * 16);
  for (int g = 0; g < circuit->n_gates; ++g) {
    const tn_gate& G = circuit->gates[g];
    ar[g] = G.arity;
    q0[g] = G.q0;
    q1[g] = G.q1;
    for (int e = 0; e < 16; ++e) mats[(size_t)g * 16 + e] = tn::cd(G.re[e], G.im[e]);
  }
  in.arity = ar.data();
  in.q0 = q0.data();
  in.q1 = q1.data();
  in.mats = mats.data();
  in.open_qubits.assign(open_spec->open_qubits, open_spec->open_qubits + open_spec->n_open);
  in.tails.assign(open_spec->tails, open_spec->tails + open_spec->n_tails);
  for (int e = 0; e < n_edges; ++e)
    in.edges.push_back({sliced_edges[e].gate, sliced_edges[e].leg, sliced_edges[e].kind, sliced_edges[e].value});
  in.order = order;
  in.n_pairs = order ? n_pairs : 0;
  bool host_only = false;
  if (opts) {
    if (opts->max_log2_elements > 0) in.cap_log2 = opts->max_log2_elements;
    in.gemm_engine = opts->gemm;
    host_only = opts->host_only != 0;
    if (opts->order_trials > 0) in.order_trials = opts->order_trials;
    if (opts->order_seed) in.order_seed = opts->order_seed;
    if (opts->max_host_absorb_log2 > 0) in.absorb_log2 = opts->max_host_absorb_log2;
    if (opts->small_max_bits != 0) in.small_max_bits = opts->small_max_bits < 0 ? -1 : std::min(4, opts->small_max_bits);
    if (opts->auto_slice < 0 || opts->auto_slice > 24) return fail(TN_ERR_INVALID, "auto_slice must be in [0, 24]");
    in.auto_slice = opts->auto_slice;
    if (opts->host_fold_log2 > 16) return fail(TN_ERR_INVALID, "host_fold_log2 must be at most 16");
    if (opts->host_fold_log2 != 0) in.fold_log2 = opts->host_fold_log2 < 0 ? -1 : opts->host_fold_log2;
    in.gemm_pair = opts->gemm_pair < 0 ? -1 : 0;
    in.side_bprep = opts->side_bprep > 0;
  }
  if (in.gemm_engine < 0 || in.gemm_engine > 4) return fail(TN_ERR_INVALID, "unknown gemm engine");
  if (in.cap_log2 > 34) return fail(TN_ERR_INVALID, "size cap above 2^34 elements");
  tn_plan_t* p = new tn_plan_t();
  std::string err;
  int rc = tn::build_plan(in, p->P, err);
  if (rc) {
    delete p;
    return fail(rc, err);
  }
  if (!host_only) {
    rc = plan_upload(p);
    if (rc) {
      plan_release(p);
      return rc;
    }
  }
  *out = p;
  return TN_OK;
}

extern "C" int tn_plan_get_stats(const tn_plan_t* plan, tn_plan_stats* s) {
  if (!plan || !s) return fail(TN_ERR_INVALID, "NULL argument");
  const tn::Plan& P = plan->P;
  std::memset(s, 0, sizeof(*s));
  s->n_qubits = P.n_qubits;
  s->n_open = (int)P.open_qubits.size();
  s->n_tails = (int64_t)P.tails_raw.size();
  s->n_patterns = P.n_patterns_final;
  s->n_sliced = P.n_sliced;
  s->n_pinned = P.n_pinned;
  s->n_leaves = (int)P.leaves.size();
  s->n_contractions = P.n_contractions;
  const double ni = std::ldexp(1.0, P.n_internal);
  s->n_launches = (int)(((int64_t)P.steps.size() + 1) << P.n_internal);
  s->tc_macs = P.tc_macs * ni;
  s->alg_bytes = P.alg_bytes * ni;
  s->n_internal_sliced = P.n_internal;
  s->gemm_pair = P.gemm_pair;
  s->n_side_bprep = P.n_side_bprep;
  s->max_log2_elements = P.max_log2;
  s->workspace_bytes = P.workspace_bytes;
  s->measured_slice_ms = plan->measured_slice_ms;
  s->autotune_candidates = plan->autotune_candidates;
  s->tune_default_ms = plan->tune_default_ms;
  s->tune_tuned_ms = plan->tune_tuned_ms;
  for (auto& st : P.steps) {
    if (st.variant != 0) ++s->n_tuned_steps;
    if (st.kind == tn::ST_GEMM_TC) ++s->n_gemm_tc;
    if (st.kind == tn::ST_GEMM_SIMT) ++s->n_gemm_simt;
    if (st.kind == tn::ST_SMALL) ++s->n_small;
    if (st.kind == tn::ST_PERMUTE) ++s->n_permute;
  }
  return TN_OK;
}

extern "C" int tn_plan_order(const tn_plan_t* plan, int32_t* pairs, int64_t cap, int64_t* n_pairs) {
  if (!plan || !n_pairs) return fail(TN_ERR_INVALID, "NULL argument");
  const auto& o = plan->P.order;
  *n_pairs = (int64_t)o.size();
  for (int64_t i = 0; i < std::min<int64_t>(cap, (int64_t)o.size()); ++i) {
    pairs[2 * i] = o[i].first;
    pairs[2 * i + 1] = o[i].second;
  }
  return TN_OK;
}

extern "C" const char* tn_plan_describe(tn_plan_t* plan, int with_data) {
  if (!plan) return "";
  plan->P.describe_cache = tn::describe_plan(plan->P, with_data != 0);
  return plan->P.describe_cache.c_str();
}

// ----------------------------------------------------------------- heads

extern "C" int tn_head_create(tn_plan_t* plan, void* dev_c128, tn_head_t** out) {
  if (!plan || !out) return fail(TN_ERR_INVALID, "NULL argument");
  *out = nullptr;
  if (!plan->on_device) return fail(TN_ERR_INVALID, "plan was made host_only");
  if (tn::fault_alloc()) return fail(TN_ERR_OOM, "head allocation failed (injected: TN_FAULT_INJECT=alloc)");
  tn_head* h = new tn_head();
  h->plan = plan;
  const int64_t L = (int64_t)plan->P.tails_raw.size();
  const int64_t elems = L << plan->P.open_qubits.size();
  if (dev_c128) {
    h->H = (double2*)dev_c128;
  } else {
    cudaError_t e = tn::device_malloc((void**)&h->H, (size_t)elems * sizeof(double2));
    if (e != cudaSuccess) {
      cudaGetLastError();
      delete h;
      return fail(TN_ERR_OOM, std::string("head allocation: ") + cudaGetErrorString(e));
    }
    h->owns = true;
  }
  cudaError_t e1 = cudaMemset(h->H, 0, (size_t)elems * sizeof(double2));
  if (e1 == cudaSuccess) e1 = cudaStreamSynchronize(0);   // zeroed before any stream, blocking or not, uses it
  cudaError_t e2 = tn::device_malloc((void**)&h->d_Z, (size_t)std::max<int64_t>(L, 1) * sizeof(double));
  if (e1 != cudaSuccess || e2 != cudaSuccess) {
    cudaGetLastError();
    tn_head_free(h);
    return fail(TN_ERR_CUDA, "head set-up failed");
  }
  *out = h;
  return TN_OK;
}

extern "C" void tn_head_free(tn_head_t* h) {
  if (!h) return;
  if (h->owns) cudaFree(h->H);
  cudaFree(h->d_Z);
  cudaFree(h->d_stage);
  delete h;
}

extern "C" void* tn_head_data(tn_head_t* h) {
  if (!h) return nullptr;
  h->exposed = true;
  return h->H;
}

static int64_t head_elems(const tn_head_t* h) {
  return (int64_t)h->plan->P.tails_raw.size() << h->plan->P.open_qubits.size();
}

extern "C" int tn_head_reset(tn_head_t* h, void* stream) {
  if (!h) return fail(TN_ERR_INVALID, "NULL head");
  CUDA_TRY(cudaMemsetAsync(h->H, 0, (size_t)head_elems(h) * sizeof(double2), (cudaStream_t)stream));
  h->done.clear();
  h->slices_done = 0;
  h->f_override = false;
  h->invalid = false;
  return TN_OK;
}

extern "C" int tn_head_fidelity(const tn_head_t* h, double* f_est, int64_t* slices_done) {
  if (!h) return fail(TN_ERR_INVALID, "NULL head");
  const tn::Plan& P = h->plan->P;
  double f = h->f_override ? h->f_value
                           : std::ldexp((double)h->slices_done, -P.n_sliced) * std::ldexp(1.0, -P.n_pinned) *
                                 P.companion_factor;
  if (f_est) *f_est = f;
  if (slices_done) *slices_done = h->slices_done;
  return TN_OK;
}

extern "C" int tn_head_set_fidelity(tn_head_t* h, double f) {
  if (!h || !(f >= 0.0) || f > 1.0) return fail(TN_ERR_INVALID, "bad head or fidelity");
  h->f_override = true;
  h->f_value = f;
  return TN_OK;
}

// -------------------------------------------------------- slice execution

// b: the pass's place in its chunk, which selects its copies of batched
// buffers and of the scale slots
static inline float2* buf_ptr(const tn_plan_t* p, const tn::Ref& r, int b) {
  const tn::BufInfo& bi = p->P.bufs[r.id];
  return (float2*)(p->d_arena + bi.off + (bi.batch ? b * p->P.batch_stride : 0));
}

static inline const float2* ref_ptr(const tn_plan_t* p, const tn::Ref& r, int64_t s, int b) {
  if (r.kind == 0) {
    const tn::LeafInfo& li = p->P.leaf_info[r.id];
    int64_t v = 0;
    for (size_t t = 0; t < li.var_slice_bits.size(); ++t) v |= ((s >> li.var_slice_bits[t]) & 1) << t;
    return p->d_leaves + li.off + v * li.size;
  }
  return buf_ptr(p, r, b);
}

// FP16x3 scale slot -> device address (static slots first, then the per-pass ones)
static unsigned int* scale_ptr(const tn_plan_t* p, int slot, int b) {
  if (slot == -1) return nullptr;
  const int64_t n_static = (int64_t)p->P.scale_static.size();
  return p->d_scale + (slot >= 0 ? n_static + (int64_t)b * p->P.n_scale_slots + slot : (int64_t)(-(slot + 2)));
}

// An operand of a batched launch: base address of batch element 0 and how the others follow.
static const float2* batch_operand(const tn_plan_t* p, const tn::Ref& r, tn::BatchOperand& o) {
  o = tn::BatchOperand();
  if (r.kind == 1) {
    o.stride = p->P.batch_stride / (int64_t)sizeof(float2);
    return buf_ptr(p, r, 0);
  }
  const tn::LeafInfo& li = p->P.leaf_info[r.id];
  o.var_size = li.size;
  o.n_bits = std::min((int)li.var_slice_bits.size(), 8);   // at most 8 (mark_batched)
  for (int t = 0; t < o.n_bits; ++t) o.bits[t] = (uint8_t)li.var_slice_bits[t];
  return p->d_leaves + li.off;
}

// Passes q0 .. q0 + n - 1 for a launch of them all.
static void batch_range(const tn_plan_t* p, int64_t q0, int n, tn::BatchParams& q) {
  q.n_batch = n;
  q.q0 = q0;
  q.ni = p->P.n_internal;
  q.k = p->P.n_sliced;
  q.amax_stride = p->P.n_scale_slots;
}

// Launch parameters of a permute step (for a B preparation in the permute form:
// of its schedule) and of a B preparation by gather.
static tn::PermParams perm_params(const tn_plan_t* p, const tn::Step& x, int64_t s, int b) {
  tn::PermParams pp;
  pp.in = ref_ptr(p, x.a, s, b);
  pp.out = buf_ptr(p, x.c, b);
  pp.pstride = 1LL << x.rA;
  pp.P = x.PA;
  pp.t = x.t_bits;
  pp.n_rest = x.n_rest;
  std::memcpy(pp.rest_in, x.rest_in, sizeof(pp.rest_in));
  std::memcpy(pp.rest_out, x.rest_out, sizeof(pp.rest_out));
  pp.tab = p->d_meta + x.tab_off;
  pp.split = x.split;
  pp.scale = scale_ptr(p, x.slot, b);
  pp.vec4 = x.vec4;
  return pp;
}

static tn::BPrepParams bprep_params(const tn_plan_t* p, const tn::Step& x, int64_t s, int b) {
  tn::BPrepParams bp;
  bp.B = ref_ptr(p, x.a, s, b);
  bp.out = buf_ptr(p, x.c, b);
  bp.b_pstride = 1LL << x.rA;
  bp.PB = x.PA;
  bp.nk = x.nk;
  bp.nn = x.nn;
  bp.bk = p->d_meta + x.bk_off;
  bp.bn = p->d_meta + x.bn_off;
  bp.h16 = x.h16;
  bp.scale = scale_ptr(p, x.slot, b);
  return bp;
}

static bool bprep_embeds(const tn::Step& x) {
  return x.kind == tn::ST_BPREP_TC && !x.alts.empty() && (x.variant == 0) == (x.bprep_embed0 != 0);
}

// Whether the permute step x and the step y after it are the two operands of one
// GEMM that launch_operands prepares together (y does not read x's result: it
// prepares the other operand).
static bool joined_operands(const tn::Step& x, const tn::Step& y) {
  return x.kind == tn::ST_PERMUTE && x.split >= 1 && y.kind == tn::ST_BPREP_TC && y.h16 + 1 == x.split &&
         y.contraction == x.contraction && y.fork < 0 && !bprep_embeds(y);
}

// Launch one step of the launch list for the full slice id s on stream st
// (`side`: a B-prep beside a running GEMM, launched with one block per SM); b is
// the pass's place in its chunk.  n_batch > 1: a batched step, for the passes
// q0 .. q0 + n_batch - 1 at once.
static cudaError_t launch_step(tn_plan_t* p, const tn::Step& x, int64_t s, cudaStream_t st, bool side, int b,
                               int n_batch = 1, int64_t q0 = 0) {
  const tn::Plan& P = p->P;
  NvtxRange range(step_range_name(x.kind));
  cudaError_t e = cudaSuccess;
  switch (x.kind) {
    case tn::ST_SMALL: {
      if (x.direct) {
        const tn::Ref &rx = x.dp.swap ? x.b : x.a, &ry = x.dp.swap ? x.a : x.b;
        tn::DirectParams dp{};
        tn::direct_fill(x.dp, x.PC, dp);
        dp.X = ref_ptr(p, rx, s, b);
        dp.Y = ref_ptr(p, ry, s, b);
        dp.C = buf_ptr(p, x.c, b);
        dp.x_pstride = 1LL << (x.dp.swap ? x.rB : x.rA);
        dp.y_pstride = 1LL << (x.dp.swap ? x.rA : x.rB);
        dp.c_pstride = 1LL << x.rC;
        dp.mapX = p->d_meta + (x.dp.swap ? x.mapB_off : x.mapA_off);
        dp.mapY = p->d_meta + (x.dp.swap ? x.mapA_off : x.mapB_off);
        dp.mapX_mode = x.dp.swap ? x.mapB_mode : x.mapA_mode;
        dp.mapY_mode = x.dp.swap ? x.mapA_mode : x.mapB_mode;
        dp.bf16 = P.gemm_engine == TN_GEMM_TC_BF16X3 && x.nk >= 2;   // K = 2 GEMM steps run in tf32
        dp.vec = 1;                      // buffers start on 256 bytes, rows pair up from even ones
        dp.amax = scale_ptr(p, x.max_slot, b);
        if (n_batch > 1) {
          batch_range(p, q0, n_batch, dp);
          dp.X = batch_operand(p, rx, dp.bA);
          dp.Y = batch_operand(p, ry, dp.bB);
          batch_operand(p, x.c, dp.bC);
        }
        e = tn::launch_direct(dp, x.dp.config, st);
        break;
      }
      tn::SmallParams sp;
      sp.A = ref_ptr(p, x.a, s, b);
      sp.B = ref_ptr(p, x.b, s, b);
      sp.C = buf_ptr(p, x.c, b);
      sp.a_pstride = 1LL << x.rA;
      sp.b_pstride = 1LL << x.rB;
      sp.c_pstride = 1LL << x.rC;
      sp.M = 1LL << (x.rA - x.nk);
      sp.PC = x.PC;
      sp.rA = x.rA;
      sp.nk = x.nk;
      sp.nn = x.nn;
      for (int j = 0; j < 4; ++j) sp.kpos[j] = x.kposA[j];
      std::memcpy(sp.boffK, x.boffK, sizeof(sp.boffK));
      std::memcpy(sp.boffN, x.boffN, sizeof(sp.boffN));
      sp.mapA = p->d_meta + x.mapA_off;
      sp.mapB = p->d_meta + x.mapB_off;
      sp.mapA_mode = x.mapA_mode;
      sp.mapB_mode = x.mapB_mode;
      sp.amax = scale_ptr(p, x.max_slot, b);
      if (n_batch > 1) {
        batch_range(p, q0, n_batch, sp);
        sp.A = batch_operand(p, x.a, sp.bA);
        sp.B = batch_operand(p, x.b, sp.bB);
        batch_operand(p, x.c, sp.bC);
      }
      e = tn::launch_small(sp, st);
      break;
    }
    case tn::ST_PERMUTE: {
      const tn::PermParams pp = perm_params(p, x, s, b);
      e = tn::launch_permute(pp, st);
      break;
    }
    case tn::ST_BPREP_C:
    case tn::ST_BPREP_TC: {
      if (bprep_embeds(x)) {
        // the permute kernel onto [N][K] order, writing the real embedding
        tn::PermParams pp = perm_params(p, x, s, b);
        pp.split = 4 + x.h16;
        pp.embed_nk = x.nk;
        e = tn::launch_permute(pp, st);
        break;
      }
      const tn::BPrepParams bp = bprep_params(p, x, s, b);
      e = x.kind == tn::ST_BPREP_C ? tn::launch_bprep_c(bp, st) : tn::launch_bprep_tc(bp, st, side);
      break;
    }
    case tn::ST_GEMM_SIMT:
    case tn::ST_GEMM_TC: {
      tn::GemmParams gp;
      gp.A = ref_ptr(p, x.a, s, b);
      gp.B = (const void*)ref_ptr(p, x.b, s, b);
      gp.C = buf_ptr(p, x.c, b);
      gp.M = 1LL << x.nm;
      gp.N = 1LL << x.nn;
      gp.K = 1LL << x.nk;
      gp.PA = x.PA;
      gp.PB = x.PB;
      gp.PC = x.PC;
      gp.mapA = p->d_meta + x.mapA_off;
      gp.mapB = p->d_meta + x.mapB_off;
      gp.mapA_mode = x.mapA_mode;
      gp.mapB_mode = x.mapB_mode;
      gp.h16 = x.h16;
      gp.scaleA = scale_ptr(p, x.slot, b);
      gp.scaleB = scale_ptr(p, x.slotB, b);
      gp.amax = scale_ptr(p, x.max_slot, b);
      gp.pair = P.gemm_pair < 0 ? -1 : x.pair;
      gp.tile_cap = x.tile_cap;
      if (x.grp_fold > 0) {
        gp.grp = p->d_meta + x.grp_off;
        gp.grp_fold = x.grp_fold;
        gp.n_groups = x.n_groups;
      }
      e = x.kind == tn::ST_GEMM_SIMT ? tn::launch_gemm_simt(gp, st) : tn::launch_gemm_tc(gp, p->d_status, st);
      break;
    }
    case tn::ST_ABSMAX: {
      tn::AbsmaxParams ap;
      ap.in = ref_ptr(p, x.a, s, b);
      ap.n = x.PA << x.rA;
      ap.out = scale_ptr(p, x.slot, b);
      e = tn::launch_absmax(ap, st);
      break;
    }
    default:
      return cudaErrorInvalidValue;
  }
  return e;
}

static tn::AccumParams accum_params(const tn_plan_t* p, double2* H) {
  const tn::Plan& P = p->P;
  tn::AccumParams ap;
  ap.H = H;
  ap.f_pstride = 1LL << P.fin.rF;
  ap.L = (int64_t)P.tails_raw.size();
  ap.h = (int)P.open_qubits.size();
  ap.pidx = p->d_meta + P.fin.pidx_off;
  for (int j = 0; j < ap.h && j < 32; ++j) ap.open_pos[j] = P.fin.open_pos[j];
  return ap;
}

// One pass of the launch list for the full slice id s (user bits, then the
// bits of automatically sliced edges).  With per-launch timing events (ev)
// every step runs in order on st; otherwise a B-prep step with fork f is
// launched on the plan's side stream just before step f (after everything
// before f is done) and step f + ... waits for it right before the GEMM that
// consumes its output.
// chunk_pass >= 0: this pass of a chunk, whose batched steps have run and whose
// scale slots were zeroed; -1: the whole launch list.
static int run_pass(tn_plan_t* p, int64_t s, double2* H, cudaStream_t st, cudaEvent_t* ev, int chunk_pass = -1) {
  const tn::Plan& P = p->P;
  NvtxRange range("tn pass");
  const int b = std::max(chunk_pass, 0);
  if (P.n_scale_slots > 0 && chunk_pass < 0) {
    cudaError_t e = cudaMemsetAsync(p->d_scale + P.scale_static.size(), 0,
                                    (size_t)P.n_scale_slots * sizeof(unsigned int), st);
    if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("scale reset: ") + cudaGetErrorString(e));
  }
  const bool use_side = !ev && p->side_stream != nullptr;
  std::vector<int> pending;      // side steps launched and not yet joined
  auto join_pending = [&]() {
    for (int j : pending) cudaStreamWaitEvent(st, p->side_join[j], 0);
    pending.clear();
  };
  int si = 0;
  for (const tn::Step& x : P.steps) {
    cudaError_t e = cudaSuccess;
    if (chunk_pass >= 0 && x.batch) {
      ++si;
      continue;
    }
    if (use_side && !p->forks_at[si].empty()) {
      e = cudaEventRecord(p->side_fork[si], st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(p->side_stream, p->side_fork[si], 0);
      for (int j : p->forks_at[si]) {
        if (e == cudaSuccess) e = launch_step(p, P.steps[j], s, p->side_stream, true, b);
        if (e == cudaSuccess) e = cudaEventRecord(p->side_join[j], p->side_stream);
        if (e == cudaSuccess) pending.push_back(j);
      }
      if (e != cudaSuccess) {
        join_pending();
        return fail(TN_ERR_CUDA, std::string("side launch: ") + cudaGetErrorString(e));
      }
    }
    if (ev) cudaEventRecord(ev[2 * si], st);
    if (use_side && x.fork >= 0) {
      // launched on the side stream before step x.fork: wait for it here
      e = cudaStreamWaitEvent(st, p->side_join[si], 0);
      pending.erase(std::remove(pending.begin(), pending.end(), si), pending.end());
    } else if (!ev && si > 0 && joined_operands(P.steps[si - 1], x)) {
      // launched with the permute before it
    } else if (!ev && si + 1 < (int)P.steps.size() && joined_operands(x, P.steps[si + 1])) {
      NvtxRange range("tn operands");
      e = tn::launch_operands(perm_params(p, x, s, b), bprep_params(p, P.steps[si + 1], s, b), st);
    } else {
      e = launch_step(p, x, s, st, false, b);
    }
    if (e == cudaErrorInvalidValue && (x.kind < 0 || x.kind > tn::ST_ABSMAX)) {
      join_pending();
      return fail(TN_ERR_INVALID, "internal: unknown step kind");
    }
    if (e != cudaSuccess) {
      join_pending();
      return fail(TN_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
    }
    if (ev) cudaEventRecord(ev[2 * si + 1], st);
    ++si;
  }
  join_pending();
  if (ev) cudaEventRecord(ev[2 * si], st);
  tn::AccumParams ap = accum_params(p, H);
  ap.F = ref_ptr(p, P.fin.ref, s, b);
  cudaError_t e = tn::launch_accum(ap, st);
  if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("accumulate launch: ") + cudaGetErrorString(e));
  if (ev) cudaEventRecord(ev[2 * si + 1], st);
  return TN_OK;
}

// Passes [q, q_end) of the plan (pass q: user slice q >> n_internal, value
// q & (2^n_internal - 1) of the automatically sliced edges), each accumulating
// into H, in chunks whose batched steps are launched for all their passes at
// once.  *done (if given) receives the end of the passes enqueued whole: a
// failing pass fails before its accumulation launch, so exactly those reach H.
static int run_passes(tn_plan_t* p, int64_t q, int64_t q_end, double2* H, cudaStream_t st, int64_t* done = nullptr) {
  const tn::Plan& P = p->P;
  const int ni = P.n_internal;
  auto slice_id = [&](int64_t x) { return (x >> ni) | ((x & ((1LL << ni) - 1)) << P.n_sliced); };
  auto injected = [&](int64_t x) {
    const int64_t s = x >> ni, t = x & ((1LL << ni) - 1);
    if (!tn::fault_slice(s, t)) return (int)TN_OK;
    return fail(TN_ERR_CUDA, "injected failure before pass " + std::to_string(t) + " of slice " + std::to_string(s) +
                                 " (TN_FAULT_INJECT)");
  };
  bool all_batched = true;
  for (const tn::Step& x : P.steps) all_batched = all_batched && x.batch;
  if (done) *done = q;
  while (q < q_end) {
    const int n = (int)std::min<int64_t>(P.batch_max, q_end - q);
    if (n == 1) {
      if (int rc = injected(q)) return rc;
      if (int rc = run_pass(p, slice_id(q), H, st, nullptr)) return rc;
      ++q;
      if (done) *done = q;
      continue;
    }
    NvtxRange range("tn chunk");
    if (P.n_scale_slots > 0) {
      const cudaError_t e = cudaMemsetAsync(p->d_scale + P.scale_static.size(), 0,
                                            (size_t)n * P.n_scale_slots * sizeof(unsigned int), st);
      if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("scale reset: ") + cudaGetErrorString(e));
    }
    for (const tn::Step& x : P.steps) {
      if (!x.batch) continue;
      const cudaError_t e = launch_step(p, x, 0, st, false, 0, n, q);
      if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
    }
    if (all_batched) {
      int rc = TN_OK, m = 0;
      while (m < n && (rc = injected(q + m)) == TN_OK) ++m;
      if (m > 0) {
        tn::AccumParams ap = accum_params(p, H);
        batch_range(p, q, m, ap);
        ap.F = batch_operand(p, P.fin.ref, ap.bA);
        const cudaError_t e = tn::launch_accum(ap, st);
        if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("accumulate launch: ") + cudaGetErrorString(e));
      }
      q += m;
      if (done) *done = q;
      if (rc) return rc;
      continue;
    }
    for (int b = 0; b < n; ++b, ++q) {
      if (int rc = injected(q)) return rc;
      if (int rc = run_pass(p, slice_id(q), H, st, nullptr, b)) return rc;
      if (done) *done = q + 1;
    }
  }
  return TN_OK;
}

static int run_slice(tn_plan_t* p, int64_t s, double2* H, cudaStream_t st) {
  return run_passes(p, s << p->P.n_internal, (s + 1) << p->P.n_internal, H, st);
}

static int check_range(tn_plan_t* plan, tn_range r, tn_head_t* head) {
  if (!plan || !head) return fail(TN_ERR_INVALID, "NULL argument");
  if (head->plan != plan) return fail(TN_ERR_INVALID, "head belongs to another plan");
  if (!plan->on_device) return fail(TN_ERR_INVALID, "plan was made host_only");
  if (head->invalid)
    return fail(TN_ERR_INVALID, "head is invalid after a failed or timed-out contraction; call tn_head_reset");
  const int64_t ns = 1LL << plan->P.n_sliced;
  if (r.begin < 0 || r.end > ns || r.begin > r.end) return fail(TN_ERR_INVALID, "slice range outside [0, 2^k)");
  auto it = head->done.upper_bound(r.begin);
  if (it != head->done.begin()) {
    auto pv = std::prev(it);
    if (pv->second > r.begin && r.begin < r.end)
      return fail(TN_ERR_INVALID, "slice range overlaps slices already accumulated");
  }
  if (it != head->done.end() && it->first < r.end)
    return fail(TN_ERR_INVALID, "slice range overlaps slices already accumulated");
  return TN_OK;
}

static void mark_done(tn_head_t* head, tn_range r) {
  if (r.begin >= r.end) return;   // an empty range records nothing (and must not replace [b, e))
  head->done[r.begin] = r.end;
  head->slices_done += r.end - r.begin;
}

extern "C" int tn_profile_slices(tn_plan_t* plan, tn_range r, tn_head_t* head, void* stream, double* step_ms,
                                 int64_t n_entries) {
  int rc = check_range(plan, r, head);
  if (rc) return rc;
  const int64_t ns = (int64_t)plan->P.steps.size() + 1;
  if (!step_ms || n_entries < ns) return fail(TN_ERR_INVALID, "step_ms needs n_launches entries");
  for (int64_t i = 0; i < ns; ++i) step_ms[i] = 0.0;
  if (r.begin == r.end) return TN_OK;
  cudaStream_t st = (cudaStream_t)stream;
  // events for up to kBatch passes, recorded back to back and read after one
  // synchronisation per batch (no host round trip between the passes of a batch)
  constexpr int64_t kBatch = 64;
  const int64_t ni = 1LL << plan->P.n_internal;
  const int64_t npass = (r.end - r.begin) * ni;
  const size_t need = (size_t)(2 * ns * std::min(npass, kBatch));
  auto& ev = plan->prof_events;
  while (ev.size() < need) {
    cudaEvent_t e;
    CUDA_TRY(cudaEventCreate(&e));
    ev.push_back(e);
  }
  int status = TN_OK;
  int64_t passes_run = 0;
  for (int64_t q0 = 0; q0 < npass && status == TN_OK; q0 += kBatch) {
    const int64_t nb = std::min(kBatch, npass - q0);
    for (int64_t j = 0; j < nb && status == TN_OK; ++j) {
      const int64_t q = r.begin * ni + q0 + j;
      const int64_t s = (q / ni) | ((q % ni) << plan->P.n_sliced);
      status = run_pass(plan, s, head->H, st, ev.data() + 2 * ns * j);
      if (status == TN_OK) ++passes_run;
    }
    if (status) break;
    cudaError_t e = cudaEventSynchronize(ev[(size_t)(2 * ns * nb - 1)]);
    if (e != cudaSuccess) { status = fail(TN_ERR_CUDA, cudaGetErrorString(e)); break; }
    for (int64_t j = 0; j < nb; ++j)
      for (int64_t i = 0; i < ns; ++i) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[(size_t)(2 * ns * j + 2 * i)], ev[(size_t)(2 * ns * j + 2 * i + 1)]);
        step_ms[i] += ms;
      }
  }
  if (status == TN_OK) mark_done(head, r);
  else if (passes_run > 0) head->invalid = true;   // H holds an unrecorded part of the range
  return status;
}

extern "C" int tn_plan_step_info(const tn_plan_t* plan, int64_t i, int* kind, double* macs, double* bytes) {
  if (!plan) return fail(TN_ERR_INVALID, "NULL plan");
  const int64_t ns = (int64_t)plan->P.steps.size();
  if (i < 0 || i > ns) return fail(TN_ERR_INVALID, "step index out of range");
  if (i == ns) {
    const tn::Plan& P = plan->P;
    const double L = (double)P.tails_raw.size(), l = std::ldexp(1.0, (int)P.open_qubits.size());
    if (kind) *kind = -1;
    if (macs) *macs = 0.0;
    if (bytes) *bytes = L * l * (8.0 + 32.0);   // read F (c64), read+write H (c128)
    return TN_OK;
  }
  const tn::Step& x = plan->P.steps[i];
  if (kind) *kind = x.kind;
  if (macs) *macs = x.macs;
  if (bytes) *bytes = x.bytes;
  return TN_OK;
}

// ------------------------------------------------ per-step tile variants

namespace {

struct GemmVariant {
  int cap, pair;
};
// widest tile (real columns) and CTA pairs allowed (0) or not (-1)
constexpr GemmVariant kGemmVariants[] = {{256, 0}, {256, -1}, {128, 0}, {64, 0}, {32, 0}};
constexpr int kNumGemmVariants = (int)(sizeof(kGemmVariants) / sizeof(kGemmVariants[0]));

// Indices into kGemmVariants of the choices that launch differently for
// tensor-core GEMM step x (independent of the plan-wide pair flag, so that a
// step's variant numbers never change): the launched form, merges included.  A
// step with a table of pattern groups uses it whenever 256 columns are allowed;
// its pattern-by-pattern variants are those narrower than a pattern's own tile.
std::vector<int> gemm_variants(const tn::Plan& P, const tn::Step& x) {
  std::vector<int> out;
  std::vector<tn::GemmForm> seen;
  for (int v = 0; v < kNumGemmVariants; ++v) {
    tn::GemmShape gs = tn::step_gemm_shape(P, x);
    gs.pair = kGemmVariants[v].pair;
    gs.tile_cap = kGemmVariants[v].cap;
    tn::GemmForm t = tn::gemm_form(gs, tn::kGemmSMs);
    if (t.grouped) {
      const bool paired = t.paired;
      gs.grp_fold = 0;
      t = tn::gemm_form(gs, tn::kGemmSMs);
      t.paired = paired;
    }
    bool dup = false;
    for (const tn::GemmForm& q : seen) dup |= q.bn == t.bn && q.fold == t.fold && q.paired == t.paired;
    if (!dup) {
      seen.push_back(t);
      out.push_back(v);
    }
  }
  return out;
}

// Whether a GEMM step of the plan runs on CTA pairs where they are allowed.
bool any_paired(const tn::Plan& P) {
  for (const tn::Step& x : P.steps) {
    if (x.kind != tn::ST_GEMM_TC) continue;
    tn::GemmShape gs = tn::step_gemm_shape(P, x);
    gs.pair = x.pair;
    if (tn::gemm_form(gs, tn::kGemmSMs).paired) return true;
  }
  return false;
}

int step_variant_count(const tn::Plan& P, const tn::Step& x) {
  if (x.kind == tn::ST_GEMM_TC) return (int)gemm_variants(P, x).size();
  if (x.kind == tn::ST_PERMUTE) return std::max<int>(1, (int)x.alts.size());
  if (x.kind == tn::ST_BPREP_TC) return x.alts.empty() ? 1 : 2;
  return 1;
}

void apply_step_variant(const tn::Plan& P, tn::Step& x, int v) {
  x.variant = v;
  if (x.kind == tn::ST_GEMM_TC) {
    const GemmVariant& g = kGemmVariants[gemm_variants(P, x)[(size_t)v]];
    x.tile_cap = g.cap;
    x.pair = g.pair;
  } else if (x.kind == tn::ST_PERMUTE && !x.alts.empty()) {
    tn::apply_perm_schedule(x, x.alts[(size_t)v]);
  }
}

// Captured graphs replay the launches they recorded: drop them, and give the
// plan a new serial so that the batch graph cache (keyed on it) misses too.
void drop_graphs(tn_plan_t* p) {
  for (auto& g : p->graphs) cudaGraphExecDestroy(g.exec);
  p->graphs.clear();
  p->serial = tn::next_serial();
}

}  // namespace

extern "C" int tn_plan_step_variants(const tn_plan_t* plan, int64_t i, int* n_variants, int* chosen) {
  if (!plan) return fail(TN_ERR_INVALID, "NULL plan");
  if (i < 0 || i >= (int64_t)plan->P.steps.size()) return fail(TN_ERR_INVALID, "step index out of range");
  const tn::Step& x = plan->P.steps[(size_t)i];
  if (n_variants) *n_variants = step_variant_count(plan->P, x);
  if (chosen) *chosen = x.variant;
  return TN_OK;
}

extern "C" int tn_plan_set_step_variant(tn_plan_t* plan, int64_t i, int variant) {
  if (!plan) return fail(TN_ERR_INVALID, "NULL plan");
  if (i < 0 || i >= (int64_t)plan->P.steps.size()) return fail(TN_ERR_INVALID, "step index out of range");
  tn::Step& x = plan->P.steps[(size_t)i];
  if (variant < 0 || variant >= step_variant_count(plan->P, x)) return fail(TN_ERR_INVALID, "variant out of range");
  if (x.variant != variant) {
    apply_step_variant(plan->P, x, variant);
    drop_graphs(plan);
  }
  return TN_OK;
}

extern "C" int tn_plan_tune_steps(tn_plan_t* plan, int reps, void* stream, double* default_ms, double* tuned_ms) {
  if (!plan) return fail(TN_ERR_INVALID, "NULL plan");
  if (!plan->on_device) return fail(TN_ERR_INVALID, "plan was made host_only");
  if (reps < 1 || reps > 64) return fail(TN_ERR_INVALID, "reps must be in [1, 64]");
  tn::Plan& P = plan->P;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t ns = (int64_t)P.steps.size();
  std::vector<int> start(ns), count(ns);
  int max_v = 1;
  for (int64_t i = 0; i < ns; ++i) {
    start[i] = P.steps[i].variant;
    count[i] = step_variant_count(P, P.steps[i]);
    max_v = std::max(max_v, count[i]);
  }
  tn_head_t* h = nullptr;
  int rc = tn_head_create(plan, nullptr, &h);
  if (rc) return rc;
  auto& ev = plan->prof_events;
  while (ev.size() < (size_t)(2 * (ns + 1))) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) {
      tn_head_free(h);
      return fail(TN_ERR_CUDA, "event creation failed");
    }
    ev.push_back(e);
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    tn_head_free(h);
    return fail(TN_ERR_CUDA, "event creation failed");
  }
  auto set_all = [&](const std::vector<int>& v) {
    for (int64_t i = 0; i < ns; ++i)
      if (P.steps[i].variant != v[i]) apply_step_variant(P, P.steps[i], v[i]);
  };
  // 1. per-step times of variant v of every step (v past a step's count: its default)
  std::vector<double> best_ms(ns, 1e300);
  std::vector<int> best_v(start);
  for (int v = 0; v < max_v && rc == TN_OK; ++v) {
    std::vector<int> cur(ns);
    for (int64_t i = 0; i < ns; ++i) cur[i] = v < count[i] ? v : 0;
    set_all(cur);
    for (int r = 0; r <= reps && rc == TN_OK; ++r) {
      rc = run_pass(plan, 0, h->H, st, ev.data());
      if (rc) break;
      const cudaError_t e = cudaEventSynchronize(ev[(size_t)(2 * ns + 1)]);
      if (e != cudaSuccess) {
        rc = fail(TN_ERR_CUDA, std::string("tuning pass: ") + cudaGetErrorString(e));
        break;
      }
      if (r == 0) continue;   // untimed
      for (int64_t i = 0; i < ns; ++i) {
        if (v >= count[i]) continue;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[(size_t)(2 * i)], ev[(size_t)(2 * i + 1)]);
        if (ms < best_ms[i]) {
          best_ms[i] = ms;
          best_v[i] = v;
        }
      }
    }
  }
  // 2. one pass of slice 0 each (a whole slice unless the plan has automatically
  // sliced edges) on the plan's own execution path, starting set against the
  // chosen one, alternating
  double t_start = 1e300, t_best = 1e300;
  for (int r = 0; r <= reps && rc == TN_OK; ++r)
    for (int which = 0; which < 2 && rc == TN_OK; ++which) {
      set_all(which == 0 ? start : best_v);
      cudaEventRecord(e0, st);
      rc = run_pass(plan, 0, h->H, st, nullptr);
      cudaEventRecord(e1, st);
      if (rc) break;
      const cudaError_t e = cudaEventSynchronize(e1);
      if (e != cudaSuccess) {
        rc = fail(TN_ERR_CUDA, std::string("tuning slice: ") + cudaGetErrorString(e));
        break;
      }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (r == 0) continue;   // untimed
      double& t = which == 0 ? t_start : t_best;
      t = std::min(t, (double)ms);
    }
  unsigned int word = 0;
  if (rc == TN_OK && cudaMemcpy(&word, plan->d_status, sizeof(word), cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = fail(TN_ERR_CUDA, "status read-back failed");
  if (rc == TN_OK && word) {
    cudaMemset(plan->d_status, 0, sizeof(word));
    rc = fail(TN_ERR_TIMEOUT, "a bounded device wait gave up while tuning (status " + std::to_string(word) + ")");
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  tn_head_free(h);
  const bool keep = rc == TN_OK && t_best < t_start;
  set_all(keep ? best_v : start);
  drop_graphs(plan);
  if (rc) return rc;
  plan->tune_default_ms = t_start;
  plan->tune_tuned_ms = t_best;
  if (default_ms) *default_ms = t_start;
  if (tuned_ms) *tuned_ms = t_best;
  return TN_OK;
}

extern "C" int tn_contract_slices(tn_plan_t* plan, tn_range r, tn_head_t* head, void* stream) {
  int rc = check_range(plan, r, head);
  if (rc) return rc;
  if (r.begin == r.end) return TN_OK;
  cudaStream_t st = (cudaStream_t)stream;
  int64_t done_end = r.end;
  rc = tn::enqueue_slices(plan, r, head->H, st, &done_end);
  if (rc) {
    // the whole slices enqueued before the failure stay recorded (a retry of
    // the rest is accepted); a slice left partly accumulated invalidates H
    if (done_end < 0) {
      head->invalid = true;
      g_err += "; the head holds part of a slice and is invalid until tn_head_reset";
    } else {
      mark_done(head, {r.begin, done_end});
      g_err += "; slices [" + std::to_string(r.begin) + ", " + std::to_string(done_end) + ") were accumulated";
    }
    return rc;
  }
  mark_done(head, r);
  if (tn::fault_status())   // injected: as if a bounded wait of this contraction had given up
    CUDA_TRY(cudaMemsetAsync(plan->d_status, 1, sizeof(unsigned int), st));
  return TN_OK;
}

// ---------------------------------------------------------- CUDA graphs

// Branch streams of this thread (and the stream that captures): one set, reused.
static int branch_streams(int n, std::vector<cudaStream_t>** out) {
  static thread_local std::vector<cudaStream_t> streams;
  while ((int)streams.size() < n) {
    cudaStream_t st;
    CUDA_TRY(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    streams.push_back(st);
  }
  *out = &streams;
  return TN_OK;
}

// Enqueue the slices of every (plan, head) item, item i on branch stream
// 1 + branch_of[i], between a fork from `main` and a join into it (events).
static int fork_items(const std::vector<tn_plan_t*>& plans, const std::vector<tn_range>& ranges,
                      const std::vector<tn_head_t*>& heads, const std::vector<int>& branch_of, int n_branches,
                      cudaStream_t main, const std::vector<cudaStream_t>& streams) {
  static thread_local std::vector<cudaEvent_t> ev;
  while ((int)ev.size() < n_branches + 1) {
    cudaEvent_t e;
    CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    ev.push_back(e);
  }
  int rc = TN_OK;
  cudaError_t ce = cudaEventRecord(ev[0], main);
  for (int b = 0; b < n_branches && ce == cudaSuccess; ++b) ce = cudaStreamWaitEvent(streams[1 + b], ev[0], 0);
  if (ce != cudaSuccess) rc = fail(TN_ERR_CUDA, std::string("fork: ") + cudaGetErrorString(ce));
  for (size_t i = 0; i < plans.size() && rc == TN_OK; ++i)
    rc = run_passes(plans[i], ranges[i].begin << plans[i]->P.n_internal, ranges[i].end << plans[i]->P.n_internal,
                    heads[i]->H, streams[1 + branch_of[i]]);
  // joined on failure too, so that what was enqueued stays ordered before the caller's next work
  for (int b = 0; b < n_branches; ++b) {
    ce = cudaEventRecord(ev[1 + b], streams[1 + b]);
    if (ce == cudaSuccess) ce = cudaStreamWaitEvent(main, ev[1 + b], 0);
    if (rc == TN_OK && ce != cudaSuccess) rc = fail(TN_ERR_CUDA, std::string("join: ") + cudaGetErrorString(ce));
  }
  return rc;
}

// The same, captured into an executable graph.
static int capture_items(const std::vector<tn_plan_t*>& plans, const std::vector<tn_range>& ranges,
                         const std::vector<tn_head_t*>& heads, const std::vector<int>& branch_of, int n_branches,
                         cudaGraphExec_t* exec_out) {
  std::vector<cudaStream_t>* streams = nullptr;
  if (int rc = branch_streams(n_branches + 1, &streams)) return rc;
  cudaStream_t main = (*streams)[0];
  CUDA_TRY(cudaStreamBeginCapture(main, cudaStreamCaptureModeThreadLocal));
  int rc = fork_items(plans, ranges, heads, branch_of, n_branches, main, *streams);
  cudaGraph_t graph = nullptr;
  cudaError_t ce = cudaStreamEndCapture(main, &graph);
  if (rc == TN_OK && ce != cudaSuccess) rc = fail(TN_ERR_CUDA, std::string("end capture: ") + cudaGetErrorString(ce));
  if (rc == TN_OK) {
    ce = cudaGraphInstantiate(exec_out, graph, 0);
    if (ce != cudaSuccess) rc = fail(TN_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(ce));
  }
  if (graph) cudaGraphDestroy(graph);
  cudaGetLastError();
  return rc;
}

extern "C" int tn_contract_slices_graph(tn_plan_t* plan, tn_range r, tn_head_t* head, void* stream) {
  int rc = check_range(plan, r, head);
  if (rc) return rc;
  if (r.begin == r.end) return TN_OK;
  GraphEntry* hit = nullptr;
  for (auto& g : plan->graphs)
    if (g.begin == r.begin && g.end == r.end && g.H == (void*)head->H) hit = &g;
  if (!hit) {
    GraphEntry g;
    g.begin = r.begin;
    g.end = r.end;
    g.H = head->H;
    rc = capture_items({plan}, {r}, {head}, {0}, 1, &g.exec);
    if (rc) return rc;
    // bounded cache: the least recently replayed graph goes (an in-flight
    // executable graph is freed by CUDA once its launch completes)
    constexpr size_t kGraphCache = 16;
    if (plan->graphs.size() >= kGraphCache) {
      auto lru = std::min_element(plan->graphs.begin(), plan->graphs.end(),
                                  [](const GraphEntry& a, const GraphEntry& b) { return a.last_use < b.last_use; });
      cudaGraphExecDestroy(lru->exec);
      plan->graphs.erase(lru);
    }
    plan->graphs.push_back(g);
    hit = &plan->graphs.back();
  }
  hit->last_use = ++plan->graph_clock;
  CUDA_TRY(cudaGraphLaunch(hit->exec, (cudaStream_t)stream));
  mark_done(head, r);
  return TN_OK;
}

extern "C" int tn_contract_batch(tn_plan_t* const* plans, const tn_range* ranges, tn_head_t* const* heads, int n,
                                 void* stream) {
  if (n < 0 || (n > 0 && (!plans || !ranges || !heads))) return fail(TN_ERR_INVALID, "bad batch arrays");
  if (n == 0) return TN_OK;
  std::vector<tn_plan_t*> P(plans, plans + n);
  std::vector<tn_range> R(ranges, ranges + n);
  std::vector<tn_head_t*> Hs(heads, heads + n);
  std::vector<int> branch(n);
  std::map<tn_plan_t*, int> branch_of_plan;   // items of one plan share its arena: same branch
  std::map<tn_head_t*, int> head_seen;
  for (int i = 0; i < n; ++i) {
    int rc = check_range(P[i], R[i], Hs[i]);
    if (rc) return rc;
    if (head_seen.count(Hs[i])) return fail(TN_ERR_INVALID, "a head appears twice in one batch");
    head_seen[Hs[i]] = i;
    auto it = branch_of_plan.find(P[i]);
    if (it == branch_of_plan.end()) it = branch_of_plan.emplace(P[i], (int)branch_of_plan.size()).first;
    branch[i] = it->second;
  }
  const int n_branches = std::min<int>((int)branch_of_plan.size(), 32);
  for (int i = 0; i < n; ++i) branch[i] %= n_branches;
  // A batch is known by its handles' serials (never reused) and ranges.  The
  // first time one is seen its launches may go straight to the branch streams
  // (below), which takes less host time than capturing and instantiating a graph;
  // from the second time on a captured graph is replayed.  Per thread, the graphs
  // of the kBatchGraphs batches replayed last are kept, and the keys of the
  // kBatchSeen seen last.
  struct Batch {
    std::vector<uint64_t> p, h;
    std::vector<int64_t> r;
    cudaGraphExec_t exec = nullptr;
    uint64_t last_use = 0;
    bool same(const Batch& o) const { return p == o.p && h == o.h && r == o.r; }
  };
  constexpr size_t kBatchGraphs = 8, kBatchSeen = 32;
  static thread_local std::vector<Batch> known;
  static thread_local uint64_t clock = 0;
  Batch key;
  for (auto* x : P) key.p.push_back(x->serial);
  for (auto* x : Hs) key.h.push_back(x->serial);
  for (auto& x : R) { key.r.push_back(x.begin); key.r.push_back(x.end); }
  auto it = std::find_if(known.begin(), known.end(), [&](const Batch& b) { return b.same(key); });
  const bool seen = it != known.end();
  if (!seen) {
    if (known.size() >= kBatchSeen) {
      auto lru = std::min_element(known.begin(), known.end(),
                                  [](const Batch& a, const Batch& b) { return a.last_use < b.last_use; });
      if (lru->exec) cudaGraphExecDestroy(lru->exec);
      known.erase(lru);
    }
    known.push_back(key);
    it = std::prev(known.end());
  }
  it->last_use = ++clock;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  CUDA_TRY(cudaStreamIsCapturing((cudaStream_t)stream, &cap));
  // Launched directly where a failure on the way can be undone: heads that are
  // still zero and that nobody else can write.  Otherwise, and into a capture of
  // the caller's, only as a graph, which runs whole or not at all.
  bool undoable = cap == cudaStreamCaptureStatusNone;
  for (int i = 0; i < n; ++i)
    undoable = undoable && (R[i].begin == R[i].end || (Hs[i]->owns && !Hs[i]->exposed && Hs[i]->done.empty()));
  if (!seen && undoable) {
    std::vector<cudaStream_t>* streams = nullptr;
    if (int rc = branch_streams(n_branches + 1, &streams)) return rc;
    if (const int rc = fork_items(P, R, Hs, branch, n_branches, (cudaStream_t)stream, *streams)) {
      for (int i = 0; i < n; ++i)
        if (R[i].begin < R[i].end && cudaMemsetAsync(Hs[i]->H, 0, (size_t)head_elems(Hs[i]) * sizeof(double2),
                                                     (cudaStream_t)stream) != cudaSuccess) {
          cudaGetLastError();
          Hs[i]->invalid = true;
        }
      return rc;
    }
  } else {
    if (!it->exec) {
      size_t graphs = 0;
      for (const Batch& b : known) graphs += b.exec != nullptr;
      if (graphs >= kBatchGraphs) {
        auto lru = known.end();
        for (auto b = known.begin(); b != known.end(); ++b)
          if (b->exec && (lru == known.end() || b->last_use < lru->last_use)) lru = b;
        cudaGraphExecDestroy(lru->exec);
        lru->exec = nullptr;
      }
      const int rc = capture_items(P, R, Hs, branch, n_branches, &it->exec);
      if (rc) {
        it->exec = nullptr;
        return rc;
      }
    }
    CUDA_TRY(cudaGraphLaunch(it->exec, (cudaStream_t)stream));
  }
  for (int i = 0; i < n; ++i) mark_done(Hs[i], R[i]);
  return TN_OK;
}

// ------------------------------------------------------ amplitudes, sampling

static int ensure_stage(tn_head* h, size_t bytes) {
  if (h->stage_bytes >= bytes) return TN_OK;
  cudaFree(h->d_stage);
  h->d_stage = nullptr;
  h->stage_bytes = 0;
  cudaError_t e = tn::device_malloc(&h->d_stage, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(TN_ERR_OOM, "staging buffer allocation failed");
  }
  h->stage_bytes = bytes;
  return TN_OK;
}

// A buffer that kernels can use as it is: device or managed memory, or pinned
// host memory, which GB300 reads and writes over NVLink-C2C without a copy, if
// it starts on the `align` bytes that the kernel moves at a time.  Other buffers
// go through the head's staging buffer.
static bool kernel_ptr(const void* p, size_t align) {
  if (!tn::kernel_aligned(p, align)) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged ||
         (a.type == cudaMemoryTypeHost && a.devicePointer == p);
}

extern "C" int tn_amplitudes(tn_head_t* h, const uint64_t* bitstrings, int64_t n, void* out, int dtype, void* stream) {
  if (!h || (n > 0 && (!bitstrings || !out))) return fail(TN_ERR_INVALID, "NULL argument");
  if (n < 0) return fail(TN_ERR_INVALID, "n < 0");
  if (dtype != TN_C64 && dtype != TN_C128) return fail(TN_ERR_INVALID, "dtype must be TN_C64 or TN_C128");
  if (h->invalid) return fail(TN_ERR_INVALID, "head is invalid after a failed or timed-out contraction");
  if (n == 0) return TN_OK;
  tn_plan_t* p = h->plan;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t esz = dtype == TN_C128 ? 16 : 8;
  // bitstrings that the output covers are copied before any of it is written
  const bool dev_in =
      kernel_ptr(bitstrings, 8) && !tn::ranges_overlap(bitstrings, (size_t)n * 8, out, (size_t)n * esz);
  const bool dev_out = kernel_ptr(out, esz);
  size_t need = 0;
  if (!dev_in) need += (size_t)n * 8;
  size_t out_off = (need + 255) / 256 * 256;
  if (!dev_out) need = out_off + (size_t)n * esz;
  if (need) {
    int rc = ensure_stage(h, need);
    if (rc) return rc;
  }
  ScratchLease lease(st);
  if (int rc = lease.take(0)) return rc;
  const uint64_t* d_bits = bitstrings;
  if (!dev_in) {
    CUDA_TRY(cudaMemcpyAsync(h->d_stage, bitstrings, (size_t)n * 8, cudaMemcpyDefault, st));
    d_bits = (const uint64_t*)h->d_stage;
  }
  void* d_out = dev_out ? out : (void*)((char*)h->d_stage + out_off);
  CUDA_TRY(tn::launch_amplitudes(h->H, (int)p->P.open_qubits.size(), p->d_keys, p->d_key_groups, p->n_keys,
                                 p->P.tail_mask, p->d_open, d_bits, n, d_out, dtype == TN_C128 ? 1 : 0,
                                 &lease.c.rep->missing, st, nullptr, 1, lease.c.rep, p->d_status));
  if (!dev_out) CUDA_TRY(cudaMemcpyAsync(out, d_out, (size_t)n * esz, cudaMemcpyDefault, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  const tn::HeadReport rep = lease.done();
  if (int rc = tn::report_status(h, rep.word, st)) return rc;
  if (rep.missing != ~0ULL)
    return fail(TN_ERR_NOT_IN_STATE, "bitstring " + std::to_string(rep.missing) + " has a tail that is not a group");
  return TN_OK;
}

extern "C" int tn_xeb(tn_head_t* h, const uint64_t* samples, int64_t n, double* linear, double* log_xeb,
                      void* stream) {
  if (!h || (n > 0 && !samples)) return fail(TN_ERR_INVALID, "NULL argument");
  if (n < 1) return fail(TN_ERR_INVALID, "n must be >= 1");
  if (h->invalid) return fail(TN_ERR_INVALID, "head is invalid after a failed or timed-out contraction");
  tn_plan_t* p = h->plan;
  cudaStream_t st = (cudaStream_t)stream;
  const uint64_t* d_bits = samples;
  if (!kernel_ptr(samples, 8)) {
    if (int rc = ensure_stage(h, (size_t)n * 8)) return rc;
    CUDA_TRY(cudaMemcpyAsync(h->d_stage, samples, (size_t)n * 8, cudaMemcpyDefault, st));
    d_bits = (const uint64_t*)h->d_stage;
  }
  ScratchLease lease(st);
  if (int rc = lease.take(0)) return rc;
  CUDA_TRY(tn::launch_xeb(h->H, (int)p->P.open_qubits.size(), p->d_keys, p->d_key_groups, p->n_keys, p->P.tail_mask,
                          p->d_open, d_bits, n, lease.c.part, lease.c.rep, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  const tn::HeadReport rep = lease.done();
  if (rep.missing != ~0ULL)
    return fail(TN_ERR_NOT_IN_STATE, "sample " + std::to_string(rep.missing) + " has a tail that is not a group");
  const int nq = p->P.n_qubits;
  if (linear) *linear = std::ldexp(rep.sum[0] / (double)n, nq) - 1.0;
  if (log_xeb) *log_xeb = nq * std::log(2.0) + 0.57721566490153286 + rep.sum[1] / (double)n;
  return TN_OK;
}

extern "C" int tn_head_norm(tn_head_t* h, double* norm, double* group_norms, void* stream) {
  if (!h) return fail(TN_ERR_INVALID, "NULL head");
  if (h->invalid) return fail(TN_ERR_INVALID, "head is invalid after a failed or timed-out contraction");
  tn_plan_t* p = h->plan;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t L = (int64_t)p->P.tails_raw.size();
  // the group norms of up to 8,192 groups come back through mapped memory, as
  // the norm does; more by a copy (one block writes them)
  const bool mapped = group_norms && L <= 8192;
  ScratchLease lease(st);
  if (int rc = lease.take(0, mapped ? (size_t)L * sizeof(double) : 0)) return rc;
  CUDA_TRY(tn::launch_group_norms(h->H, L, (int)p->P.open_qubits.size(), h->d_Z, nullptr, lease.c.part, st,
                                  lease.c.rep, p->d_status, mapped ? (double*)lease.c.host : nullptr));
  if (group_norms && !mapped)
    CUDA_TRY(cudaMemcpyAsync(group_norms, h->d_Z, (size_t)L * sizeof(double), cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  const tn::HeadReport rep = lease.done();
  if (norm) *norm = rep.sum[0];
  if (mapped) std::memcpy(group_norms, lease.c.host, (size_t)L * sizeof(double));
  return tn::report_status(h, rep.word, st);
}

static int sample_impl(tn_head_t* h, int64_t n, double target_fidelity, uint64_t seed, int method, int64_t param,
                       uint64_t* out, void* stream);

extern "C" int tn_sample(tn_head_t* h, int64_t n, double target_fidelity, uint64_t seed, uint64_t* out, void* stream) {
  return sample_impl(h, n, target_fidelity, seed, TN_SAMPLE_EXACT, 0, out, stream);
}

extern "C" int tn_sample_ex(tn_head_t* h, int64_t n, double target_fidelity, uint64_t seed, int method,
                            int64_t param, uint64_t* out, void* stream) {
  return sample_impl(h, n, target_fidelity, seed, method, param, out, stream);
}

static int sample_impl(tn_head_t* h, int64_t n, double target_fidelity, uint64_t seed, int method, int64_t param,
                       uint64_t* out, void* stream) {
  if (!h || (n > 0 && !out)) return fail(TN_ERR_INVALID, "NULL argument");
  if (method < TN_SAMPLE_EXACT || method > TN_SAMPLE_FRUGAL) return fail(TN_ERR_INVALID, "unknown sampling method");
  const int64_t l = 1LL << h->plan->P.open_qubits.size();
  if (method == TN_SAMPLE_METROPOLIS && param == 0) param = l;
  if (method == TN_SAMPLE_FRUGAL && param == 0) param = 10;
  if (param < 0 || (method == TN_SAMPLE_METROPOLIS && param > (1LL << 32)) ||
      (method == TN_SAMPLE_FRUGAL && param > (1LL << 20)))
    return fail(TN_ERR_INVALID, "sampling parameter out of range");
  if (n < 0) return fail(TN_ERR_INVALID, "n < 0");
  if (h->invalid) return fail(TN_ERR_INVALID, "head is invalid after a failed or timed-out contraction");
  if (n == 0) return TN_OK;
  tn_plan_t* p = h->plan;
  double f_head = 0.0;
  tn_head_fidelity(h, &f_head, nullptr);
  if (target_fidelity > f_head && target_fidelity > 0.0 && f_head > 0.0 && target_fidelity - f_head > 1e-15)
    return fail(TN_ERR_INVALID, "target fidelity above the head's estimated fidelity");
  double mix = 0.0;
  if (target_fidelity > 0.0 && f_head > 0.0 && target_fidelity < f_head) mix = 1.0 - target_fidelity / f_head;
  cudaStream_t st = (cudaStream_t)stream;
  const bool dev_out = kernel_ptr(out, 8);
  uint64_t* d_out = out;
  if (!dev_out) {
    int rc = ensure_stage(h, (size_t)n * 8);
    if (rc) return rc;
    d_out = (uint64_t*)h->d_stage;
  }
  ScratchLease lease(st);
  const int n_open = (int)p->P.open_qubits.size();
  int64_t groups = tn::sample_groups((int64_t)p->P.tails_raw.size(), n_open, n, method);
  // with memory short, the prefix sums of fewer groups at a time
  while (int rc = lease.take(8 * tn::sample_scratch_doubles(n_open, groups))) {
    if (rc != TN_ERR_OOM || groups <= 1) return rc;
    groups = (groups + 1) / 2;
  }
  tn::SampleParams sp;
  sp.H = h->H;
  sp.L = (int64_t)p->P.tails_raw.size();
  sp.h = (int)p->P.open_qubits.size();
  sp.tails = p->d_tails;
  sp.open_mask = p->P.open_mask;
  sp.open_q = p->d_open;
  sp.n_qubits = p->P.n_qubits;
  sp.n = n;
  sp.mix = mix;
  sp.seed = seed;
  sp.out = d_out;
  sp.method = method;
  sp.param = param;
  sp.carry = (double*)lease.c.buf;
  sp.carry_groups = groups;
  sp.rep = lease.c.rep;
  sp.plan_status = p->d_status;
  CUDA_TRY(tn::launch_sample(sp, st));
  if (!dev_out) CUDA_TRY(cudaMemcpyAsync(out, d_out, (size_t)n * 8, cudaMemcpyDefault, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  return tn::report_status(h, lease.done().word, st);
}

namespace tn {
int enqueue_slices(tn_plan_t* plan, tn_range r, double2* H, cudaStream_t stream, int64_t* done_end) {
  const int ni = plan->P.n_internal;
  int64_t q = 0;
  const int rc = run_passes(plan, r.begin << ni, r.end << ni, H, stream, &q);
  if (done_end) *done_end = q & ((1LL << ni) - 1) ? -1 : q >> ni;   // -1: a slice is partly accumulated
  return rc;
}
int check_slice_range(tn_plan_t* plan, tn_range r, tn_head_t* head) { return check_range(plan, r, head); }
void mark_slices_done(tn_head_t* head, tn_range r) { mark_done(head, r); }
}  // namespace tn

// ------------------------------------------------------- standalone GEMM

extern "C" int tn_gemm_c64(int engine, const void* A, const void* B, void* C, int64_t M, int64_t N, int64_t K,
                           int64_t PA, int64_t PB, int64_t PC, const int32_t* mapA, const int32_t* mapB, int pair,
                           void* stream) {
  if (engine == TN_GEMM_AUTO) engine = TN_GEMM_TC_3XTF32;
  if (engine < TN_GEMM_TC_3XTF32 || engine > TN_GEMM_TC_FP16X3) return fail(TN_ERR_INVALID, "unknown gemm engine");
  if (!A || !B || !C) return fail(TN_ERR_INVALID, "NULL operand");
  auto pow2 = [](int64_t x) { return x >= 1 && (x & (x - 1)) == 0; };
  if (!pow2(M) || !pow2(N) || !pow2(K)) return fail(TN_ERR_INVALID, "M, N and K must be powers of two");
  if (PA < 1 || PB < 1 || PC < 1) return fail(TN_ERR_INVALID, "pattern counts must be >= 1");
  if (M * K > (1LL << 32) || K * N > (1LL << 32) || M * N > (1LL << 32))
    return fail(TN_ERR_INVALID, "operand above 2^32 elements");
  const bool simt = engine == TN_GEMM_SIMT_FP32;
  int nk = 0, nn = 0, nmk = 0;
  while ((1LL << nk) < K) ++nk;
  while ((1LL << nn) < N) ++nn;
  while ((1LL << nmk) < M * K) ++nmk;
  if (!simt && nk < 1) return fail(TN_ERR_INVALID, "tensor-core engines need K >= 2");
  // like the planner: 16-bit operands need K >= 4 (16-byte rows); K = 2 uses tf32
  const int h16 = simt ? 0 : nk >= 2 ? (engine == TN_GEMM_TC_BF16X3 ? 1 : engine == TN_GEMM_TC_FP16X3 ? 2 : 0) : 0;
  // pattern maps: a table of PC entries, or identity (P == PC) / all zero (P == 1)
  int mode[2];
  std::vector<uint32_t> maps[2];
  const int32_t* user[2] = {mapA, mapB};
  const int64_t PX[2] = {PA, PB};
  for (int x = 0; x < 2; ++x) {
    if (user[x]) {
      mode[x] = 2;
      for (int64_t p = 0; p < PC; ++p) {
        if (user[x][p] < 0 || user[x][p] >= PX[x]) return fail(TN_ERR_INVALID, "pattern map entry out of range");
        maps[x].push_back((uint32_t)user[x][p]);
      }
    } else if (PX[x] == PC) {
      mode[x] = 0;
    } else if (PX[x] == 1) {
      mode[x] = 1;
    } else {
      return fail(TN_ERR_INVALID, "a pattern count differs from PC and no map is given");
    }
  }
  cudaStream_t st = (cudaStream_t)stream;
  // An operand that C covers is read before any of C is written: the tensor-core
  // path always reads planes of both, the CUDA-core one a copy of that operand.
  const size_t a_in = (size_t)(PA * M * K) * 8, b_in = (size_t)(PB * K * N) * 8, c_out = (size_t)(PC * M * N) * 8;
  const bool over_a = tn::ranges_overlap(A, a_in, C, c_out), over_b = tn::ranges_overlap(B, b_in, C, c_out);
  // The direct kernel where it is modelled faster than the three launches
  // below (as the planner chooses; C is row-major, so its rows are N and X is
  // B), and its operands, which it reads where they lie, are apart from C.
  // pair != 0 asks for the GEMM kernels themselves.
  if (!simt && pair == 0 && !over_a && !over_b && nmk <= 31 && nk + nn <= 31) {
    int nm = nmk - nk;
    std::vector<int> xr, xk, yk, yc;
    for (int j = 0; j < nn; ++j) xr.push_back(j);
    for (int q = 0; q < nk; ++q) { xk.push_back(nn + q); yk.push_back(q); }
    for (int j = 0; j < nm; ++j) yc.push_back(nk + j);
    tn::DirectPlan best;
    for (int fold = 0; fold < 2; ++fold) {
      if (fold && (PC == 1 || mode[1] != 1)) continue;
      tn::DirectShape ds;
      ds.nr = nn;
      ds.nk = nk;
      ds.nc = nm;
      ds.xr = xr.data();
      ds.xk = xk.data();
      ds.yk = yk.data();
      ds.yc = yc.data();
      ds.PC = PC;
      ds.x_shared = mode[1] == 1;
      ds.bf16 = h16 == 1;
      ds.x_elems = (double)PB * (double)(K * N);
      ds.y_elems = (double)PA * (double)(M * K);
      const tn::DirectPlan d = tn::plan_direct(ds, fold != 0);
      if (d.seconds < best.seconds) best = d;
    }
    tn::GemmShape gs;
    gs.M = M;
    gs.N = N;
    gs.PA = PA;
    gs.PB = PB;
    gs.PC = PC;
    gs.mapA_mode = mode[0];
    gs.mapB_mode = mode[1];
    gs.h16 = h16;
    if (best.seconds < tn::tc_seconds(tn::gemm_form(gs, tn::kGemmSMs), nk, (double)PA * (double)(M * K),
                                      (double)PB * (double)(K * N), (double)PC * (double)(M * N), h16 != 0)) {
      const size_t n_map = maps[0].size() + maps[1].size();
      ScratchLease lease(st);
      if (int rc = lease.take(n_map * sizeof(uint32_t), n_map * sizeof(uint32_t))) return rc;
      uint32_t* d_maps = (uint32_t*)lease.c.buf;
      if (n_map) {
        std::copy(maps[0].begin(), maps[0].end(), (uint32_t*)lease.c.host);
        std::copy(maps[1].begin(), maps[1].end(), (uint32_t*)lease.c.host + maps[0].size());
        CUDA_TRY(cudaMemcpyAsync(d_maps, lease.c.host, n_map * sizeof(uint32_t), cudaMemcpyHostToDevice, st));
      }
      tn::DirectParams dp{};
      tn::direct_fill(best, PC, dp);
      dp.X = (const float2*)B;
      dp.Y = (const float2*)A;
      dp.C = (float2*)C;
      dp.x_pstride = K * N;
      dp.y_pstride = M * K;
      dp.c_pstride = M * N;
      dp.mapX = d_maps + maps[0].size();
      dp.mapY = d_maps;
      dp.mapX_mode = mode[1];
      dp.mapY_mode = mode[0];
      dp.bf16 = h16 == 1;
      dp.vec = (uintptr_t)C % 16 == 0;
      dp.amax = nullptr;
      cudaError_t e = tn::launch_direct(dp, best.config, st, true);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("tn_gemm_c64: ") + cudaGetErrorString(e));
      lease.done();
      return TN_OK;
    }
  }
  // scratch: scale slots, pattern maps, split A planes, prepared B
  const int64_t es = h16 ? 2 : 4;
  const size_t n_map = maps[0].size() + maps[1].size();
  const size_t map_off = 256, a_off = (map_off + n_map * sizeof(uint32_t) + 1023) / 1024 * 1024;
  const size_t a_bytes = simt ? (over_a ? a_in : 0) : (size_t)(2 * PA * M * (2 * K) * es);
  const size_t b_off = a_off + (a_bytes + 1023) / 1024 * 1024;
  const size_t b_bytes = simt ? (over_b ? b_in : 0) : (size_t)(2 * PB * (2 * N) * (2 * K) * es);
  ScratchLease lease(st);
  if (int rc = lease.take(b_off + b_bytes, n_map * sizeof(uint32_t))) return rc;
  char* d = (char*)lease.c.buf;
  unsigned int* d_scale = (unsigned int*)d;   // [0] max of A, [1] max of B
  uint32_t* d_maps = (uint32_t*)(d + map_off);
  cudaError_t e = cudaSuccess;
  if (n_map) {
    std::copy(maps[0].begin(), maps[0].end(), (uint32_t*)lease.c.host);
    std::copy(maps[1].begin(), maps[1].end(), (uint32_t*)lease.c.host + maps[0].size());
    e = cudaMemcpyAsync(d_maps, lease.c.host, n_map * sizeof(uint32_t), cudaMemcpyHostToDevice, st);
  }
  tn::GemmParams gp;
  if (!simt) {
    if (e == cudaSuccess && h16 == 2) e = cudaMemsetAsync(d_scale, 0, 2 * sizeof(unsigned int), st);
    tn::GemmOperands op{(const float2*)A, (const float2*)B, d + a_off, d + b_off, PA * M * K, K, N, PB, h16, d_scale};
    if (e == cudaSuccess) e = tn::launch_gemm_operands(op, st);
  } else {
    if (e == cudaSuccess && over_a) e = cudaMemcpyAsync(d + a_off, A, a_in, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && over_b) e = cudaMemcpyAsync(d + b_off, B, b_in, cudaMemcpyDeviceToDevice, st);
  }
  if (e == cudaSuccess) {
    // the CUDA-core GEMM reads row-major operands as they are
    gp.A = simt && !over_a ? (const float2*)A : (const float2*)(d + a_off);
    gp.B = simt && !over_b ? B : (const void*)(d + b_off);
    gp.C = (float2*)C;
    gp.M = M;
    gp.N = N;
    gp.K = K;
    gp.PA = PA;
    gp.PB = PB;
    gp.PC = PC;
    gp.mapA = d_maps;
    gp.mapB = d_maps + maps[0].size();
    gp.mapA_mode = mode[0];
    gp.mapB_mode = mode[1];
    gp.h16 = h16;
    gp.scaleA = d_scale;
    gp.scaleB = d_scale + 1;
    gp.amax = nullptr;
    gp.pair = pair < 0 ? -1 : 0;
    gp.prepare = 1;
    e = simt ? tn::launch_gemm_simt(gp, st) : tn::launch_gemm_tc(gp, &lease.c.rep->word, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(TN_ERR_CUDA, std::string("tn_gemm_c64: ") + cudaGetErrorString(e));
  if (lease.done().word) return fail(TN_ERR_TIMEOUT, "tn_gemm_c64: a bounded device wait gave up");
  return TN_OK;
}

extern "C" int tn_plan_autotune(const tn_circuit* circuit, const tn_open_spec* open_spec, const tn_edge* sliced_edges,
                                int n_edges, const tn_plan_opts* opts, int n_candidates, void* stream,
                                tn_plan_t** out) {
  if (!out) return fail(TN_ERR_INVALID, "out is NULL");
  *out = nullptr;
  if (n_candidates < 1 || n_candidates > 64) return fail(TN_ERR_INVALID, "n_candidates must be in [1, 64]");
  tn_plan_opts o{};
  if (opts) o = *opts;
  if (o.host_only) return fail(TN_ERR_INVALID, "autotuning needs the device");
  const uint64_t seed0 = o.order_seed ? o.order_seed : 1;
  cudaStream_t st = (cudaStream_t)stream;
  tn_plan_t* best = nullptr;
  double best_ms = 1e300;
  int distinct = 0;
  std::vector<std::vector<std::pair<int, int>>> seen;
  cudaEvent_t e0, e1;
  CUDA_TRY(cudaEventCreate(&e0));
  CUDA_TRY(cudaEventCreate(&e1));
  int last_rc = TN_OK;
  for (int c = 0; c < n_candidates; ++c) {
    o.order_seed = seed0 + (uint64_t)c;
    tn_plan_opts ho = o;
    ho.host_only = 1;
    tn_plan_t* hp = nullptr;
    int rc = tn_plan(circuit, open_spec, sliced_edges, n_edges, nullptr, 0, &ho, &hp);
    if (rc) { last_rc = rc; continue; }
    bool dup = false;
    for (auto& s_ : seen) dup |= s_ == hp->P.order;
    if (dup) { tn_plan_free(hp); continue; }
    seen.push_back(hp->P.order);
    // upload this candidate (its edges include any automatically sliced ones)
    tn_plan_t* p = hp;
    rc = plan_upload(p);
    if (rc) { plan_release(p); last_rc = rc; continue; }
    ++distinct;
    tn_head_t* h = nullptr;
    rc = tn_head_create(p, nullptr, &h);
    double ms = 1e300;
    if (rc == TN_OK) {
      // where a GEMM runs on CTA pairs, time those and the one-CTA tiles and
      // keep the faster (unless the caller turned pairs off)
      const bool both = o.gemm_pair == 0 && any_paired(p->P);
      int best_pair = p->P.gemm_pair;
      for (int v = 0; v < (both ? 2 : 1) && rc == TN_OK; ++v) {
        if (both) p->P.gemm_pair = v == 0 ? 0 : -1;
        rc = run_slice(p, 0, h->H, st);   // untimed
        if (rc != TN_OK) break;
        cudaEventRecord(e0, st);
        rc = run_slice(p, 0, h->H, st);
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) == cudaSuccess) {
          float f = 0.f;
          cudaEventElapsedTime(&f, e0, e1);
          if (f < ms) {
            ms = f;
            best_pair = p->P.gemm_pair;
          }
        }
      }
      p->P.gemm_pair = best_pair;
      tn_head_free(h);
    }
    if (rc == TN_OK && ms < best_ms) {
      if (best) tn_plan_free(best);
      best = p;
      best_ms = ms;
    } else {
      tn_plan_free(p);
    }
    if (rc) last_rc = rc;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!best) return last_rc ? last_rc : fail(TN_ERR_OOM, "no candidate plan could be built");
  best->measured_slice_ms = best_ms;
  best->autotune_candidates = distinct;
  const double passes = std::ldexp(1.0, best->P.n_internal);
  if (o.tune_steps > 0 || (o.tune_steps == 0 && best_ms / passes <= 1000.0)) {
    double t0 = 0, t1 = 0;
    const int rc = tn_plan_tune_steps(best, o.tune_steps > 0 ? o.tune_steps : 3, stream, &t0, &t1);
    if (rc) {
      tn_plan_free(best);
      return rc;
    }
    // the tuner times one pass: a slice is 2^n_internal of them
    best->measured_slice_ms = best->P.n_internal == 0 ? std::min(t0, t1) : best_ms * std::min(t0, t1) / t0;
  }
  *out = best;
  return TN_OK;
}
