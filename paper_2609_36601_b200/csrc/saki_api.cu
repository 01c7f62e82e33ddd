// C ABI of the SAKI routing library: host-side validation, kernel selection,
// the proposal-sampling utility, the block-verification resolve and the
// host-buffer convenience entry.  See include/saki.h for the contract.
#include "saki_common.cuh"
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <iterator>
#include <map>
#include <mutex>
#include <utility>
#include <vector>
#include <algorithm>

namespace saki {

static thread_local char g_err[512] = "";
static std::atomic<uint64_t> g_launches{0};
static std::atomic<int> g_kernel{0};
static std::atomic<int> g_spec_early_out{1};
static std::atomic<int> g_phase_clock{0};
static std::atomic<long long> g_wait_limit{0};
static thread_local int g_last_kernel = 0;

static int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}
static int cuda_fail(cudaError_t e, const char* what) {
  return fail(SAKI_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// device-resident count of flagged rows (one per device that loads the library)
__device__ unsigned long long g_flagged_rows = 0ull;

static int device_ready(unsigned long long** flagged) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(SAKI_ERR_UNSUPPORTED, "no CUDA device: %s", cudaGetErrorString(e));
  // looked up once per device (a call of a few rows spends as long in these queries as in a launch)
  static std::atomic<unsigned long long*> known[64];
  if (dev < 64 && (*flagged = known[dev].load(std::memory_order_acquire)) != nullptr) return SAKI_OK;
  int major = 0;
  e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceGetAttribute");
  if (major != 10) return fail(SAKI_ERR_UNSUPPORTED, "device compute capability %d.x: this library is built for sm_100a only", major);
  e = cudaGetSymbolAddress((void**)flagged, g_flagged_rows);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
  if (dev < 64) known[dev].store(*flagged, std::memory_order_release);
  return SAKI_OK;
}

// Scratch of the two-tier routing: the float32 kernels append the rows they cannot resolve to a list
// that the float64 kernel then routes.  One buffer per (device, stream), so that calls on different
// streams do not share a list; grown on demand, kept until exit.  (Calls on one stream are ordered by the
// stream, so they may share.)  A caller holds g_redo_mu from the hand-out until its kernels are launched,
// and nothing is freed while work that may use it is in flight: a buffer that was outgrown is retired,
// not freed, and the sweep that follows many short-lived streams first waits for the device.  Every
// free bumps g_redo_generation, which the counter readers check before they follow g_last_redo_count.
struct RedoBuf {
  int32_t* list = nullptr;       // [cap] rows, followed by the counter
  int64_t cap = 0;
};
static std::mutex g_redo_mu;
static std::map<std::pair<int, cudaStream_t>, RedoBuf> g_redo;
static std::vector<std::pair<int, int32_t*>> g_retired;          // (device, buffer) outgrown, still possibly in use
static std::atomic<uint64_t> g_redo_generation{0};
static thread_local unsigned int* g_last_redo_count = nullptr;
static thread_local uint64_t g_last_redo_generation = 0;

// Zeroes device memory before it returns, on a stream of its own: the caller's may be under capture (one that lets memory be
// allocated), where a memset would only happen when the graph is launched, after ordinary calls on that stream.
static cudaError_t zero_now(void* p, size_t bytes) {
  cudaStream_t own = nullptr;
  cudaError_t e = cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(p, 0, bytes, own);
  if (e == cudaSuccess) e = cudaStreamSynchronize(own);
  cudaStreamDestroy(own);
  return e;
}

// g_redo_mu held by the caller
static int redo_scratch(int64_t n_rows, cudaStream_t st, int32_t** list, unsigned int** count) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (g_redo.size() > 256) {   // many short-lived streams: start over, once nothing on the device can still use a list
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceSynchronize (scratch sweep)");
    for (auto& kv : g_redo)
      if (kv.first.first == dev && kv.second.list) { cudaFree(kv.second.list); kv.second = RedoBuf(); }
    for (auto it = g_redo.begin(); it != g_redo.end();) it = it->second.list ? std::next(it) : g_redo.erase(it);
    for (auto& r : g_retired)
      if (r.first == dev && r.second) { cudaFree(r.second); r.second = nullptr; }
    g_retired.erase(std::remove_if(g_retired.begin(), g_retired.end(), [](const std::pair<int, int32_t*>& r) { return !r.second; }),
                    g_retired.end());
    g_redo_generation.fetch_add(1);
  }
  RedoBuf& b = g_redo[std::make_pair(dev, st)];
  if (b.cap < n_rows) {
    if (b.list) g_retired.emplace_back(dev, b.list);   // an earlier call on this stream may still be running on it
    b = RedoBuf();
    const int64_t cap = (std::max<int64_t>(n_rows, 1 << 16) + 63) & ~(int64_t)63;
    // row ids, the counters, and as many words again (block verification: one per sequence)
    cudaError_t e = cudaMalloc((void**)&b.list, (size_t)(2 * cap + CNT_WORDS) * sizeof(int32_t));
    if (e != cudaSuccess) { b = RedoBuf(); return cuda_fail(e, "cudaMalloc (redo list)"); }
    e = zero_now(b.list + cap, CNT_WORDS * sizeof(int32_t));
    if (e != cudaSuccess) { cudaFree(b.list); b = RedoBuf(); return cuda_fail(e, "zeroing the redo list's counters"); }
    b.cap = cap;
  }
  *list = b.list;
  *count = (unsigned int*)(b.list + b.cap);
  return SAKI_OK;
}
// the calling thread's last routing call's counters, or NULL if there are none (any more)
static unsigned int* last_counters() {
  return g_last_redo_generation == g_redo_generation.load() && g_last_redo_count ? g_last_redo_count + CNT_LAST : nullptr;
}

// Fixed scratch of saki_route_fwd_bwd_noalloc: the redo list of the two-tier routing for callers that must
// not allocate.  SAKI_NOALLOC_MAX_ROWS row ids plus the counter; every device that loads the library holds
// these 4 MB until the process exits.
#define SAKI_NOALLOC_MAX_ROWS (1 << 20)
static __device__ __align__(256) int32_t g_noalloc_scratch[SAKI_NOALLOC_MAX_ROWS + CNT_WORDS];
static std::mutex g_noalloc_mu;
static int32_t* g_noalloc_ptr[64] = {nullptr};   // device address of the array, per device ordinal

// In host code the array's name is only a handle; the kernels need its device address, looked up once per
// device with that device current.
static int noalloc_scratch(int32_t** list, unsigned int** count) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= 64) return fail(SAKI_ERR_UNSUPPORTED, "device ordinal %d outside the table", dev);
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    int32_t* ptr = nullptr;
    e = cudaGetSymbolAddress((void**)&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress (fixed scratch)");
    g_noalloc_ptr[dev] = ptr;
  }
  *list = g_noalloc_ptr[dev];
  *count = (unsigned int*)(g_noalloc_ptr[dev] + SAKI_NOALLOC_MAX_ROWS);
  return SAKI_OK;
}

static int check_common(const void* s, const void* t, int64_t n, int32_t V, int32_t dtype, float eps, float tau) {
  if (n < 0) return fail(SAKI_ERR_INVALID_ARG, "negative row count");
  if (V < 2) return fail(SAKI_ERR_INVALID_ARG, "V must be >= 2 (got %d)", V);
  if (dtype != SAKI_F32 && dtype != SAKI_BF16) return fail(SAKI_ERR_INVALID_ARG, "unknown dtype %d", dtype);
  if (!(eps >= 0.f)) return fail(SAKI_ERR_INVALID_ARG, "eps must be >= 0 and not NaN");
  if (!(tau > 0.f) || std::isinf(tau)) return fail(SAKI_ERR_INVALID_ARG, "temperature must be finite and > 0");
  if (n > 0 && (!s || !t)) return fail(SAKI_ERR_INVALID_ARG, "NULL logits pointer");
  return SAKI_OK;
}

// `scratch_list` / `scratch_count`: where the two-tier routing keeps its redo list (NULL: the library's
// own per-device buffer, allocated on demand).
static int dispatch_rows(RowParams p, int dtype, cudaStream_t st, int32_t* scratch_list = nullptr,
                         unsigned int* scratch_count = nullptr) {
  int launches = 0;
  cudaError_t e;
  bool served = false;
  const int which = g_kernel.load();
  if (which != 0) p.call_rows = 0;
  int used = 1;
  // Directly, float32 sums resolve KL(q||p) to a few 1e-7 absolute: enough for |d lambda| <= 1e-5 when
  // eps >= 5e-3 (measured), not below: for the cluster kernel smaller positive radii run on the float64
  // kernel.  The row-per-SM kernel gets KL for small radii from a quadrature of its slope instead
  // (relative, not absolute, accuracy) and takes every radius.
  const bool eps_ok = !(p.eps > 0.f) || p.eps >= 5e-3f;
  const bool rowsm_ok = (which == 0 || which == 3) && rowsm_can_serve(p, dtype);
  const bool fast = (which != 1) && (rowsm_ok || (eps_ok && cluster_can_serve(p, dtype)));
  p.redo_list = nullptr; p.redo_count = nullptr; p.redo_guess = nullptr; p.from_list = 0;
  p.wait_limit = std::min<long long>(g_wait_limit.load(), 1LL << 61);      // (the kernels add their own limit to it)
  g_last_redo_count = nullptr;          // the counters below describe this call only
  rowsm_layout_none();
  std::unique_lock<std::mutex> scratch_lock(g_redo_mu, std::defer_lock);
  if (fast) {
    if (scratch_list) { p.redo_list = scratch_list; p.redo_count = scratch_count; }
    else {
      scratch_lock.lock();       // until the kernels that use the list are launched
      const int rc = redo_scratch(p.n_rows, st, &p.redo_list, &p.redo_count);
      if (rc) return rc;
      // the words behind the counters (one per row; block verification keeps its sequences' stops there) take
      // what the float32 kernel made of lambda for the rows it hands over
      if (!p.spec) p.redo_guess = (float*)(p.redo_count + CNT_WORDS);
    }
    if (scratch_list) {   // shared by all callers of the device: whatever a call that was cut short may have left
      e = cudaMemsetAsync(p.redo_count, 0, CNT_LIVE * sizeof(unsigned int), st);
      if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    }
    p.phase_cycles = g_phase_clock.load() ? (unsigned long long*)(p.redo_count + CNT_PHASES) : nullptr;
    g_last_redo_count = p.redo_count;
    g_last_redo_generation = g_redo_generation.load();
  }
  // A handful of long rows (a decoding step of a small batch) finish sooner spread over the whole GPU, one row per cluster
  // of up to 16 blocks, than on one SM each: 1 / 8 / 32 rows of V = 151936 take 15.7 / 18.7 / 24.5 us there against 37 us
  // on two SMs each, of V = 32768 14 / 14 / 18 against 18 us (at V = 8192 there is no difference).
  if (fast && which == 0 && p.call_rows <= 32 && p.V >= 32768 && eps_ok && cluster_can_serve(p, dtype)) {
    e = launch_cluster(p, st, &launches, &served);
    if (e != cudaSuccess) return cuda_fail(e, "cluster kernel launch");
    if (served) used = 2;
  }
  if (fast && !served && (which == 0 || which == 3) && rowsm_can_serve(p, dtype)) {
    // Block verification with early out: positions handed out as tickets, sequences record their first stop.
    // Only with two or more sequences per SM: with fewer, most positions are handed out before their
    // predecessor's decision is known, and the bookkeeping costs more than the few skipped rows save.
    int sms = 0, dev_now = 0;
    if (p.spec && (cudaGetDevice(&dev_now) != cudaSuccess ||
                   cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev_now) != cudaSuccess)) sms = 0;
    if (p.spec && g_spec_early_out.load() && !scratch_list && sms > 0 && p.n_rows / p.K1 >= 2 * (int64_t)sms) {
      p.seq_next = p.redo_count + CNT_TICKET;
      p.seq_stop = (int*)(p.redo_count + CNT_WORDS);
      e = cudaMemsetAsync(p.seq_stop, 0x7f, (size_t)(p.n_rows / p.K1) * sizeof(int), st);   // "no stop yet": above any position
      if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
    }
    e = launch_rowsm(p, st, &launches, &served);
    p.seq_next = nullptr; p.seq_stop = nullptr;
    if (e != cudaSuccess) return cuda_fail(e, "row-per-SM kernel launch");
    if (served) used = 3;
  }
  if (fast && !served && which == 2 && cluster_can_serve(p, dtype)) {
    e = launch_cluster(p, st, &launches, &served);
    if (e != cudaSuccess) return cuda_fail(e, "cluster kernel launch");
    if (served) used = 2;
  }
  if (served) {   // second tier: the rows the float32 kernel handed over
    p.from_list = 1;
    e = launch_general(p, dtype, st, &launches);
    if (e != cudaSuccess) {
      cudaMemsetAsync(p.redo_count, 0, CNT_LIVE * sizeof(unsigned int), st);   // the kernel that would have cleared them is missing
      return cuda_fail(e, "general kernel launch (redo list)");
    }
  } else {
    e = launch_general(p, dtype, st, &launches);
    if (e != cudaSuccess) return cuda_fail(e, "general kernel launch");
  }
  g_launches += (uint64_t)launches;
  g_last_kernel = used;
  return SAKI_OK;
}

static int route_impl(const saki_in* in, const saki_out* out, void* dlogits, int64_t ld_g, float grad_scale,
                      bool bwd, void* stream, bool fixed_scratch = false, int64_t call_rows = 0) {
  g_err[0] = 0;
  if (!in || !out) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  if (fixed_scratch && in->N > SAKI_NOALLOC_MAX_ROWS)
    return fail(SAKI_ERR_INVALID_ARG, "N = %lld exceeds the fixed scratch of this entry point (%d rows): split the batch",
                (long long)in->N, SAKI_NOALLOC_MAX_ROWS);
  int rc = check_common(in->student_logits, in->teacher_logits, in->N, in->V, in->dtype, in->eps, in->temperature);
  if (rc) return rc;
  if (in->ld_s < in->V || in->ld_t < in->V) return fail(SAKI_ERR_INVALID_ARG, "row stride smaller than V");
  if (in->N > 0 && !in->proposal) return fail(SAKI_ERR_INVALID_ARG, "NULL proposal pointer");
  if (in->N > 0 && (!out->corrected || !out->token)) return fail(SAKI_ERR_INVALID_ARG, "out.corrected and out.token are required");
  if (bwd) {
    if (in->N > 0 && !dlogits) return fail(SAKI_ERR_INVALID_ARG, "NULL dlogits pointer");
    if (ld_g < in->V) return fail(SAKI_ERR_INVALID_ARG, "gradient row stride smaller than V");
    if (!std::isfinite(grad_scale)) return fail(SAKI_ERR_INVALID_ARG, "grad_scale must be finite");
  }
  if (in->N == 0) return SAKI_OK;
  unsigned long long* flagged = nullptr;
  rc = device_ready(&flagged);
  if (rc) return rc;
  RowParams p;
  memset(&p, 0, sizeof(p));
  p.s = in->student_logits; p.t = in->teacher_logits;
  p.s_seq = in->ld_s; p.s_pos = 0; p.t_seq = in->ld_t; p.t_pos = 0;
  p.n_rows = in->N; p.V = in->V; p.K1 = 1; p.spec = 0;
  p.call_rows = call_rows > 0 ? call_rows : in->N;
  p.proposal = in->proposal; p.prop_ld = 0; p.mask = in->mask;
  p.eps = in->eps; p.temperature = in->temperature; p.seed = in->seed; p.row_offset = in->row_offset;
  p.out = *out;
  p.dlogits = bwd ? dlogits : nullptr; p.ld_g = ld_g; p.grad_scale = grad_scale;
  p.flagged = flagged;
  if (fixed_scratch) {
    int32_t* list = nullptr;
    unsigned int* count = nullptr;
    rc = noalloc_scratch(&list, &count);
    if (rc) return rc;
    return dispatch_rows(p, in->dtype, (cudaStream_t)stream, list, count);
  }
  return dispatch_rows(p, in->dtype, (cudaStream_t)stream);
}

// ---- the trainer's step: loss and gradient from the rollout's metadata (Section 3.5) ----
static int meta_impl(const saki_meta_in* in, const saki_meta_out* out, void* dlogits, int64_t ld_g, float grad_scale,
                     void* stream) {
  g_err[0] = 0;
  if (!in || !out) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  if (in->N < 0) return fail(SAKI_ERR_INVALID_ARG, "negative row count");
  if (in->V < 2) return fail(SAKI_ERR_INVALID_ARG, "V must be >= 2 (got %d)", in->V);
  if (in->dtype != SAKI_F32 && in->dtype != SAKI_BF16) return fail(SAKI_ERR_INVALID_ARG, "unknown dtype %d", in->dtype);
  if (!(in->temperature > 0.f) || std::isinf(in->temperature))
    return fail(SAKI_ERR_INVALID_ARG, "temperature must be finite and > 0");
  if (in->ld_s < in->V || ld_g < in->V) return fail(SAKI_ERR_INVALID_ARG, "row stride smaller than V");
  if (!std::isfinite(grad_scale)) return fail(SAKI_ERR_INVALID_ARG, "grad_scale must be finite");
  if (in->N == 0) return SAKI_OK;
  if (!in->student_logits || !dlogits) return fail(SAKI_ERR_INVALID_ARG, "NULL logits or dlogits pointer");
  if (!in->corrected || !in->proposal || !in->teacher_top1 || !in->advantage)
    return fail(SAKI_ERR_INVALID_ARG, "corrected, proposal, teacher_top1 and advantage are required");
  unsigned long long* flagged = nullptr;
  int rc = device_ready(&flagged);
  if (rc) return rc;
  MetaParams p;
  memset(&p, 0, sizeof(p));
  p.s = in->student_logits; p.ld_s = in->ld_s; p.n_rows = in->N; p.V = in->V;
  p.corrected = in->corrected; p.proposal = in->proposal; p.teacher_top1 = in->teacher_top1;
  p.advantage = in->advantage; p.mask = in->mask; p.rollout_status = in->rollout_status;
  p.temperature = in->temperature; p.out = *out; p.dlogits = dlogits; p.ld_g = ld_g; p.grad_scale = grad_scale;
  p.flagged = flagged;
  cudaStream_t st = (cudaStream_t)stream;
  int launches = 0;
  cudaError_t e;
  bool served = false;
  int used = 1;
  g_last_redo_count = nullptr;
  std::unique_lock<std::mutex> scratch_lock(g_redo_mu, std::defer_lock);
  if (g_kernel.load() != 1 && meta_stream_can_serve(p, in->dtype)) {
    scratch_lock.lock();         // until the kernels that use the list are launched
    rc = redo_scratch(p.n_rows, st, &p.redo_list, &p.redo_count);
    if (rc) return rc;
    g_last_redo_count = p.redo_count;
    g_last_redo_generation = g_redo_generation.load();
    e = launch_meta_stream(p, st, &launches, &served);
    if (e != cudaSuccess) return cuda_fail(e, "streaming backward kernel launch");
    if (served) { used = 4; p.from_list = 1; }
  }
  e = launch_meta_general(p, in->dtype, st, &launches);
  if (e != cudaSuccess) {
    if (p.from_list) cudaMemsetAsync(p.redo_count, 0, CNT_LIVE * sizeof(unsigned int), st);
    return cuda_fail(e, "general backward kernel launch");
  }
  g_launches += (uint64_t)launches;
  g_last_kernel = used;
  return SAKI_OK;
}

// ---- block verification: per-sequence first-rejection resolve (Section 3.5) ----
__global__ void spec_resolve_kernel(int64_t B, int K, saki_out o, int32_t* n_accept, int32_t* next_token,
                                    uint8_t* next_is_corr) {
  launch_dependents();
  wait_for_predecessor();
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int K1 = K + 1;
  int n = K, stopped = 0, next = -1, isc = 0;
  for (int j = 0; j < K; ++j) {
    const int64_t r = b * K1 + j;
    if (o.token[r] < 0) { n = j; stopped = 1; break; }            // flagged row: cannot verify further
    if (o.corrected[r]) { n = j; stopped = 1; next = o.token[r]; isc = 1; break; }
  }
  if (!stopped) next = o.token[b * K1 + K];                        // bonus draw (or -1 if flagged)
  n_accept[b] = n; next_token[b] = next; next_is_corr[b] = (uint8_t)isc;
  if (stopped) {                                                   // later positions sit on an invalid prefix
    const RowResult z = zero_row(SAKI_ROW_NOT_COMPUTED);
    for (int j = n + 1; j < K1; ++j) write_row(o, b * K1 + j, z, false);
  }
}

// ---- host-buffer entry ----
// The rows go through the GPU in chunks: one stream brings logits in, without a gap, one routes, one takes the gradient out
// while later chunks come in.  What a call keeps per position (proposals, mask, outputs) is moved once for all chunks, the
// outputs through a pinned buffer (a copy per field and chunk costs more than its bytes).
constexpr int HOST_BUFS = 3;
enum { HS_IN = 0, HS_RUN, HS_OUT, HS_STREAMS };
struct HostStage {
  std::mutex mu;
  int dev = -1;
  cudaStream_t st[HS_STREAMS] = {nullptr};
  cudaEvent_t in[HOST_BUFS] = {nullptr}, run[HOST_BUFS] = {nullptr}, out[HOST_BUFS] = {nullptr};   // chunk is in / routed / out
  void* buf[HOST_BUFS] = {nullptr};
  size_t cap[HOST_BUFS] = {0};
  void* pos = nullptr;       // device: per-position arrays of the whole call
  void* pos_host = nullptr;  // pinned: the outputs among them
  size_t pos_cap = 0, pos_host_cap = 0;
};
static HostStage g_stage;

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace saki

using namespace saki;

extern "C" {

SAKI_API int saki_route_fwd(const saki_in* in, const saki_out* out, void* cuda_stream) {
  return route_impl(in, out, nullptr, 0, 0.f, false, cuda_stream);
}

SAKI_API int saki_route_fwd_bwd(const saki_in* in, const saki_out* out, void* dlogits, int64_t ld_g, float grad_scale,
                       void* cuda_stream) {
  return route_impl(in, out, dlogits, ld_g, grad_scale, true, cuda_stream);
}

SAKI_API int saki_route_fwd_bwd_noalloc(const saki_in* in, const saki_out* out, void* dlogits, int64_t ld_g,
                                        float grad_scale, void* cuda_stream) {
  return route_impl(in, out, dlogits, ld_g, grad_scale, true, cuda_stream, true);
}

SAKI_API int saki_route_bwd_from_meta(const saki_meta_in* in, const saki_meta_out* out, void* dlogits, int64_t ld_g,
                                      float grad_scale, void* cuda_stream) {
  return meta_impl(in, out, dlogits, ld_g, grad_scale, cuda_stream);
}

SAKI_API int saki_select_tm(const saki_select_in* in, uint8_t* selected, int32_t* m, void* cuda_stream) {
  g_err[0] = 0;
  if (!in) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  if (in->N < 0 || in->B < 0) return fail(SAKI_ERR_INVALID_ARG, "negative size");
  if (in->mode != SAKI_SELECT_RANDOM && in->mode != SAKI_SELECT_TV_WEIGHTED)
    return fail(SAKI_ERR_INVALID_ARG, "unknown selection mode %d", in->mode);
  if (in->B == 0 || in->N == 0) return SAKI_OK;
  if (!in->seq_start || !in->corrected || !selected) return fail(SAKI_ERR_INVALID_ARG, "seq_start, corrected and selected are required");
  if (in->mode == SAKI_SELECT_TV_WEIGHTED && !in->tv) return fail(SAKI_ERR_INVALID_ARG, "tv is required in TV-weighted mode");
  unsigned long long* flagged = nullptr;
  int rc = device_ready(&flagged);
  if (rc) return rc;
  SelectParams p;
  memset(&p, 0, sizeof(p));
  p.N = in->N; p.B = in->B; p.seq_start = in->seq_start; p.corrected = in->corrected; p.tv = in->tv;
  p.mask = in->mask; p.rollout_status = in->rollout_status; p.mode = in->mode; p.seed = in->seed;
  p.row_offset = in->row_offset; p.selected = selected; p.m = m;
  int launches = 0;
  cudaError_t e = launch_select(p, (cudaStream_t)cuda_stream, &launches);
  if (e != cudaSuccess) return cuda_fail(e, "selection kernel launch");
  g_launches += (uint64_t)launches;
  return SAKI_OK;
}

static int vshard_check(const saki_vshard_in* in, int stage) {
  if (!in) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  if (stage < 0 || stage > 3) return fail(SAKI_ERR_INVALID_ARG, "stage must be 0..3 (got %d)", stage);
  if (in->N < 0) return fail(SAKI_ERR_INVALID_ARG, "negative row count");
  if (in->V < 2) return fail(SAKI_ERR_INVALID_ARG, "V must be >= 2 (got %d)", in->V);
  if (in->world < 1 || in->rank < 0 || in->rank >= in->world) return fail(SAKI_ERR_INVALID_ARG, "rank %d outside [0, %d)", in->rank, in->world);
  if (in->V_local < 0 || in->v0 < 0 || (int64_t)in->v0 + in->V_local > in->V)
    return fail(SAKI_ERR_INVALID_ARG, "slice [%d, %d) outside [0, %d)", in->v0, in->v0 + in->V_local, in->V);
  if (in->dtype != SAKI_F32 && in->dtype != SAKI_BF16) return fail(SAKI_ERR_INVALID_ARG, "unknown dtype %d", in->dtype);
  if (!(in->eps >= 0.f)) return fail(SAKI_ERR_INVALID_ARG, "eps must be >= 0 and not NaN");
  if (!(in->temperature > 0.f) || std::isinf(in->temperature)) return fail(SAKI_ERR_INVALID_ARG, "temperature must be finite and > 0");
  if (in->N > 0 && !in->proposal) return fail(SAKI_ERR_INVALID_ARG, "NULL proposal pointer");
  return SAKI_OK;
}

static int vshard_partials(const saki_vshard_in* in, int n, int stage, const double* state, double* const* partial,
                           void* const* dlogits, const int64_t* ld_g, float grad_scale, int flags, void* cuda_stream) {
  g_err[0] = 0;
  if (n < 0) return fail(SAKI_ERR_INVALID_ARG, "negative number of slices");
  if (n > 0 && (!in || !partial || (dlogits && !ld_g))) return fail(SAKI_ERR_INVALID_ARG, "NULL argument array");
  for (int k = 0; k < n; ++k) {
    const int rc = vshard_check(in + k, stage);
    if (rc) return rc;
    if (in[k].N != in[0].N || in[k].dtype != in[0].dtype) return fail(SAKI_ERR_INVALID_ARG, "the slices of one call have the same rows and dtype");
  }
  if (n == 0 || in[0].N == 0) return SAKI_OK;
  for (int k = 0; k < n; ++k) {
    if (in[k].V_local > 0 && (!in[k].student_logits || !in[k].teacher_logits)) return fail(SAKI_ERR_INVALID_ARG, "NULL logits pointer");
    if (in[k].ld_s < in[k].V_local || in[k].ld_t < in[k].V_local) return fail(SAKI_ERR_INVALID_ARG, "row stride smaller than the slice");
    if (!partial[k] || (stage > 0 && !state)) return fail(SAKI_ERR_INVALID_ARG, "NULL partial or state pointer");
    if (dlogits && dlogits[k] && (ld_g[k] < in[k].V_local || !std::isfinite(grad_scale))) return fail(SAKI_ERR_INVALID_ARG, "bad gradient stride or scale");
  }
  unsigned long long* flagged = nullptr;
  int rc = device_ready(&flagged);
  if (rc) return rc;
  int launches = 0;
  cudaError_t e = launch_vshard_partial(in, n, stage, state, partial, dlogits, ld_g, grad_scale, g_kernel.load() != 1, flags, &launches,
                                        (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "vocabulary-sharded partial kernel launch");
  g_launches += (uint64_t)launches;
  return SAKI_OK;
}

SAKI_API int saki_vshard_partial(const saki_vshard_in* in, int stage, const double* state, double* partial,
                                 void* dlogits_slice, int64_t ld_g, float grad_scale, void* cuda_stream) {
  return vshard_partials(in, 1, stage, state, &partial, dlogits_slice ? &dlogits_slice : nullptr, &ld_g, grad_scale, 0, cuda_stream);
}

SAKI_API int saki_vshard_stage(const saki_vshard_in* in, int n, int stage, double* state, double* const* partial,
                               const double* gathered, void* const* dlogits_slice, const int64_t* ld_g, float grad_scale,
                               const saki_out* out, uint32_t* counts, int flags, void* cuda_stream) {
  const int rc = vshard_partials(in, n, stage, state, partial, dlogits_slice, ld_g, grad_scale, flags, cuda_stream);
  if (rc || n == 0 || in[0].N == 0) return rc;
  if (!gathered || !state) return fail(SAKI_ERR_INVALID_ARG, "NULL gathered or state pointer");
  if (stage == 3 && (!out || !out->corrected || !out->token)) return fail(SAKI_ERR_INVALID_ARG, "out.corrected and out.token are required at stage 3");
  saki_out none;
  memset(&none, 0, sizeof(none));
  cudaError_t e = launch_vshard_combine(in[0], stage, gathered, state, out ? *out : none, counts, counts ? counts + 1 : nullptr,
                                        g_kernel.load() != 1, (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "vocabulary-sharded combine kernel launch");
  g_launches += 1;
  return SAKI_OK;
}

SAKI_API int saki_vshard_combine(const saki_vshard_in* in, int stage, const double* gathered, double* state,
                                 const saki_out* out, uint32_t* n_solving, void* cuda_stream) {
  g_err[0] = 0;
  int rc = vshard_check(in, stage);
  if (rc) return rc;
  if (in->N == 0) return SAKI_OK;
  if (!gathered || !state) return fail(SAKI_ERR_INVALID_ARG, "NULL gathered or state pointer");
  if (stage == 3 && (!out || !out->corrected || !out->token)) return fail(SAKI_ERR_INVALID_ARG, "out.corrected and out.token are required at stage 3");
  unsigned long long* flagged = nullptr;
  rc = device_ready(&flagged);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (n_solving) {
    cudaError_t e0 = cudaMemsetAsync(n_solving, 0, sizeof(uint32_t), st);
    if (e0 != cudaSuccess) return cuda_fail(e0, "cudaMemsetAsync");
  }
  saki_out none;
  memset(&none, 0, sizeof(none));
  cudaError_t e = launch_vshard_combine(*in, stage, gathered, state, out ? *out : none, n_solving, nullptr, g_kernel.load() != 1, st);
  if (e != cudaSuccess) return cuda_fail(e, "vocabulary-sharded combine kernel launch");
  g_launches += 1;
  return SAKI_OK;
}

SAKI_API int saki_vshard_combine_host(const saki_vshard_in* in, int stage, const double* gathered, double* state,
                                      const saki_out* out, int32_t* n_solving) {
  g_err[0] = 0;
  int rc = vshard_check(in, stage);
  if (rc) return rc;
  if (n_solving) *n_solving = 0;
  if (in->N == 0) return SAKI_OK;
  if (!gathered || !state) return fail(SAKI_ERR_INVALID_ARG, "NULL gathered or state pointer");
  if (stage == 3 && (!out || !out->corrected || !out->token)) return fail(SAKI_ERR_INVALID_ARG, "out.corrected and out.token are required at stage 3");
  saki_out none;
  memset(&none, 0, sizeof(none));
  const int solving = vshard_combine_host(*in, stage, gathered, state, out ? *out : none, g_kernel.load() != 1);
  if (n_solving) *n_solving = solving;
  return SAKI_OK;
}

SAKI_API int64_t saki_lmhead_scratch_bytes(int64_t N, int32_t V) {
  if (N < 0 || V < 1) return 0;
  return lmhead_scratch_bytes(N, V);
}

SAKI_API int saki_lmhead_lse(const saki_lmhead_in* in, void* logits, int64_t ld_l, float* row_max, float* lse,
                             void* scratch, int64_t scratch_bytes, void* cuda_stream) {
  g_err[0] = 0;
  if (!in) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  if (in->N < 0) return fail(SAKI_ERR_INVALID_ARG, "negative row count");
  if (in->V < 8 || in->d < 8) return fail(SAKI_ERR_INVALID_ARG, "V and d must be >= 8 (got %d, %d)", in->V, in->d);
  if (!(in->temperature > 0.f) || std::isinf(in->temperature)) return fail(SAKI_ERR_INVALID_ARG, "temperature must be finite and > 0");
  if (in->ld_h < in->d || in->ld_w < in->d || ld_l < in->V) return fail(SAKI_ERR_INVALID_ARG, "row stride smaller than the row");
  if (in->N == 0) return SAKI_OK;
  if (!in->hidden || !in->weight || !logits || !scratch) return fail(SAKI_ERR_INVALID_ARG, "NULL hidden, weight, logits or scratch pointer");
  if (scratch_bytes < lmhead_scratch_bytes(in->N, in->V)) return fail(SAKI_ERR_INVALID_ARG, "scratch too small: %lld bytes needed", (long long)lmhead_scratch_bytes(in->N, in->V));
  auto al = [](const void* q, uintptr_t a) { return ((uintptr_t)q & (a - 1)) == 0; };
  if (!al(in->hidden, 16) || !al(in->weight, 16) || !al(logits, 16) || !al(scratch, 256) || in->ld_h % 8 || in->ld_w % 8 || ld_l % 8 || in->V % 8)
    return fail(SAKI_ERR_UNSUPPORTED, "pointers must be 16-byte aligned (scratch 256), strides and V multiples of 8");
  unsigned long long* flagged = nullptr;
  int rc = device_ready(&flagged);
  if (rc) return rc;
  const char* why = nullptr;
  cudaError_t e = launch_lmhead(*in, logits, ld_l, row_max, lse, scratch, (cudaStream_t)cuda_stream, &why);
  if (e != cudaSuccess) return why ? fail(SAKI_ERR_CUDA, "%s", why) : cuda_fail(e, "lm-head kernel launch");
  g_launches += 2;
  return SAKI_OK;
}

SAKI_API int saki_spec_verify(const saki_spec_in* in, const saki_spec_out* out, void* cuda_stream) {
  g_err[0] = 0;
  if (!in || !out) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  int rc = check_common(in->student_logits, in->teacher_logits, in->B, in->V, in->dtype, in->eps, in->temperature);
  if (rc) return rc;
  if (in->K < 1 || in->K > 16) return fail(SAKI_ERR_INVALID_ARG, "K must be in [1,16] (got %d)", in->K);
  if (in->ss_pos < in->V || in->ts_pos < in->V) return fail(SAKI_ERR_INVALID_ARG, "position stride smaller than V");
  if (in->ss_seq < in->ss_pos || in->ts_seq < in->ts_pos) return fail(SAKI_ERR_INVALID_ARG, "sequence stride smaller than position stride");
  if (in->B > 0 && (!in->draft || in->draft_ld < in->K)) return fail(SAKI_ERR_INVALID_ARG, "bad draft pointer or stride");
  if (in->B > 0 && (!out->n_accept || !out->next_token || !out->next_is_correction || !out->per_pos.corrected ||
                    !out->per_pos.token))
    return fail(SAKI_ERR_INVALID_ARG, "n_accept, next_token, next_is_correction, per_pos.corrected and per_pos.token are required");
  if (in->B == 0) return SAKI_OK;
  unsigned long long* flagged = nullptr;
  rc = device_ready(&flagged);
  if (rc) return rc;
  RowParams p;
  memset(&p, 0, sizeof(p));
  p.s = in->student_logits; p.t = in->teacher_logits;
  p.s_seq = in->ss_seq; p.s_pos = in->ss_pos; p.t_seq = in->ts_seq; p.t_pos = in->ts_pos;
  p.K1 = in->K + 1; p.n_rows = p.call_rows = in->B * p.K1; p.V = in->V; p.spec = 1;
  p.proposal = in->draft; p.prop_ld = in->draft_ld; p.mask = nullptr;
  p.eps = in->eps; p.temperature = in->temperature; p.seed = in->seed;
  p.row_offset = in->seq_offset * (uint64_t)p.K1;
  p.out = out->per_pos;
  p.out.loss = nullptr;
  p.dlogits = nullptr; p.ld_g = 0; p.grad_scale = 0.f; p.flagged = flagged;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  rc = dispatch_rows(p, in->dtype, st);
  if (rc) return rc;
  const int th = 128;
  cudaError_t e = launch_pdl(spec_resolve_kernel, dim3((unsigned)((in->B + th - 1) / th)), th, 0, st, true, in->B, in->K, p.out,
                             out->n_accept, out->next_token, out->next_is_correction);
  g_launches += 1;
  if (e != cudaSuccess) return cuda_fail(e, "resolve kernel launch");
  return SAKI_OK;
}

SAKI_API int saki_sample_proposal(const void* logits, int64_t ld, int64_t N, int32_t V, int32_t dtype, float temperature,
                         uint64_t seed, uint64_t row_offset, int32_t* out, void* cuda_stream) {
  g_err[0] = 0;
  int rc = check_common(logits, logits, N, V, dtype, 0.f, temperature);
  if (rc) return rc;
  if (ld < V) return fail(SAKI_ERR_INVALID_ARG, "row stride smaller than V");
  if (N > 0 && !out) return fail(SAKI_ERR_INVALID_ARG, "NULL output pointer");
  if (N == 0) return SAKI_OK;
  unsigned long long* flagged = nullptr;
  rc = device_ready(&flagged);
  if (rc) return rc;
  cudaError_t e = launch_propose(logits, ld, N, V, dtype, temperature, seed, row_offset, out, (cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "proposal kernel launch");
  g_launches += 1;
  return SAKI_OK;
}

SAKI_API int saki_check(void* cuda_stream, uint64_t* n_flagged) {
  g_err[0] = 0;
  unsigned long long* flagged = nullptr;
  int rc = device_ready(&flagged);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  cudaError_t e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  unsigned long long h = 0, zero = 0;
  e = cudaMemcpy(&h, flagged, sizeof(h), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  e = cudaMemcpy(flagged, &zero, sizeof(zero), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  if (n_flagged) *n_flagged = h;
  if (h) return fail(SAKI_ERR_ROW_STATUS, "%llu row(s) flagged (non-finite logits, bad proposal id or timeout)", h);
  return SAKI_OK;
}

SAKI_API int saki_route_host(const saki_in* in, const saki_out* out, void* dlogits, int64_t ld_g, float grad_scale) {
  g_err[0] = 0;
  if (!in || !out) return fail(SAKI_ERR_INVALID_ARG, "NULL argument struct");
  int rc = check_common(in->student_logits, in->teacher_logits, in->N, in->V, in->dtype, in->eps, in->temperature);
  if (rc) return rc;
  if (in->ld_s < in->V || in->ld_t < in->V) return fail(SAKI_ERR_INVALID_ARG, "row stride smaller than V");
  if (dlogits && ld_g < in->V) return fail(SAKI_ERR_INVALID_ARG, "gradient row stride smaller than V");
  if (in->N > 0 && (!in->proposal || !out->corrected || !out->token))
    return fail(SAKI_ERR_INVALID_ARG, "proposal, out.corrected and out.token are required");
  if (in->N == 0) return SAKI_OK;
  unsigned long long* flagged = nullptr;
  rc = device_ready(&flagged);
  if (rc) return rc;

  std::lock_guard<std::mutex> lock(g_stage.mu);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaError_t e;
  if (g_stage.dev != dev) {   // (re)create the staging streams on this device
    g_stage.dev = -1;
    if (g_stage.pos) { cudaFree(g_stage.pos); g_stage.pos = nullptr; g_stage.pos_cap = 0; }
    for (int k = 0; k < HOST_BUFS; ++k) {
      if (g_stage.buf[k]) { cudaFree(g_stage.buf[k]); g_stage.buf[k] = nullptr; g_stage.cap[k] = 0; }
      for (cudaEvent_t* ev : {&g_stage.in[k], &g_stage.run[k], &g_stage.out[k]}) {
        if (*ev) { cudaEventDestroy(*ev); *ev = nullptr; }
        e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return cuda_fail(e, "cudaEventCreate");
      }
    }
    for (cudaStream_t& st : g_stage.st) {
      if (st) { cudaStreamDestroy(st); st = nullptr; }
      e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
      if (e != cudaSuccess) return cuda_fail(e, "cudaStreamCreate");
    }
    g_stage.dev = dev;
  }
  const size_t es = in->dtype == SAKI_BF16 ? 2 : 4;
  const size_t Vp = align_up((size_t)in->V, 16);   // padded device row stride: rows stay 16-byte aligned
  const size_t row_bytes = Vp * es;
  const int64_t N = in->N;
  // A chunk is half of what is left, between 4 and 32 MB of logits.  The gradient is half of the logits, so a chunk's way
  // out takes as long as the next one's way in, and only the last, short chunk is routed and taken out with nothing beside
  // it.  Copies are few because each costs some 5 us beyond its bytes, more where both directions are busy: 512 rows of
  // 32000 (66 MB in: 1.21 ms, 33 MB out: 0.60 ms; 1.27 ms both at once in one piece each) took 1.94 ms in one chunk, 1.51
  // to 1.60 ms in twelve, 1.74 ms in eight, 1.55 ms with the gradient stored into host memory by the kernels.
  const int64_t pair_bytes = 2 * (int64_t)row_bytes;
  auto chunk_rows = [&](int64_t left) {
    const int64_t bytes = std::min<int64_t>(32 << 20, std::max<int64_t>(4 << 20, left * pair_bytes / 2));
    const int64_t n = std::max<int64_t>(1, bytes / pair_bytes);
    return left * pair_bytes <= (6 << 20) ? left : std::min(left, n);     // (no crumbs)
  };
  int64_t chunk = 0;
  for (int64_t r0 = 0, n = 0; r0 < N && r0 < 8 * std::max<int64_t>(1, chunk); r0 += n) { n = chunk_rows(N - r0); chunk = std::max(chunk, n); }
  const size_t total = (size_t)chunk * row_bytes * (dlogits ? 3 : 2);
  for (int k = 0; k < HOST_BUFS; ++k) {
    if (g_stage.cap[k] < total) {
      if (g_stage.buf[k]) cudaFree(g_stage.buf[k]);
      g_stage.buf[k] = nullptr; g_stage.cap[k] = 0;
      e = cudaMalloc(&g_stage.buf[k], total);
      if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (staging)");
      g_stage.cap[k] = total;
    }
  }
  // per-position arrays: the 15 outputs first (copied back as one block), then proposals and mask
  struct Field { void* host; size_t size, off; };
  Field f[15] = {{out->token, 4, 0}, {out->teacher_top1, 4, 0}, {out->row_status, 4, 0}, {out->lambda, 4, 0}, {out->kl, 4, 0},
                 {out->tv, 4, 0}, {out->accept_prob, 4, 0}, {out->logp_x, 4, 0}, {out->logq_x, 4, 0}, {out->logT_x, 4, 0},
                 {out->logp_y, 4, 0}, {out->logq_y, 4, 0}, {out->logT_y, 4, 0}, {out->loss, 4, 0}, {out->corrected, 1, 0}};
  size_t off = 0;
  for (Field& x : f)
    if (x.host) { x.off = off; off += align_up((size_t)N * x.size, 16); }
  const size_t out_bytes = off, o_prop = off, o_mask = o_prop + align_up((size_t)N * 4, 16), pos_bytes = o_mask + (size_t)N;
  if (g_stage.pos_cap < pos_bytes) {
    if (g_stage.pos) cudaFree(g_stage.pos);
    g_stage.pos = nullptr; g_stage.pos_cap = 0;
    e = cudaMalloc(&g_stage.pos, pos_bytes);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc (staging)");
    g_stage.pos_cap = pos_bytes;
  }
  if (g_stage.pos_host_cap < out_bytes) {
    if (g_stage.pos_host) cudaFreeHost(g_stage.pos_host);
    g_stage.pos_host = nullptr; g_stage.pos_host_cap = 0;
    e = cudaMallocHost(&g_stage.pos_host, out_bytes);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocHost (staging)");
    g_stage.pos_host_cap = out_bytes;
  }
  char* const pos = (char*)g_stage.pos;
  auto field = [&](int q, int64_t r0) -> void* { return f[q].host ? pos + f[q].off + (size_t)r0 * f[q].size : nullptr; };
  // rows whose strides agree are one piece
  auto copy_rows = [&](void* dst, size_t dpitch, const void* src, size_t spitch, int64_t n, cudaMemcpyKind kind, cudaStream_t st) {
    const size_t width = (size_t)in->V * es;
    if (dpitch == width && spitch == width) return cudaMemcpyAsync(dst, src, width * (size_t)n, kind, st);
    return cudaMemcpy2DAsync(dst, dpitch, src, spitch, width, (size_t)n, kind, st);
  };
  cudaStream_t const s_in = g_stage.st[HS_IN], s_run = g_stage.st[HS_RUN], s_out = g_stage.st[HS_OUT];
  int result = SAKI_OK;
  auto ok = [&](cudaError_t err, const char* what) {
    if (err != cudaSuccess && result == SAKI_OK) result = cuda_fail(err, what);
  };
  ok(cudaMemcpyAsync(pos + o_prop, in->proposal, (size_t)N * 4, cudaMemcpyHostToDevice, s_in), "host-to-device copy");
  if (in->mask) ok(cudaMemcpyAsync(pos + o_mask, in->mask, (size_t)N, cudaMemcpyHostToDevice, s_in), "host-to-device copy");
  int64_t i = 0;                                     // chunk number
  for (int64_t r0 = 0, n = 0; r0 < N && result == SAKI_OK; r0 += n, ++i) {
    const int k = (int)(i % HOST_BUFS);
    n = chunk_rows(N - r0);
    char* const b_s = (char*)g_stage.buf[k];
    char* const b_t = b_s + (size_t)chunk * row_bytes;
    char* const b_g = b_t + (size_t)chunk * row_bytes;
    if (i >= HOST_BUFS) ok(cudaStreamWaitEvent(s_in, g_stage.run[k], 0), "cudaStreamWaitEvent");   // the buffer's last rows are routed
    ok(copy_rows(b_s, row_bytes, (const char*)in->student_logits + (size_t)r0 * in->ld_s * es, in->ld_s * es, n, cudaMemcpyHostToDevice, s_in), "host-to-device copy");
    ok(copy_rows(b_t, row_bytes, (const char*)in->teacher_logits + (size_t)r0 * in->ld_t * es, in->ld_t * es, n, cudaMemcpyHostToDevice, s_in), "host-to-device copy");
    ok(cudaEventRecord(g_stage.in[k], s_in), "cudaEventRecord");
    ok(cudaStreamWaitEvent(s_run, g_stage.in[k], 0), "cudaStreamWaitEvent");
    if (dlogits && i >= HOST_BUFS) ok(cudaStreamWaitEvent(s_run, g_stage.out[k], 0), "cudaStreamWaitEvent");
    if (result != SAKI_OK) break;
    saki_in din = *in;
    din.student_logits = b_s; din.teacher_logits = b_t; din.ld_s = din.ld_t = (int64_t)Vp;
    din.N = n; din.proposal = (const int32_t*)(pos + o_prop) + r0;
    din.mask = in->mask ? (const uint8_t*)(pos + o_mask) + r0 : nullptr;
    din.row_offset = in->row_offset + (uint64_t)r0;
    saki_out dout;
    dout.token = (int32_t*)field(0, r0); dout.teacher_top1 = (int32_t*)field(1, r0); dout.row_status = (uint32_t*)field(2, r0);
    float** const df[11] = {&dout.lambda, &dout.kl, &dout.tv, &dout.accept_prob, &dout.logp_x, &dout.logq_x, &dout.logT_x,
                            &dout.logp_y, &dout.logq_y, &dout.logT_y, &dout.loss};
    for (int q = 0; q < 11; ++q) *df[q] = (float*)field(3 + q, r0);
    dout.corrected = (uint8_t*)field(14, r0);
    result = route_impl(&din, &dout, dlogits ? b_g : nullptr, (int64_t)Vp, grad_scale, dlogits != nullptr, s_run, false, N);
    if (result != SAKI_OK) break;
    ok(cudaEventRecord(g_stage.run[k], s_run), "cudaEventRecord");
    if (dlogits) {
      ok(cudaStreamWaitEvent(s_out, g_stage.run[k], 0), "cudaStreamWaitEvent");
      ok(copy_rows((char*)dlogits + (size_t)r0 * ld_g * es, ld_g * es, b_g, row_bytes, n, cudaMemcpyDeviceToHost, s_out), "device-to-host copy");
      ok(cudaEventRecord(g_stage.out[k], s_out), "cudaEventRecord");
    }
  }
  if (result == SAKI_OK) ok(cudaMemcpyAsync(g_stage.pos_host, pos, out_bytes, cudaMemcpyDeviceToHost, s_run), "device-to-host copy");
  for (cudaStream_t st : g_stage.st) ok(cudaStreamSynchronize(st), "cudaStreamSynchronize");
  if (result == SAKI_OK)
    for (const Field& x : f) if (x.host) memcpy(x.host, (const char*)g_stage.pos_host + x.off, (size_t)N * x.size);
  return result;
}

SAKI_API int saki_set_kernel(int which) {
  if (which < 0 || which > 3) which = 0;
  return g_kernel.exchange(which);
}

SAKI_API int saki_last_kernel(void) { return g_last_kernel; }

SAKI_API void saki_last_layout(int32_t* blocks_per_row, int32_t* blocks_per_sm, int32_t* resident_rows) {
  int l[3];
  general_layout(l);
  if (blocks_per_row) *blocks_per_row = l[0];
  if (blocks_per_sm) *blocks_per_sm = l[1];
  if (resident_rows) *resident_rows = l[2];
}

SAKI_API void saki_last_rowsm_layout(int32_t* blocks_per_row, int32_t* blocks_per_sm) {
  int l[2];
  rowsm_layout(l);
  if (blocks_per_row) *blocks_per_row = l[0];
  if (blocks_per_sm) *blocks_per_sm = l[1];
}

SAKI_API int saki_redo_count(void* cuda_stream, uint64_t* n_rows) {
  g_err[0] = 0;
  if (!n_rows) return fail(SAKI_ERR_INVALID_ARG, "NULL output pointer");
  *n_rows = 0;
  unsigned int* const counters = last_counters();
  if (!counters) return SAKI_OK;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  unsigned int h = 0;
  e = cudaMemcpy(&h, counters, sizeof(h), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  *n_rows = h;
  return SAKI_OK;
}

SAKI_API int saki_solve_evaluations(void* cuda_stream, uint64_t* n_passes) {
  g_err[0] = 0;
  if (!n_passes) return fail(SAKI_ERR_INVALID_ARG, "NULL output pointer");
  *n_passes = 0;
  unsigned int* const counters = last_counters();
  if (!counters) return SAKI_OK;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  unsigned int h = 0;
  e = cudaMemcpy(&h, counters + CNT_EVALS, sizeof(h), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  *n_passes = h;
  return SAKI_OK;
}

SAKI_API int64_t saki_set_wait_limit(int64_t cycles) { return (int64_t)g_wait_limit.exchange(cycles > 0 ? (long long)cycles : 0); }

SAKI_API int saki_set_phase_clock(int on) { return g_phase_clock.exchange(on ? 1 : 0); }

SAKI_API int saki_phase_cycles(void* cuda_stream, uint64_t* cycles) {
  g_err[0] = 0;
  if (!cycles) return fail(SAKI_ERR_INVALID_ARG, "NULL output pointer");
  memset(cycles, 0, SAKI_PHASE_COUNTERS * sizeof(uint64_t));
  unsigned int* const counters = last_counters();
  if (!counters) return SAKI_OK;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  e = cudaMemcpy(cycles, counters + CNT_PHASES, SAKI_PHASE_COUNTERS * sizeof(uint64_t), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  return SAKI_OK;
}

SAKI_API int saki_set_spec_early_out(int on) { return g_spec_early_out.exchange(on ? 1 : 0); }

SAKI_API int saki_spec_positions_routed(void* cuda_stream, uint64_t* n_positions) {
  g_err[0] = 0;
  if (!n_positions) return fail(SAKI_ERR_INVALID_ARG, "NULL output pointer");
  *n_positions = 0;
  unsigned int* const counters = last_counters();
  if (!counters) return SAKI_OK;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)cuda_stream);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  unsigned int h = 0;
  e = cudaMemcpy(&h, counters + CNT_ROUTED, sizeof(h), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy");
  *n_positions = h;
  return SAKI_OK;
}

SAKI_API uint64_t saki_launch_count(void) { return g_launches.load(); }

SAKI_API const char* saki_last_error(void) { return g_err; }

SAKI_API int saki_version(void) { return 100; }

}  // extern "C"
