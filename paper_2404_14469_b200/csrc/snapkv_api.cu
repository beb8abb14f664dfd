// C ABI of libsnapkv: argument validation, workspace layout, and the sequence of
// launches that makes up the compression step (Listing 1).
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "../../include/snapkv.h"
#include "launch.cuh"
#include "snapkv_binding.h"
#include "snapkv_internal.h"

namespace snapkv {

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Clears the status block and the unit counters behind it (n16 vectors) and marks the partial
// slots that follow as not written (up to n16_all).  A kernel rather than memsets so that the
// scoring kernel behind it can be made resident early.
__global__ void clear_kernel(uint4* p, int n16, int n16_all) {
  pdl_launch_dependents();
  pdl_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n16_all; i += gridDim.x * blockDim.x) {
    const uint32_t x = i < n16 ? 0u : NO_PARTIAL;
    p[i] = make_uint4(x, x, x, x);
  }
}

// `keep_status`: leave the status block alone (a later part of one logical call must not wipe
// an error an earlier part recorded).
static cudaError_t launch_clear(uint8_t* ws, const WorkspaceLayout& w, cudaStream_t s,
                                bool keep_status = false) {
  const size_t from = keep_status ? w.off_counters : w.off_status;
  const int n16 = static_cast<int>((w.off_partials - from) / 16);
  const int n16_all = static_cast<int>((w.off_lse - from) / 16);
  const int blocks = n16_all > 256 * 148 ? 148 : (n16_all + 255) / 256;
  return launch_pdl(clear_kernel, dim3(blocks), dim3(256), 0, s,
                    reinterpret_cast<uint4*>(ws + from), n16, n16_all);
}

// Zeroes the status block alone.  Entry points that run several single-sequence steps on one
// workspace do this once, up front, and then run every step with keep_status set, so that the
// block ends up holding the first error of any step.
static cudaError_t clear_status(void* ws, cudaStream_t s) {
  return cudaMemsetAsync(ws, 0, STATUS_BYTES, s);
}

static bool workspace_ok(const void* ws, size_t bytes, size_t need) {
  return ws && (reinterpret_cast<uintptr_t>(ws) & 255) == 0 && bytes >= need;
}

WorkspaceLayout make_layout(const ScorePlan& p, int B, int Hq, int n, bool need_vote,
                            bool need_pooled) {
  WorkspaceLayout w;
  size_t off = 0;
  w.off_status = off;
  off += STATUS_BYTES;
  w.off_counters = off;
  off = align_up(off + sizeof(int) * static_cast<size_t>(p.units), 256);
  w.off_partials = off;
  off = align_up(off + sizeof(float) * static_cast<size_t>(p.units) * p.maxseg * MAX_COLS, 256);
  w.off_lse = off;
  off = align_up(off + sizeof(float) * static_cast<size_t>(p.units) * MAX_COLS, 256);
  w.off_vote = off;
  const size_t row_bytes = sizeof(float) * static_cast<size_t>(B) * Hq * (n > 0 ? n : 0);
  if (need_vote) off = align_up(off + row_bytes, 256);
  w.off_pooled = off;
  if (need_pooled) off = align_up(off + select_scratch_bytes(B * Hq, n), 256);
  w.total = off;
  return w;
}

static thread_local int g_last_launches = 0;

static std::atomic<unsigned long long> g_wait_limit_ns{1000ull * 1000ull * 1000ull};
unsigned long long wait_limit_setting() { return g_wait_limit_ns.load(std::memory_order_relaxed); }

// Side streams (one per direction) and events of snapkv_compress_host, one set per device, created
// on first use and kept for the life of the process (nullptr if they cannot be created: the entry
// point then copies on the caller's stream).  `mu` is held while a call enqueues its work: an event
// belongs to one call from its record to the wait for it.
constexpr int HOST_PARTS = 8;
struct HostSide {
  std::mutex mu;
  cudaStream_t in, back;
  cudaEvent_t start, done;
  cudaEvent_t arrived[HOST_PARTS], computed[HOST_PARTS];
};
static HostSide* host_side() {
  constexpr int MAX_DEV = 64;
  static std::mutex mu;
  static HostSide* table[MAX_DEV] = {};
  static bool failed[MAX_DEV] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (table[dev] || failed[dev]) return table[dev];
  HostSide* h = new HostSide();
  bool ok = cudaStreamCreateWithFlags(&h->in, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&h->back, cudaStreamNonBlocking) == cudaSuccess;
  auto event = [](cudaEvent_t* e) { return cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess; };
  for (int i = 0; ok && i < HOST_PARTS; ++i) ok = event(&h->arrived[i]) && event(&h->computed[i]);
  ok = ok && event(&h->start) && event(&h->done);
  if (!ok) {
    failed[dev] = true;
    delete h;
    return nullptr;
  }
  table[dev] = h;
  return h;
}

static snapkv_status_t check_common(int B, int Hq, int Hkv, int L, int d, int W) {
  if (B < 1 || Hq < 1 || Hkv < 1 || L < 1 || d < 1 || W < 1) return SNAPKV_ERR_INVALID_ARG;
  if (Hq % Hkv != 0 || W > L) return SNAPKV_ERR_INVALID_ARG;
  if (d != 64 && d != 128) return SNAPKV_ERR_UNSUPPORTED;
  if (W > MAX_COLS) return SNAPKV_ERR_UNSUPPORTED;
  if (static_cast<double>(B) * Hkv * L * d >= 1099511627776.0) return SNAPKV_ERR_UNSUPPORTED;
  if (static_cast<double>(B) * Hq * L >= 2147483647.0 * 16) return SNAPKV_ERR_UNSUPPORTED;
  return SNAPKV_OK;
}

static snapkv_status_t check_pool(int pool_kernel, int pool_type) {
  if (pool_kernel < 1 || (pool_kernel & 1) == 0) return SNAPKV_ERR_INVALID_ARG;
  if (pool_type != SNAPKV_POOL_MAX && pool_type != SNAPKV_POOL_AVG) return SNAPKV_ERR_INVALID_ARG;
  if (pool_kernel > 63) return SNAPKV_ERR_UNSUPPORTED;
  return SNAPKV_OK;
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// out[i] = log sum_r exp(parts[r][i]), folded in the order of r (the same on every rank).
__global__ void lse_merge_kernel(const float* __restrict__ parts, int R, int count, float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  float M = -INFINITY, S = 0.f;
  for (int r = 0; r < R; ++r) {
    const float p = parts[static_cast<size_t>(r) * count + i];
    const float Mn = fmaxf(fmaxf(M, p), -1e30f);
    S = S * expf(M - Mn) + expf(p - Mn);
    M = Mn;
  }
  out[i] = M + logf(S);
}

}  // namespace snapkv

using namespace snapkv;

extern "C" {

const char* snapkv_status_string(int status) {
  switch (status) {
    case SNAPKV_OK: return "SNAPKV_OK";
    case SNAPKV_ERR_INVALID_ARG: return "SNAPKV_ERR_INVALID_ARG";
    case SNAPKV_ERR_UNSUPPORTED: return "SNAPKV_ERR_UNSUPPORTED";
    case SNAPKV_ERR_WORKSPACE: return "SNAPKV_ERR_WORKSPACE";
    case SNAPKV_ERR_CUDA: return "SNAPKV_ERR_CUDA";
    case SNAPKV_ERR_TIMEOUT: return "SNAPKV_ERR_TIMEOUT";
    default: return "SNAPKV_UNKNOWN_STATUS";
  }
}

int snapkv_out_rows(int L, int budget) { return budget < L ? budget : L; }

int snapkv_last_launch_count(void) { return g_last_launches; }

size_t snapkv_workspace_size(int B, int Hq, int Hkv, int L, int d, int W, int pool_kernel,
                             int pool_type, int budget) {
  if (check_common(B, Hq, Hkv, L, d, W) != SNAPKV_OK) return 0;
  if (check_pool(pool_kernel, pool_type) != SNAPKV_OK) return 0;
  if (budget <= W) return 0;
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, L, d, W, &p)) return 0;
  const int n = L - W;
  return make_layout(p, B, Hq, n, true, select_needs_scratch(n)).total;
}

size_t snapkv_pool_topk_workspace_size(int rows, int n) {
  if (rows < 1 || n < 1) return 0;
  return select_scratch_bytes(rows, n);
}

static snapkv_status_t window_scores_impl(const void* q_obs, const void* k, const float* lse_obs,
                                          int B, int Hq, int Hkv, int L, int d, int W,
                                          float* out_vote, void* workspace,
                                          size_t workspace_bytes, void* stream) {
  snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
  if (st != SNAPKV_OK) return st;
  if (W >= L) return SNAPKV_ERR_INVALID_ARG;
  if (!q_obs || !k || !out_vote) return SNAPKV_ERR_INVALID_ARG;
  if (!aligned16(q_obs) || !aligned16(k) || (reinterpret_cast<uintptr_t>(out_vote) & 3))
    return SNAPKV_ERR_INVALID_ARG;
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, L, d, W, &p)) return SNAPKV_ERR_UNSUPPORTED;
  const WorkspaceLayout w = make_layout(p, B, Hq, L - W, false, false);
  if (!workspace_ok(workspace, workspace_bytes, w.total)) return SNAPKV_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // with a supplied normaliser the conversion kernel clears what the clear kernel would
  int launches = 0;
  if (!lse_obs) {
    if (launch_clear(ws, w, s) != cudaSuccess) return SNAPKV_ERR_CUDA;
    launches = 1;
  }
  cudaError_t e = launch_window_scores(
      q_obs, k, dense_strides(Hkv, L, d), B, Hq, Hkv, L, d, W, p, out_vote, reinterpret_cast<int*>(ws + w.off_status),
      reinterpret_cast<int*>(ws + w.off_counters), reinterpret_cast<float*>(ws + w.off_partials),
      reinterpret_cast<float*>(ws + w.off_lse), s, &launches, lse_obs);
  if (e != cudaSuccess) return SNAPKV_ERR_CUDA;
  g_last_launches = launches;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_window_scores(const void* q_obs, const void* k, int B, int Hq, int Hkv,
                                     int L, int d, int W, float* out_vote, void* workspace,
                                     size_t workspace_bytes, void* stream) {
  return window_scores_impl(q_obs, k, nullptr, B, Hq, Hkv, L, d, W, out_vote, workspace,
                            workspace_bytes, stream);
}

snapkv_status_t snapkv_window_scores_lse(const void* q_obs, const void* k, const float* lse_obs,
                                         int B, int Hq, int Hkv, int L, int d, int W,
                                         float* out_vote, void* workspace, size_t workspace_bytes,
                                         void* stream) {
  if (!lse_obs || (reinterpret_cast<uintptr_t>(lse_obs) & 3)) return SNAPKV_ERR_INVALID_ARG;
  return window_scores_impl(q_obs, k, lse_obs, B, Hq, Hkv, L, d, W, out_vote, workspace,
                            workspace_bytes, stream);
}

snapkv_status_t snapkv_pool_topk(const float* vote, int rows, int n, int pool_kernel, int pool_type,
                                 int ksel, int32_t* out_idx, void* workspace,
                                 size_t workspace_bytes, void* stream) {
  if (rows < 1 || n < 1 || ksel < 1 || ksel > n || !vote || !out_idx) return SNAPKV_ERR_INVALID_ARG;
  snapkv_status_t st = check_pool(pool_kernel, pool_type);
  if (st != SNAPKV_OK) return st;
  const size_t need = snapkv_pool_topk_workspace_size(rows, n);
  if (need > 0 &&
      (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need))
    return SNAPKV_ERR_WORKSPACE;
  int launches = 0;
  cudaError_t e = launch_pool_topk(vote, rows, n, pool_kernel, pool_type, ksel, out_idx,
                                   static_cast<float*>(workspace),
                                   static_cast<cudaStream_t>(stream), &launches);
  return e == cudaSuccess ? SNAPKV_OK : SNAPKV_ERR_CUDA;
}

snapkv_status_t snapkv_gather(const void* k, const void* v, const int32_t* idx, int B, int Hq,
                              int Hkv, int L, int d, int W, int ksel, void* out_k, void* out_v,
                              void* stream) {
  snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
  if (st != SNAPKV_OK) return st;
  if (ksel < 0 || ksel > L - W || !k || !v || !out_k || !out_v || (ksel > 0 && !idx))
    return SNAPKV_ERR_INVALID_ARG;
  if (!aligned16(k) || !aligned16(v) || !aligned16(out_k) || !aligned16(out_v))
    return SNAPKV_ERR_INVALID_ARG;
  int launches = 0;
  const KVStrides ds = dense_strides(Hkv, L, d);
  cudaError_t e = launch_gather(k, v, ds, ds, idx, B, Hq, Hkv, L, d, W, ksel, ksel + W, out_k,
                                out_v, static_cast<cudaStream_t>(stream), &launches);
  return e == cudaSuccess ? SNAPKV_OK : SNAPKV_ERR_CUDA;
}

static snapkv_status_t compress_impl(const void* q_obs, const void* k, const void* v, int B, int Hq,
                                     int Hkv, int L, int d, int W, int pool_kernel, int pool_type,
                                     int budget, void* out_k, void* out_v, int32_t* out_idx,
                                     void* workspace, size_t workspace_bytes, void* stream,
                                     bool keep_status, const float* lse_obs = nullptr,
                                     const KVStrides* k_str = nullptr,
                                     const KVStrides* v_str = nullptr, bool grouped = false,
                                     const PagedKV* paged = nullptr, bool host_part = false) {
  snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
  if (st != SNAPKV_OK) return st;
  st = check_pool(pool_kernel, pool_type);
  if (st != SNAPKV_OK) return st;
  if (budget <= W) return SNAPKV_ERR_INVALID_ARG;
  if (!q_obs || !k || !v || !out_k || !out_v) return SNAPKV_ERR_INVALID_ARG;
  if (!aligned16(q_obs) || !aligned16(k) || !aligned16(v) || !aligned16(out_k) || !aligned16(out_v))
    return SNAPKV_ERR_INVALID_ARG;
  const int n = L - W;
  if (!out_idx && n > 0) return SNAPKV_ERR_INVALID_ARG;
  const KVStrides ks = k_str ? *k_str : dense_strides(Hkv, L, d);
  const KVStrides vs = v_str ? *v_str : dense_strides(Hkv, L, d);
  // shared selection: the votes of a group's query heads are summed when the select kernel
  // loads them, and the cache keeps Hkv heads
  const int Ho = grouped ? Hkv : Hq;
  const int gsum = grouped ? Hq / Hkv : 1;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int launches = 0;
  if (budget >= L) {
    // Listing 1's early return: nothing is dropped, the cache is expanded to Hq heads.
    if (launch_iota_idx(out_idx, B * Ho, n, budget - W, s, &launches) != cudaSuccess)
      return SNAPKV_ERR_CUDA;
    if (launch_gather(k, v, ks, vs, nullptr, B, Ho, Hkv, L, d, W, n, budget, out_k, out_v, s,
                      &launches, paged) != cudaSuccess)
      return SNAPKV_ERR_CUDA;
    // no kernel of this path can time out, but a caller that passes a workspace may read its
    // status afterwards: it must not find what an earlier use of the memory left there
    if (!keep_status && workspace_ok(workspace, workspace_bytes, STATUS_BYTES) &&
        clear_status(workspace, s) != cudaSuccess)
      return SNAPKV_ERR_CUDA;
    g_last_launches = launches;
    return SNAPKV_OK;
  }
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, L, d, W, &p)) return SNAPKV_ERR_UNSUPPORTED;
  const bool scratch = select_needs_scratch(n);
  const WorkspaceLayout w = make_layout(p, B, Hq, n, true, scratch);
  if (!workspace_ok(workspace, workspace_bytes, w.total)) return SNAPKV_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  if (!lse_obs) {
    if (launch_clear(ws, w, s, keep_status) != cudaSuccess) return SNAPKV_ERR_CUDA;
    launches += 1;
  }
  float* vote = reinterpret_cast<float*>(ws + w.off_vote);
  const int ksel = budget - W;
  if (launch_window_scores(q_obs, k, ks, B, Hq, Hkv, L, d, W, p, vote,
                           reinterpret_cast<int*>(ws + w.off_status),
                           reinterpret_cast<int*>(ws + w.off_counters),
                           reinterpret_cast<float*>(ws + w.off_partials),
                           reinterpret_cast<float*>(ws + w.off_lse), s, &launches, lse_obs,
                           keep_status, false, paged, nullptr, false, host_part) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  if (launch_pool_topk(vote, B * Ho, n, pool_kernel, pool_type, ksel, out_idx,
                       scratch ? reinterpret_cast<float*>(ws + w.off_pooled) : nullptr, s,
                       &launches, gsum, /*vote_is_scratch=*/true) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  if (launch_gather(k, v, ks, vs, out_idx, B, Ho, Hkv, L, d, W, ksel, budget, out_k, out_v, s,
                    &launches, paged) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  g_last_launches = launches;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_compress(const void* q_obs, const void* k, const void* v, int B, int Hq,
                                int Hkv, int L, int d, int W, int pool_kernel, int pool_type,
                                int budget, void* out_k, void* out_v, int32_t* out_idx,
                                void* workspace, size_t workspace_bytes, void* stream) {
  return compress_impl(q_obs, k, v, B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget, out_k,
                       out_v, out_idx, workspace, workspace_bytes, stream, false);
}

snapkv_status_t snapkv_compress_lse(const void* q_obs, const void* k, const void* v,
                                    const float* lse_obs, int B, int Hq, int Hkv, int L, int d,
                                    int W, int pool_kernel, int pool_type, int budget, void* out_k,
                                    void* out_v, int32_t* out_idx, void* workspace,
                                    size_t workspace_bytes, void* stream) {
  if (!lse_obs || (reinterpret_cast<uintptr_t>(lse_obs) & 3)) return SNAPKV_ERR_INVALID_ARG;
  return compress_impl(q_obs, k, v, B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget, out_k,
                       out_v, out_idx, workspace, workspace_bytes, stream, false, lse_obs);
}

// One stride triple of snapkv_compress_strided: positive, whole 16-byte vectors, rows of d
// elements do not overlap, and within what a tensor map can address (byte stride < 2^40).
static bool strides_ok(const int64_t* st, int d, KVStrides* out) {
  if (!st) return false;
  for (int i = 0; i < 3; ++i)
    if (st[i] <= 0 || (st[i] & 7) != 0 || st[i] >= (1ll << 39)) return false;
  if (st[2] < d) return false;
  out->b = st[0];
  out->h = st[1];
  out->l = st[2];
  return true;
}

snapkv_status_t snapkv_compress_strided(const void* q_obs, const void* k, const void* v,
                                        const int64_t* k_strides, const int64_t* v_strides,
                                        const float* lse_obs, int B, int Hq, int Hkv, int L,
                                        int d, int W, int pool_kernel, int pool_type, int budget,
                                        void* out_k, void* out_v, int32_t* out_idx,
                                        void* workspace, size_t workspace_bytes, void* stream) {
  KVStrides ks, vs;
  if (!strides_ok(k_strides, d, &ks) || !strides_ok(v_strides, d, &vs))
    return SNAPKV_ERR_INVALID_ARG;
  if (lse_obs && (reinterpret_cast<uintptr_t>(lse_obs) & 3)) return SNAPKV_ERR_INVALID_ARG;
  return compress_impl(q_obs, k, v, B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget, out_k,
                       out_v, out_idx, workspace, workspace_bytes, stream, false, lse_obs, &ks,
                       &vs);
}

snapkv_status_t snapkv_compress_grouped(const void* q_obs, const void* k, const void* v,
                                        const int64_t* k_strides, const int64_t* v_strides,
                                        const float* lse_obs, int B, int Hq, int Hkv, int L,
                                        int d, int W, int pool_kernel, int pool_type, int budget,
                                        void* out_k, void* out_v, int32_t* out_idx,
                                        void* workspace, size_t workspace_bytes, void* stream) {
  KVStrides ks, vs;
  if ((k_strides && !strides_ok(k_strides, d, &ks)) || (v_strides && !strides_ok(v_strides, d, &vs)))
    return SNAPKV_ERR_INVALID_ARG;
  if (lse_obs && (reinterpret_cast<uintptr_t>(lse_obs) & 3)) return SNAPKV_ERR_INVALID_ARG;
  return compress_impl(q_obs, k, v, B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget, out_k,
                       out_v, out_idx, workspace, workspace_bytes, stream, false, lse_obs,
                       k_strides ? &ks : nullptr, v_strides ? &vs : nullptr, true);
}

// ---- prompts of different lengths
// The sequences are independent (Sec. 4.1).  Those longer than the budget are scored and selected
// in groups of up to RAGGED_MAX, each group in one set of launches; a group is as large as the
// workspace allows, one sequence always fits.  One gather launch then serves up to RAGGED_MAX
// consecutive sequences, those that are copied through included.
static void ragged_layout(RaggedBatch* rb, int Hq) {
  size_t off = STATUS_BYTES;
  const size_t units = static_cast<size_t>(rb->plan[0].units);
  rb->off_counters = off;
  off = align_up(off + sizeof(int) * units * rb->count, 256);
  rb->off_partials = off;
  long long slots = 0, votes = 0;
  for (int i = 0; i < rb->count; ++i) {
    rb->part0[i] = slots;
    slots += static_cast<long long>(units) * rb->plan[i].maxseg;
    rb->vote0[i] = votes;
    votes += static_cast<long long>(Hq) * rb->plan[i].n_vote;
  }
  off = align_up(off + sizeof(float) * static_cast<size_t>(slots) * MAX_COLS, 256);
  rb->off_lse = off;
  off = align_up(off + sizeof(float) * units * rb->count * MAX_COLS, 256);
  rb->off_vote = off;
  rb->total = align_up(off + sizeof(float) * static_cast<size_t>(votes), 256);
}

// The group of sequences longer than the budget that starts at or behind sequence `b`; returns the
// sequence behind it.
static int ragged_group(const int32_t* lens, int B, int b, int Hq, int Hkv, int d, int W, int budget,
                        size_t workspace_bytes, RaggedBatch* rb) {
  rb->count = 0;
  rb->total = 0;
  int waves = 0, upw = 1;
  for (; b < B; ++b) {
    if (budget >= lens[b]) continue;
    if (rb->count == RAGGED_MAX) break;
    const int i = rb->count;
    if (!make_score_plan(1, Hq, Hkv, lens[b], d, W, &rb->plan[i])) break;
    // (with supplied normalisers a sequence is one wave of all its units)
    if (rb->plan[i].units > upw) upw = rb->plan[i].units;
    waves += rb->plan[i].nwaves;
    if (waves > most_waves_per_launch(upw)) break;
    rb->L[i] = lens[b];
    rb->batch[i] = b;
    rb->count = i + 1;
    ragged_layout(rb, Hq);
    if (i > 0 && rb->total > workspace_bytes) {
      rb->count = i;
      ragged_layout(rb, Hq);
      break;
    }
  }
  return b;
}

// Whether sequences of these lengths can share launches at all (one too long, or a pooling radius that
// the cluster kernel does not take, and each goes through by itself).
static bool ragged_shares_launches(const int32_t* lens, int B, int Hq, int Hkv, int d, int W, int pool_kernel,
                                   int pool_type, int budget) {
  int longest = 0;
  for (int b = 0; b < B; ++b)
    if (lens[b] > longest) longest = lens[b];
  if (Hq > 65535 || !ragged_select_applies(longest - W > 0 ? longest - W : 1, pool_kernel, pool_type)) return false;
  ScorePlan p;  // the longest sequence has the most waves
  return longest <= budget ||
         (make_score_plan(1, Hq, Hkv, longest, d, W, &p) && p.nwaves <= most_waves_per_launch(p.units));
}

struct RaggedCall {
  const void *q_obs, *k, *v;
  KVStrides ks, vs;
  const int64_t *k_off, *v_off;  // per sequence, or nullptr: b * stride
  const int32_t* lens;
  const float* lse_obs;
  int B, Hq, Hkv, d, W, pool_kernel, pool_type, budget;
  void *out_k, *out_v;
  int32_t* out_idx;
  void* workspace;
  size_t workspace_bytes;
  cudaStream_t stream;
  const PagedKV* paged;
  bool fill;
};

// Lengths and workspace, before anything is launched.
static snapkv_status_t ragged_check(const RaggedCall& c, int Lmax) {
  for (int b = 0; b < c.B; ++b) {
    if (c.lens[b] < c.W || c.lens[b] > Lmax) return SNAPKV_ERR_INVALID_ARG;
    if (c.k_off && (c.k_off[b] < 0 || (c.k_off[b] & 7))) return SNAPKV_ERR_INVALID_ARG;
    if (c.v_off && (c.v_off[b] < 0 || (c.v_off[b] & 7))) return SNAPKV_ERR_INVALID_ARG;
    if (!c.out_idx && c.lens[b] > c.W) return SNAPKV_ERR_INVALID_ARG;
  }
  for (int b = 0; b < c.B; ++b) {
    if (c.budget >= c.lens[b]) continue;  // copied through: no scratch
    const size_t need =
        snapkv_workspace_size(1, c.Hq, c.Hkv, c.lens[b], c.d, c.W, c.pool_kernel, c.pool_type, c.budget);
    if (need == 0) return SNAPKV_ERR_INVALID_ARG;
    if (!workspace_ok(c.workspace, c.workspace_bytes, need)) return SNAPKV_ERR_WORKSPACE;
  }
  return SNAPKV_OK;
}

static snapkv_status_t ragged_impl(const RaggedCall& c) {
  const size_t head_rows = static_cast<size_t>(c.Hq) * c.budget * c.d * 2;  // bytes of one sequence's out_k
  const bool have_ws = workspace_ok(c.workspace, c.workspace_bytes, STATUS_BYTES);
  int launches = 0;
  if (c.out_idx && ragged_shares_launches(c.lens, c.B, c.Hq, c.Hkv, c.d, c.W, c.pool_kernel, c.pool_type, c.budget)) {
    uint8_t* ws = static_cast<uint8_t*>(c.workspace);
    bool first = true;  // the first group's launches clear the status block, later ones leave it
    for (int b = 0; b < c.B;) {
      RaggedBatch rb;
      b = ragged_group(c.lens, c.B, b, c.Hq, c.Hkv, c.d, c.W, c.budget, c.workspace_bytes, &rb);
      if (rb.count == 0) {
        if (b < c.B) return SNAPKV_ERR_UNSUPPORTED;  // no plan for sequence b
        break;
      }
      for (int i = 0; i < rb.count; ++i)
        rb.k_off[i] = c.paged ? 0 : (c.k_off ? c.k_off[rb.batch[i]] : rb.batch[i] * c.ks.b);
      if (launch_ragged_scores(rb, c.q_obs, c.k, c.ks, c.B, c.Hq, c.Hkv, c.d, c.W, ws, c.stream, &launches,
                               c.lse_obs, !first, c.paged) != cudaSuccess)
        return SNAPKV_ERR_CUDA;
      if (launch_ragged_select(rb, reinterpret_cast<const float*>(ws + rb.off_vote), c.Hq, c.W, c.pool_kernel,
                               c.pool_type, c.budget - c.W, c.out_idx, reinterpret_cast<int*>(ws) + STATUS_READY, c.stream,
                               &launches) != cudaSuccess)
        return SNAPKV_ERR_CUDA;
      first = false;
    }
    if (first && have_ws && clear_status(c.workspace, c.stream) != cudaSuccess) return SNAPKV_ERR_CUDA;
    const int most = 65535 / c.Hq < RAGGED_MAX ? 65535 / c.Hq : RAGGED_MAX;
    for (int b0 = 0; b0 < c.B; b0 += most) {
      const int count = c.B - b0 < most ? c.B - b0 : most;
      long long ko[RAGGED_MAX], vo[RAGGED_MAX];
      for (int i = 0; i < count; ++i) {
        ko[i] = c.k_off ? c.k_off[b0 + i] : (b0 + i) * c.ks.b;
        vo[i] = c.v_off ? c.v_off[b0 + i] : (b0 + i) * c.vs.b;
      }
      if (launch_ragged_gather(c.k, c.v, c.ks, c.vs, c.lens + b0, ko, vo, b0, count, c.Hq, c.Hkv, c.d, c.W, c.budget,
                               c.fill, c.out_idx, c.out_k, c.out_v, c.stream, &launches, c.paged) != cudaSuccess)
        return SNAPKV_ERR_CUDA;
    }
    g_last_launches = launches;
    return SNAPKV_OK;
  }
  // pooling radii or lengths that the shared select launch does not take: one single-sequence step
  // each, one after the other on the same stream and workspace; the status block keeps the first
  // error of any of them
  if (have_ws && clear_status(c.workspace, c.stream) != cudaSuccess) return SNAPKV_ERR_CUDA;
  if (c.fill && (cudaMemsetAsync(c.out_k, 0, head_rows * c.B, c.stream) != cudaSuccess ||
                 cudaMemsetAsync(c.out_v, 0, head_rows * c.B, c.stream) != cudaSuccess ||
                 cudaMemsetAsync(c.out_idx, 0xff, sizeof(int32_t) * c.B * c.Hq * (c.budget - c.W), c.stream) != cudaSuccess))
    return SNAPKV_ERR_CUDA;
  for (int b = 0; b < c.B; ++b) {
    const long long ko = c.paged ? 0 : (c.k_off ? c.k_off[b] : b * c.ks.b);
    const long long vo = c.paged ? 0 : (c.v_off ? c.v_off[b] : b * c.vs.b);
    PagedKV one = {};
    if (c.paged) {
      one = *c.paged;
      one.table += static_cast<size_t>(b) * one.pages_per_seq;
    }
    const snapkv_status_t st = compress_impl(
        static_cast<const uint8_t*>(c.q_obs) + static_cast<size_t>(b) * c.Hq * c.W * c.d * 2,
        static_cast<const uint8_t*>(c.k) + ko * 2, static_cast<const uint8_t*>(c.v) + vo * 2, 1, c.Hq, c.Hkv,
        c.lens[b], c.d, c.W, c.pool_kernel, c.pool_type, c.budget, static_cast<uint8_t*>(c.out_k) + b * head_rows,
        static_cast<uint8_t*>(c.out_v) + b * head_rows,
        c.out_idx ? c.out_idx + static_cast<size_t>(b) * c.Hq * (c.budget - c.W) : nullptr, c.workspace,
        c.workspace_bytes, c.stream, /*keep_status=*/true,
        c.lse_obs ? c.lse_obs + static_cast<size_t>(b) * c.Hq * c.W : nullptr, &c.ks, &c.vs, false,
        c.paged ? &one : nullptr);
    if (st != SNAPKV_OK) return st;
    launches += g_last_launches;
  }
  g_last_launches = launches;
  return SNAPKV_OK;
}

size_t snapkv_varlen_workspace_size(const int32_t* seq_lens, int B, int Hq, int Hkv, int d, int W, int pool_kernel,
                                    int pool_type, int budget) {
  if (!seq_lens || B < 1 || check_pool(pool_kernel, pool_type) != SNAPKV_OK || budget <= W) return 0;
  size_t need = STATUS_BYTES;
  for (int b = 0; b < B; ++b) {
    if (check_common(1, Hq, Hkv, seq_lens[b], d, W) != SNAPKV_OK) return 0;
    if (seq_lens[b] <= budget) continue;
    const size_t one = snapkv_workspace_size(1, Hq, Hkv, seq_lens[b], d, W, pool_kernel, pool_type, budget);
    if (one == 0) return 0;
    if (one > need) need = one;
  }
  if (!ragged_shares_launches(seq_lens, B, Hq, Hkv, d, W, pool_kernel, pool_type, budget)) return need;
  for (int b = 0; b < B;) {
    RaggedBatch rb;
    b = ragged_group(seq_lens, B, b, Hq, Hkv, d, W, budget, ~static_cast<size_t>(0), &rb);
    if (rb.count == 0) break;
    if (rb.total > need) need = rb.total;
  }
  return need;
}

snapkv_status_t snapkv_binding_varlen(const void* q_obs, const void* k, const void* v, const int64_t* k_strides,
                                      const int64_t* v_strides, const int64_t* k_seq_offsets,
                                      const int64_t* v_seq_offsets, const int32_t* seq_lens, const float* lse_obs,
                                      int B, int Hq, int Hkv, int Lmax, int d, int W, int pool_kernel, int pool_type,
                                      int budget, void* out_k, void* out_v, int32_t* out_idx, void* workspace,
                                      size_t workspace_bytes, void* stream, int fill) {
  snapkv_status_t st = check_common(B, Hq, Hkv, Lmax, d, W);
  if (st != SNAPKV_OK) return st;
  if (!seq_lens || budget <= W || !q_obs || !k || !v || !out_k || !out_v) return SNAPKV_ERR_INVALID_ARG;
  KVStrides ks = dense_strides(Hkv, Lmax, d), vs = ks;
  if ((k_strides && !strides_ok(k_strides, d, &ks)) || (v_strides && !strides_ok(v_strides, d, &vs)))
    return SNAPKV_ERR_INVALID_ARG;
  if (lse_obs && (reinterpret_cast<uintptr_t>(lse_obs) & 3)) return SNAPKV_ERR_INVALID_ARG;
  // every sequence, every pointer and the workspace are checked before the first launch
  st = check_pool(pool_kernel, pool_type);
  if (st != SNAPKV_OK) return st;
  if (!aligned16(q_obs) || !aligned16(k) || !aligned16(v) || !aligned16(out_k) || !aligned16(out_v))
    return SNAPKV_ERR_INVALID_ARG;
  const RaggedCall c = {q_obs, k, v, ks, vs, k_seq_offsets, v_seq_offsets, seq_lens, lse_obs, B, Hq, Hkv, d, W,
                        pool_kernel, pool_type, budget, out_k, out_v, out_idx, workspace, workspace_bytes,
                        static_cast<cudaStream_t>(stream), nullptr, fill != 0};
  st = ragged_check(c, Lmax);
  return st != SNAPKV_OK ? st : ragged_impl(c);
}

snapkv_status_t snapkv_compress_varlen(const void* q_obs, const void* k, const void* v,
                                       const int64_t* k_strides, const int64_t* v_strides,
                                       const int64_t* k_seq_offsets, const int64_t* v_seq_offsets,
                                       const int32_t* seq_lens, const float* lse_obs, int B,
                                       int Hq, int Hkv, int Lmax, int d, int W, int pool_kernel,
                                       int pool_type, int budget, void* out_k, void* out_v,
                                       int32_t* out_idx, void* workspace, size_t workspace_bytes,
                                       void* stream) {
  return snapkv_binding_varlen(q_obs, k, v, k_strides, v_strides, k_seq_offsets, v_seq_offsets, seq_lens, lse_obs, B,
                               Hq, Hkv, Lmax, d, W, pool_kernel, pool_type, budget, out_k, out_v, out_idx, workspace,
                               workspace_bytes, stream, 0);
}

snapkv_status_t snapkv_binding_paged(const void* q_obs, const void* k_pool, const void* v_pool,
                                     const int64_t* k_strides, const int64_t* v_strides, const int32_t* page_table,
                                     int pages_per_seq, int page_size, int num_pages, const int32_t* seq_lens,
                                     const float* lse_obs, int B, int Hq, int Hkv, int L, int d, int W,
                                     int pool_kernel, int pool_type, int budget, void* out_k, void* out_v,
                                     int32_t* out_idx, void* workspace, size_t workspace_bytes, void* stream,
                                     int fill) {
  snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
  if (st != SNAPKV_OK) return st;
  st = check_pool(pool_kernel, pool_type);
  if (st != SNAPKV_OK) return st;
  if (budget <= W || !q_obs || !k_pool || !v_pool || !out_k || !out_v || !page_table)
    return SNAPKV_ERR_INVALID_ARG;
  if (!aligned16(q_obs) || !aligned16(k_pool) || !aligned16(v_pool) || !aligned16(out_k) ||
      !aligned16(out_v) || (reinterpret_cast<uintptr_t>(page_table) & 3))
    return SNAPKV_ERR_INVALID_ARG;
  if (lse_obs && (reinterpret_cast<uintptr_t>(lse_obs) & 3)) return SNAPKV_ERR_INVALID_ARG;
  // a tile of TILE_KEYS keys must lie inside one page
  if (page_size < TILE_KEYS || page_size % TILE_KEYS != 0 || num_pages < 1 || pages_per_seq < 1)
    return SNAPKV_ERR_INVALID_ARG;
  if (static_cast<long long>(pages_per_seq) * page_size < L) return SNAPKV_ERR_INVALID_ARG;
  KVStrides ks, vs;
  if (!strides_ok(k_strides, d, &ks) || !strides_ok(v_strides, d, &vs)) return SNAPKV_ERR_INVALID_ARG;
  const PagedKV paged = {page_table, pages_per_seq, page_size, num_pages};
  if (!seq_lens)
    return compress_impl(q_obs, k_pool, v_pool, B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget,
                         out_k, out_v, out_idx, workspace, workspace_bytes, stream, false, lse_obs,
                         &ks, &vs, false, &paged);
  const RaggedCall c = {q_obs, k_pool, v_pool, ks, vs, nullptr, nullptr, seq_lens, lse_obs, B, Hq, Hkv, d, W,
                        pool_kernel, pool_type, budget, out_k, out_v, out_idx, workspace, workspace_bytes,
                        static_cast<cudaStream_t>(stream), &paged, fill != 0};
  st = ragged_check(c, L);
  return st != SNAPKV_OK ? st : ragged_impl(c);
}

snapkv_status_t snapkv_compress_paged(const void* q_obs, const void* k_pool, const void* v_pool,
                                      const int64_t* k_strides, const int64_t* v_strides,
                                      const int32_t* page_table, int pages_per_seq, int page_size,
                                      int num_pages, const int32_t* seq_lens, const float* lse_obs,
                                      int B, int Hq, int Hkv, int L, int d, int W, int pool_kernel,
                                      int pool_type, int budget, void* out_k, void* out_v,
                                      int32_t* out_idx, void* workspace, size_t workspace_bytes,
                                      void* stream) {
  return snapkv_binding_paged(q_obs, k_pool, v_pool, k_strides, v_strides, page_table, pages_per_seq, page_size,
                              num_pages, seq_lens, lse_obs, B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget,
                              out_k, out_v, out_idx, workspace, workspace_bytes, stream, 0);
}

// ---- a prompt sharded along its length over several GPUs: the per-shard steps
static snapkv_status_t shard_common(const void* q_obs, const void* k_shard, int B, int Hq, int Hkv,
                                    int Ls, int d, int W) {
  snapkv_status_t st = check_common(B, Hq, Hkv, Ls, d, W);
  if (st != SNAPKV_OK) return st;
  if (!q_obs || !k_shard || !aligned16(q_obs) || !aligned16(k_shard)) return SNAPKV_ERR_INVALID_ARG;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_shard_lse(const void* q_obs, const void* k_shard, int B, int Hq, int Hkv,
                                 int Ls, int d, int W, int mask_n, float* out_lse, void* workspace,
                                 size_t workspace_bytes, void* stream) {
  snapkv_status_t st = shard_common(q_obs, k_shard, B, Hq, Hkv, Ls, d, W);
  if (st != SNAPKV_OK) return st;
  if (!out_lse || (reinterpret_cast<uintptr_t>(out_lse) & 3)) return SNAPKV_ERR_INVALID_ARG;
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, Ls, d, W, &p)) return SNAPKV_ERR_UNSUPPORTED;
  const WorkspaceLayout w = make_layout(p, B, Hq, 0, false, false);
  if (!workspace_ok(workspace, workspace_bytes, w.total)) return SNAPKV_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (launch_clear(ws, w, s) != cudaSuccess) return SNAPKV_ERR_CUDA;
  int launches = 1;
  const ShardMode shard = {mask_n, out_lse};
  if (launch_window_scores(q_obs, k_shard, dense_strides(Hkv, Ls, d), B, Hq, Hkv, Ls, d, W, p, nullptr,
                           reinterpret_cast<int*>(ws + w.off_status),
                           reinterpret_cast<int*>(ws + w.off_counters),
                           reinterpret_cast<float*>(ws + w.off_partials),
                           reinterpret_cast<float*>(ws + w.off_lse), s, &launches, nullptr, false,
                           false, nullptr, &shard) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  g_last_launches = launches;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_lse_merge(const float* parts, int R, int count, float* out, void* stream) {
  if (!parts || !out || R < 1 || count < 1) return SNAPKV_ERR_INVALID_ARG;
  lse_merge_kernel<<<(count + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(parts, R, count, out);
  g_last_launches = 1;
  return cudaGetLastError() == cudaSuccess ? SNAPKV_OK : SNAPKV_ERR_CUDA;
}

snapkv_status_t snapkv_shard_votes(const void* q_obs, const void* k_shard, const float* lse_obs,
                                   int B, int Hq, int Hkv, int Ls, int d, int W, int n_vote,
                                   float* out_vote, void* workspace, size_t workspace_bytes,
                                   void* stream) {
  snapkv_status_t st = shard_common(q_obs, k_shard, B, Hq, Hkv, Ls, d, W);
  if (st != SNAPKV_OK) return st;
  if (!lse_obs || !out_vote || n_vote < 1 || n_vote > Ls) return SNAPKV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(lse_obs) & 3) || (reinterpret_cast<uintptr_t>(out_vote) & 3))
    return SNAPKV_ERR_INVALID_ARG;
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, Ls, d, W, &p, n_vote)) return SNAPKV_ERR_UNSUPPORTED;
  const WorkspaceLayout w = make_layout(p, B, Hq, 0, false, false);
  if (!workspace_ok(workspace, workspace_bytes, w.total)) return SNAPKV_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  int launches = 0;
  if (launch_window_scores(q_obs, k_shard, dense_strides(Hkv, Ls, d), B, Hq, Hkv, Ls, d, W, p, out_vote,
                           reinterpret_cast<int*>(ws + w.off_status),
                           reinterpret_cast<int*>(ws + w.off_counters),
                           reinterpret_cast<float*>(ws + w.off_partials),
                           reinterpret_cast<float*>(ws + w.off_lse), static_cast<cudaStream_t>(stream),
                           &launches, lse_obs) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  g_last_launches = launches;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_gather_range(const void* k_shard, const void* v_shard, const int32_t* idx,
                                    int B, int Hq, int Hkv, int Ls, int d, int pos0, int ksel,
                                    int append, void* out_k, void* out_v, int out_rows,
                                    int32_t* seg, void* stream) {
  if (B < 1 || Hq < 1 || Hkv < 1 || Hq % Hkv != 0 || Ls < 1 || (d != 64 && d != 128))
    return SNAPKV_ERR_INVALID_ARG;
  if (pos0 < 0 || ksel < 0 || append < 0 || append > Ls || !k_shard || !v_shard || !out_k || !out_v || !seg ||
      (ksel > 0 && !idx))
    return SNAPKV_ERR_INVALID_ARG;
  if (!aligned16(k_shard) || !aligned16(v_shard) || !aligned16(out_k) || !aligned16(out_v))
    return SNAPKV_ERR_INVALID_ARG;
  if (static_cast<long long>(B) * Hq > 65535) return SNAPKV_ERR_UNSUPPORTED;
  const int most = (ksel < Ls ? ksel : Ls) + append;  // rows a head can get from this shard
  if (out_rows < most) return SNAPKV_ERR_INVALID_ARG;
  int launches = 0;
  const KVStrides ds = dense_strides(Hkv, Ls, d);
  const cudaError_t e = launch_gather_range(k_shard, v_shard, ds, ds, idx, B, Hq, Hkv, Ls, d, pos0, ksel,
                                            append, out_rows, out_k, out_v, seg,
                                            static_cast<cudaStream_t>(stream), &launches);
  g_last_launches = launches;
  return e == cudaSuccess ? SNAPKV_OK : SNAPKV_ERR_CUDA;
}

size_t snapkv_host_staging_size(int B, int Hq, int Hkv, int L, int d, int W, int pool_kernel,
                                int pool_type, int budget) {
  if (check_common(B, Hq, Hkv, L, d, W) != SNAPKV_OK) return 0;
  if (check_pool(pool_kernel, pool_type) != SNAPKV_OK || budget <= W) return 0;
  const size_t qb = align_up(static_cast<size_t>(B) * Hq * W * d * 2, 256);
  const size_t kb = align_up(static_cast<size_t>(B) * Hkv * L * d * 2, 256);
  const size_t ob = align_up(static_cast<size_t>(B) * Hq * budget * d * 2, 256);
  const size_t ib = align_up(static_cast<size_t>(B) * Hq * (budget - W) * 4, 256);
  size_t ws = 0;
  if (budget < L) {
    // the entry point works through the (batch, KV head) pairs in parts, each a problem of
    // its own; the workspace must hold the largest of them (and the whole, if it runs as one)
    ws = snapkv_workspace_size(B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget);
    const int pairs = B * Hkv, g = Hq / Hkv;
    const int parts = pairs < HOST_PARTS ? pairs : HOST_PARTS;
    const int per = (pairs + parts - 1) / parts;
    const int sizes[2] = {per, pairs % per};
    for (int np : sizes)
      if (np > 0) {
        const size_t w1 = snapkv_workspace_size(1, np * g, np, L, d, W, pool_kernel, pool_type, budget);
        if (w1 > ws) ws = w1;
      }
  }
  return qb + 2 * kb + 2 * ob + ib + align_up(ws, 256);
}

snapkv_status_t snapkv_compress_host(const void* q_obs, const void* k, const void* v, int B, int Hq,
                                     int Hkv, int L, int d, int W, int pool_kernel, int pool_type,
                                     int budget, void* out_k, void* out_v, int32_t* out_idx,
                                     void* staging, size_t staging_bytes, void* stream) {
  const size_t need =
      snapkv_host_staging_size(B, Hq, Hkv, L, d, W, pool_kernel, pool_type, budget);
  if (need == 0) {
    snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
    if (st != SNAPKV_OK) return st;
    st = check_pool(pool_kernel, pool_type);
    return st != SNAPKV_OK ? st : SNAPKV_ERR_INVALID_ARG;
  }
  if (!q_obs || !k || !v || !out_k || !out_v || !out_idx) return SNAPKV_ERR_INVALID_ARG;
  if (!staging || (reinterpret_cast<uintptr_t>(staging) & 255) || staging_bytes < need)
    return SNAPKV_ERR_WORKSPACE;
  const size_t q_raw = static_cast<size_t>(B) * Hq * W * d * 2;
  const size_t k_raw = static_cast<size_t>(B) * Hkv * L * d * 2;
  const size_t o_raw = static_cast<size_t>(B) * Hq * budget * d * 2;
  const size_t i_raw = static_cast<size_t>(B) * Hq * (budget - W) * 4;
  uint8_t* p = static_cast<uint8_t*>(staging);
  uint8_t* dq = p; p += align_up(q_raw, 256);
  uint8_t* dk = p; p += align_up(k_raw, 256);
  uint8_t* dv = p; p += align_up(k_raw, 256);
  uint8_t* dok = p; p += align_up(o_raw, 256);
  uint8_t* dov = p; p += align_up(o_raw, 256);
  uint8_t* di = p; p += align_up(i_raw, 256);
  uint8_t* dws = p;
  const size_t ws_bytes = staging_bytes - static_cast<size_t>(dws - static_cast<uint8_t*>(staging));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // The (batch, KV head) pairs are independent: they go through in up to HOST_PARTS parts, with
  // the copies in and the copies back on a stream each, so that a part computes while the next
  // one's keys and values arrive and the previous one's results leave; PCIe carries both directions
  // at once.  What bounds the call is the link: 33.8 MB in and 33.6 MB back at 8192 positions and
  // 2048 kept, both at once at 39 GB/s each (950 us; 1310 with the copies in on the caller's stream).
  const int pairs = B * Hkv, g = Hq / Hkv;
  HostSide* side = host_side();
  std::unique_lock<std::mutex> lock;
  if (side) lock = std::unique_lock<std::mutex>(side->mu);
  int parts = side ? (pairs < HOST_PARTS ? pairs : HOST_PARTS) : 1;
  const int per = (pairs + parts - 1) / parts;
  parts = (pairs + per - 1) / per;
  const size_t q_pair = static_cast<size_t>(g) * W * d * 2, k_pair = static_cast<size_t>(L) * d * 2;
  const size_t o_pair = static_cast<size_t>(g) * budget * d * 2;
  const size_t i_pair = static_cast<size_t>(g) * (budget - W) * 4;
  cudaStream_t in = side ? side->in : s, back = side ? side->back : s;
  // makes `waiter` wait for what `stream` holds by now
  auto order = [](cudaStream_t stream, cudaEvent_t ev, cudaStream_t waiter) {
    return cudaEventRecord(ev, stream) == cudaSuccess && cudaStreamWaitEvent(waiter, ev, 0) == cudaSuccess;
  };
  auto to_device = [&](void* dst, const void* src, size_t at, size_t bytes) {
    return cudaMemcpyAsync(static_cast<uint8_t*>(dst) + at, static_cast<const uint8_t*>(src) + at, bytes,
                           cudaMemcpyHostToDevice, in) == cudaSuccess;
  };
  auto to_host = [&](void* dst, const void* src, size_t at, size_t bytes) {
    return cudaMemcpyAsync(static_cast<uint8_t*>(dst) + at, static_cast<const uint8_t*>(src) + at, bytes,
                           cudaMemcpyDeviceToHost, back) == cudaSuccess;
  };
  int launches = 0;
  // (no workspace part in the staging buffer when the cache is copied through, budget >= L)
  if (workspace_ok(dws, ws_bytes, STATUS_BYTES) && clear_status(dws, s) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  // the staging buffer and the host buffers are the caller's stream's
  if (side && !order(s, side->start, in)) return SNAPKV_ERR_CUDA;
  snapkv_status_t st = SNAPKV_OK;
  if (!to_device(dq, q_obs, 0, q_raw)) st = SNAPKV_ERR_CUDA;
  for (int c = 0; c < parts && st == SNAPKV_OK; ++c) {
    const int p0 = c * per, np = (pairs - p0 < per) ? pairs - p0 : per;
    const size_t qo = p0 * q_pair, ko = p0 * k_pair, oo = p0 * o_pair, io = p0 * i_pair;
    if (!to_device(dk, k, ko, np * k_pair) || !to_device(dv, v, ko, np * k_pair) ||
        (side && !order(in, side->arrived[c], s))) {
      st = SNAPKV_ERR_CUDA;
      break;
    }
    // one part is a problem of its own with batch 1 and np KV heads (the layouts are flat
    // over batch and KV head); the parts share the workspace, which the stream serialises
    st = compress_impl(
        dq + qo, dk + ko, dv + ko, 1, np * g, np, L, d, W, pool_kernel, pool_type, budget,
        dok + oo, dov + oo, reinterpret_cast<int32_t*>(di + io), dws, ws_bytes, stream,
        /*keep_status=*/true, nullptr, nullptr, nullptr, false, nullptr, /*host_part=*/true);
    if (st != SNAPKV_OK) break;
    launches += g_last_launches;
    if ((side && !order(s, side->computed[c], back)) || !to_host(out_k, dok, oo, np * o_pair) ||
        !to_host(out_v, dov, oo, np * o_pair) || !to_host(out_idx, di, io, np * i_pair))
      st = SNAPKV_ERR_CUDA;
  }
  // the caller's stream is complete only when the last copy is, after an error too
  if (side && (!order(in, side->arrived[0], s) || !order(back, side->done, s))) st = SNAPKV_ERR_CUDA;
  if (st != SNAPKV_OK) return st;
  g_last_launches = launches;
  return SNAPKV_OK;
}

int snapkv_schedule_items(int B, int Hq, int Hkv, int L, int d, int W, int votes_only, int grid,
                          int cta, int32_t* out_items, int max_items, int32_t* out_plan) {
  if (check_common(B, Hq, Hkv, L, d, W) != SNAPKV_OK || W >= L) return -1;
  if (grid < 1 || grid > MAX_GRID || cta < 0 || cta >= grid || max_items < 0) return -1;
  if (max_items > 0 && !out_items) return -1;
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, L, d, W, &p)) return -1;
  if (out_plan) {
    out_plan[0] = p.units;
    out_plan[1] = votes_only ? p.units : p.units_per_wave;
    out_plan[2] = votes_only ? 1 : p.nwaves;
    out_plan[3] = p.tiles_stats;
    out_plan[4] = p.tiles_vote;
    out_plan[5] = p.maxseg;
    out_plan[6] = WAVE_LAG;
    out_plan[7] = p.ncols;
  }
  return list_schedule_items(p, L, W, Hkv, votes_only ? 1 : 0, grid, cta, out_items, max_items);
}

int snapkv_binding_shared_fold(int B, int Hq, int Hkv, int L, int d, int W, int host_part) {
  ScorePlan p;
  if (check_common(B, Hq, Hkv, L, d, W) != SNAPKV_OK || !make_score_plan(B, Hq, Hkv, L, d, W, &p)) return -1;
  return shared_fold(p, W, items_per_phase(p.units_per_wave, score_grid()), host_part != 0) ? 1 : 0;
}

int snapkv_binding_ragged_items(const int32_t* seq_lens, int B, int Hq, int Hkv, int d, int W, int votes_only,
                                int grid, int cta, int32_t* out_items, int max_items) {
  if (!seq_lens || B < 1 || max_items < 0 || (max_items > 0 && !out_items)) return -1;
  if (grid < 1 || grid > MAX_GRID || cta < 0 || cta >= grid) return -1;
  for (int b = 0; b < B; ++b)
    if (check_common(1, Hq, Hkv, seq_lens[b], d, W) != SNAPKV_OK || seq_lens[b] <= W) return -1;
  RaggedBatch rb;
  ragged_group(seq_lens, B, 0, Hq, Hkv, d, W, W, ~static_cast<size_t>(0), &rb);
  return rb.count == B ? list_ragged_items(rb, W, Hkv, votes_only ? 1 : 0, grid, cta, out_items, max_items) : -1;
}

unsigned long long snapkv_set_wait_limit_ns(unsigned long long limit_ns) {
  // at least a millisecond: a limit near the length of an ordinary wait would turn a busy
  // memory system into an error
  if (limit_ns < 1000000ull) limit_ns = 1000000ull;
  return g_wait_limit_ns.exchange(limit_ns, std::memory_order_relaxed);
}

snapkv_status_t snapkv_selftest_stalled_scores(const void* q_obs, const void* k, int B, int Hq,
                                               int Hkv, int L, int d, int W, float* out_vote,
                                               void* workspace, size_t workspace_bytes,
                                               void* stream) {
  snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
  if (st != SNAPKV_OK) return st;
  if (W >= L || !q_obs || !k || !out_vote) return SNAPKV_ERR_INVALID_ARG;
  if (!aligned16(q_obs) || !aligned16(k) || (reinterpret_cast<uintptr_t>(out_vote) & 3))
    return SNAPKV_ERR_INVALID_ARG;
  ScorePlan p;
  if (!make_score_plan(B, Hq, Hkv, L, d, W, &p)) return SNAPKV_ERR_UNSUPPORTED;
  const WorkspaceLayout w = make_layout(p, B, Hq, L - W, false, false);
  if (!workspace_ok(workspace, workspace_bytes, w.total)) return SNAPKV_ERR_WORKSPACE;
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int launches = 1;
  // counters cleared and never raised: every unit looks as if its statistics were still
  // on their way, for ever
  if (launch_clear(ws, w, s) != cudaSuccess) return SNAPKV_ERR_CUDA;
  cudaError_t e = launch_window_scores(
      q_obs, k, dense_strides(Hkv, L, d), B, Hq, Hkv, L, d, W, p, out_vote,
      reinterpret_cast<int*>(ws + w.off_status), reinterpret_cast<int*>(ws + w.off_counters),
      reinterpret_cast<float*>(ws + w.off_partials), reinterpret_cast<float*>(ws + w.off_lse), s,
      &launches, nullptr, false, /*never_ready=*/true);
  if (e != cudaSuccess) return SNAPKV_ERR_CUDA;
  g_last_launches = launches;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_selftest_withheld_partials(const void* q_obs, const void* k, const int32_t* seq_lens, int B,
                                                  int Hq, int Hkv, int L, int d, int W, void* workspace,
                                                  size_t workspace_bytes, void* stream) {
  snapkv_status_t st = check_common(B, Hq, Hkv, L, d, W);
  if (st != SNAPKV_OK) return st;
  if (W >= L || !q_obs || !k || !aligned16(q_obs) || !aligned16(k)) return SNAPKV_ERR_INVALID_ARG;
  const KVStrides ks = dense_strides(Hkv, L, d);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int launches = 0;
  if (seq_lens) {
    for (int b = 0; b < B; ++b)
      if (seq_lens[b] <= W || seq_lens[b] > L) return SNAPKV_ERR_INVALID_ARG;
    RaggedBatch rb;
    ragged_group(seq_lens, B, 0, Hq, Hkv, d, W, W, workspace_bytes, &rb);
    if (rb.count != B || !workspace_ok(workspace, workspace_bytes, rb.total)) return SNAPKV_ERR_WORKSPACE;
    for (int i = 0; i < B; ++i) rb.k_off[i] = i * ks.b;
    if (launch_ragged_scores(rb, q_obs, k, ks, B, Hq, Hkv, d, W, ws, s, &launches, nullptr, false, nullptr,
                             /*withhold=*/true) != cudaSuccess)
      return SNAPKV_ERR_CUDA;
  } else {
    ScorePlan p;
    if (!make_score_plan(B, Hq, Hkv, L, d, W, &p)) return SNAPKV_ERR_UNSUPPORTED;
    const WorkspaceLayout w = make_layout(p, B, Hq, L - W, true, false);
    if (!workspace_ok(workspace, workspace_bytes, w.total)) return SNAPKV_ERR_WORKSPACE;
    if (launch_clear(ws, w, s) != cudaSuccess) return SNAPKV_ERR_CUDA;
    launches = 1;
    if (launch_window_scores(q_obs, k, ks, B, Hq, Hkv, L, d, W, p, reinterpret_cast<float*>(ws + w.off_vote),
                             reinterpret_cast<int*>(ws + w.off_status), reinterpret_cast<int*>(ws + w.off_counters),
                             reinterpret_cast<float*>(ws + w.off_partials), reinterpret_cast<float*>(ws + w.off_lse), s,
                             &launches, nullptr, false, false, nullptr, nullptr, /*withhold=*/true) != cudaSuccess)
      return SNAPKV_ERR_CUDA;
  }
  g_last_launches = launches;
  return SNAPKV_OK;
}

snapkv_status_t snapkv_device_status(const void* workspace, void* stream, int* detail) {
  if (!workspace) return SNAPKV_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int host[2] = {0, 0};
  if (cudaMemcpyAsync(host, workspace, sizeof(host), cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return SNAPKV_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return SNAPKV_ERR_CUDA;
  if (detail) *detail = host[1];
  return host[0] == 0 ? SNAPKV_OK : static_cast<snapkv_status_t>(host[0]);
}

}  // extern "C"
