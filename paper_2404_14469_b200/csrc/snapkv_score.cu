// Host side of the window scoring: plan, tensor maps and launch of the scoring kernel, and the
// small kernels around it.
#include <atomic>

#include "score_kernel.cuh"

namespace snapkv {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Looked up by the first call; others that come meanwhile wait for it (a local static).
EncodeTiledFn get_encode_fn() {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    return cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
                   qres == cudaDriverEntryPointSuccess
               ? reinterpret_cast<EncodeTiledFn>(p)
               : nullptr;
  }();
  return fn;
}

}  // namespace

bool encode_tensor_map(CUtensorMap* m, const void* base, int rank, const unsigned long long* dims,
                       const unsigned long long* strides_bytes, const unsigned* box) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  cuuint64_t d64[5] = {}, s64[5] = {};
  for (int i = 0; i < rank; ++i) d64[i] = dims[i];
  for (int i = 0; i + 1 < rank; ++i) s64[i] = strides_bytes[i];
  auto encode = [&] {
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), d64, s64, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  };
  CUresult r = encode();
  if (r != CUDA_SUCCESS && r != CUDA_ERROR_INVALID_VALUE) {
    // A driver call needs a context, and a thread gets its device's only with the first runtime call
    // that touches the device: for a thread that starts with a decode step, this is before any.
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess) r = encode();
  }
  return r == CUDA_SUCCESS;
}

int sm_count() {
  static std::atomic<int> cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SM_COUNT_HINT;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
      n = SM_COUNT_HINT;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

namespace {

// Supplied-normaliser variant: the caller hands in each window row's natural-log sum-exp
// (what a prefill attention kernel keeps per query row).  This kernel puts it where the vote
// pass expects the merged statistics - minus the log2-sum-exp, one row of MAX_COLS per unit -
// and marks every unit as merged, so the scoring kernel runs its vote phases only.
constexpr int COUNTER_READY = 1 << 30;
__global__ void lse_prep_kernel(const float* __restrict__ lse_obs, float* __restrict__ lse2,
                                int* __restrict__ counters, int* __restrict__ status,
                                int keep_status, int units, int sub_per_kv, int g, int hpu, int W,
                                int ncols) {
  pdl_launch_dependents();
  pdl_wait();
  const int u = blockIdx.x, c = threadIdx.x;  // one block per unit, one thread per column
  // this kernel stands in for the clear kernel of the two-sweep path: the status block too,
  // unless an earlier part of the same logical call may have left an error there
  if (u == 0 && c < STATUS_BYTES / 4 && !keep_status) status[c] = 0;
  if (u >= units || c >= MAX_COLS) return;
  const int ukv = u / sub_per_kv;
  const int hq0 = ukv * g + (u - ukv * sub_per_kv) * hpu;  // flat over the batch
  float out = 0.f;
  if (c < ncols) {
    const int hl = c / W, i = c - hl * W;
    out = -lse_obs[static_cast<size_t>(hq0 + hl) * W + i] * 1.4426950408889634f;
  }
  lse2[static_cast<size_t>(u) * MAX_COLS + c] = out;
  if (c == 0) counters[u] = COUNTER_READY;
}

// After a statistics-only launch: folds every unit's partials, in slot order as the vote sweep
// would, into one natural-log sum-exp per window row (counters[u] is the number of partials the
// unit got).  One block per unit, one thread per window column.
__global__ void lse_finish_kernel(const float* __restrict__ partials, const int* __restrict__ counters,
                                  float* __restrict__ lse_out, int units, int maxseg, int sub_per_kv,
                                  int g, int hpu, int W, int ncols) {
  const int u = blockIdx.x, c = threadIdx.x;
  if (u >= units || c >= ncols) return;
  const int nseg = counters[u];
  const float* pp = partials + static_cast<size_t>(u) * maxseg * MAX_COLS + c;
  float M = -INFINITY, S = 0.f;
  for (int sg = 0; sg < nseg; ++sg) {
    const float pv = pp[static_cast<size_t>(sg) * MAX_COLS];
    const float Mn = fmaxf(fmaxf(M, pv), -1e30f);
    S = S * ex2_approx(M - Mn) + ex2_approx(pv - Mn);
    M = Mn;
  }
  const int ukv = u / sub_per_kv;
  const int hq0 = ukv * g + (u - ukv * sub_per_kv) * hpu;
  const int hl = c / W, i = c - hl * W;
  // log2 -> natural log; a row that saw no key of this shard has S = 0: log gives -inf
  lse_out[static_cast<size_t>(hq0 + hl) * W + i] = (M + log2f(S)) * 0.6931471805599453f;
}

}  // namespace

int score_grid() { return sm_count() < MAX_GRID ? sm_count() : MAX_GRID; }

// The part of the kernel's arguments that fixes the schedule (what the work items follow from).
score::ScoreArgs score_args(const ScorePlan& plan, int L, int W, int Hkv, int votes_only) {
  score::ScoreArgs a = {};
  a.L = L;
  a.n = plan.n_vote;
  a.mask_n = L - W;
  a.stats_only = 0;
  a.W = W;
  a.Hkv = Hkv;
  a.hpu = plan.hpu;
  a.ncols = plan.ncols;
  a.npad = plan.npad;
  a.sub_per_kv = plan.sub_per_kv;
  a.g = plan.g;
  a.units = plan.units;
  a.upw = plan.units_per_wave;
  a.nwaves = plan.nwaves;
  a.T1 = plan.tiles_stats;
  a.T2 = plan.tiles_vote;
  a.maxseg = plan.maxseg;
  a.votes_only = votes_only;
  if (votes_only) {  // nothing couples the units any more: one phase over all of them (over 4096 at most)
    a.upw = plan.units < 4096 ? plan.units : 4096;
    a.nwaves = (plan.units + a.upw - 1) / a.upw;
  }
  return a;
}

int list_schedule_items(const ScorePlan& plan, int L, int W, int Hkv, int votes_only, int grid,
                        int cta, int32_t* out, int max_items) {
  const score::ScoreArgs a = score_args(plan, L, W, Hkv, votes_only);
  int count = 0;
  for (int p = 0; p < score::phase_count(a, score::NotRagged{}); ++p) {
    const score::Phase ph = score::phase_at(a, score::NotRagged{}, grid, p);
    const score::Share share = score::share_of(a, score::NotRagged{}, ph, cta, grid);
    int m = 0;
    for (score::Item it = share.item(0); it.t0 < it.t1; it = share.item(++m), ++count) {
      if (count >= max_items) continue;
      int32_t* o = out + static_cast<size_t>(count) * 6;
      o[0] = it.unit; o[1] = it.t0; o[2] = it.t1; o[3] = ph.vote; o[4] = it.slot; o[5] = it.nseg;
    }
  }
  return count;
}

// A share of a phase of nu units over `grid` CTAs has at most this many items.
int items_per_phase(int nu, int grid) { return (nu + grid - 1) / grid + 1; }
int most_waves_per_launch(int upw) { return score::MAX_RECORDS / (2 * items_per_phase(upw, score_grid())); }

// Whether the publisher folds half of the columns of a launch's vote rows (us per call, one warp and both;
// 32 query heads on 8 KV heads unless stated).
//  - Not with more vote items in a phase than row buffers: the publisher would wait for the softmax warps
//    to use up rows while they wait for it to publish.
//  - Not with few partials per unit: with 14 the two are level (four prompts of 8192 73.2 and 73.0, of 16000
//    104.2 and 104.9, of 32768 169.2 and 169.6), and then the publisher is better left alone.  From 17 on
//    both are level or faster: 17 partials 60.1 and 59.1 (three of 8192), 25 22.9 and 22.3 (one of 3001, 16-row
//    windows), 28 68.9 and 68.5 (two of 20011), 33 46.5 and 46.7 (two of 8192), 52 39.3 and 37.2 (one of 13013),
//    64 24.8 and 23.0 (one KV head of 8192), 192 32.8 and 28.8 (one KV head of 30000).
//  - Not in a part of a call on host buffers that is one KV head.  The part alone gains as above, but the
//    call, which PCIe bounds, does not: 8192 positions 955-959 and 968-988, with 64-row windows 951 and 954-1008;
//    other lengths differ by 1 % at most, either way, and with two KV heads a part the call is faster
//    with both warps (two prompts of 8192: 2026-2079 and 2008-2016).  Why is not known: the copies of one
//    part fall differently against those of the next.
bool shared_fold(const ScorePlan& plan, int W, int per, bool host_part) {
  return !(host_part && plan.units == plan.sub_per_kv) && score::split_columns(plan.npad, W) &&
         per <= score::NLB && plan.maxseg > SHARED_FOLD_ABOVE;
}

bool make_score_plan(int B, int Hq, int Hkv, int L, int d, int W, ScorePlan* plan, int n_vote) {
  if (B < 1 || Hq < 1 || Hkv < 1 || L < 1 || W < 1 || W > L || Hq % Hkv != 0) return false;
  if (n_vote > L) return false;
  if (W > MAX_COLS || (d != 64 && d != 128)) return false;
  ScorePlan p;
  p.g = Hq / Hkv;
  p.hpu = 1;
  for (int h = 1; h <= p.g; ++h)
    if (p.g % h == 0 && h * W <= MAX_COLS) p.hpu = h;
  p.sub_per_kv = p.g / p.hpu;
  const long long units = static_cast<long long>(B) * Hkv * p.sub_per_kv;
  if (units > (1 << 24)) return false;
  p.units = static_cast<int>(units);
  p.ncols = p.hpu * W;
  p.npad = p.ncols <= 32 ? 32 : (p.ncols <= 64 ? 64 : 128);
  const int n = n_vote >= 0 ? n_vote : L - W;
  p.n_vote = n;
  p.tiles_stats = (L + TILE_KEYS - 1) / TILE_KEYS;
  p.tiles_vote = (n + TILE_KEYS - 1) / TILE_KEYS;
  // A wave is a set of units whose keys are swept twice, WAVE_BYTES of keys; the statistics
  // run WAVE_LAG waves ahead of the votes.  Units too big for a wave take one wave each.
  const long long kbytes = static_cast<long long>(L) * d * 2;
  // With 128 window columns on one unit per KV head a vote tile costs the same from L2 as from
  // HBM (the softmax warps are its bound), so nothing is lost by waves too big for L2, and fewer,
  // longer phases split more evenly over the CTAs: such shapes take waves of twice the size
  // (191.6 vs 193.6 us per layer on the 32K GQA workload when the hand-over took longer, 193.1 vs
  // 192.6 with the present one; narrower units and KV heads with two sub-groups, whose vote tiles
  // do gain from L2, are 3-5 % slower that way).
  const long long wave_bytes = (p.ncols == 128 && p.sub_per_kv == 1) ? 2 * score::WAVE_BYTES : score::WAVE_BYTES;
  long long kv_per_wave = wave_bytes / kbytes;
  // units bigger than a wave run one per wave: their second sweep comes from HBM, but the
  // statistics of the next unit still hide the hand-over between the two passes
  if (kv_per_wave < 1) kv_per_wave = 1;
  long long upw = kv_per_wave * p.sub_per_kv;
  // at most 128 units per wave: a CTA's share of a phase then spans few units, which
  // bounds the work items per phase (the book-keeper's buffers are sized for that)
  if (upw > 128) upw = 128 / p.sub_per_kv * p.sub_per_kv;
  if (upw < p.sub_per_kv) upw = p.sub_per_kv;
  if (upw > 4096) upw = 4096;  // (thousands of sub-groups per KV head: a CTA's item list holds 192)
  if (upw > units) upw = units;
  // the bigger waves must not leave a single wave where two of the plain size were possible:
  // with one wave the votes start right behind the statistics and wait for the hand-over
  // (60.2 -> 57.2 us for 2 x 8 KV heads of 32K keys)
  if (wave_bytes != score::WAVE_BYTES && upw >= units && units >= 2 * p.sub_per_kv)
    upw = ((units / p.sub_per_kv + 1) / 2) * p.sub_per_kv;
  p.units_per_wave = static_cast<int>(upw);
  p.nwaves = (p.units + p.units_per_wave - 1) / p.units_per_wave;
  // partial slots per unit: a unit of T1 tiles is shared by at most ceil(T1 / q) + 1 CTAs
  // when every CTA gets at least q = floor(TT / G) tiles of the wave (G up to MAX_GRID)
  auto segs = [&](int nu) {
    const long long TT = static_cast<long long>(nu) * p.tiles_stats;
    const long long q = TT / MAX_GRID;
    long long s = q >= 1 ? (p.tiles_stats + q - 1) / q + 1 : p.tiles_stats;
    if (s > MAX_GRID) s = MAX_GRID;
    return static_cast<int>(s);
  };
  const int last_nu = p.units - (p.nwaves - 1) * p.units_per_wave;
  p.maxseg = segs(p.units_per_wave);
  if (segs(last_nu) > p.maxseg) p.maxseg = segs(last_nu);
  *plan = p;
  return true;
}

cudaError_t launch_window_scores(const void* q_obs, const void* k, const KVStrides& ks, int B,
                                 int Hq, int Hkv, int L, int d, int W, const ScorePlan& plan,
                                 float* vote, int* status,
                                 int* counters, float* partials, float* lse2, cudaStream_t stream,
                                 int* launches, const float* lse_obs, bool keep_status,
                                 bool never_ready, const PagedKV* paged, const ShardMode* shard, bool withhold,
                                 bool host_part) {
  CUtensorMap tmK, tmQ;
  {
    // (d, position, KV head, batch) with the caller's strides: any layout whose rows of d
    // elements are contiguous is one tensor map, e.g. [B, L, Hkv, d] as well as [B, Hkv, L, d].
    // A paged cache is the same map over the pool: (d, position in page, KV head, page); rows
    // past a page's end or pages outside the pool read as zeros.
    using u64 = unsigned long long;
    const u64 dims[4] = {static_cast<u64>(d), static_cast<u64>(paged ? paged->page_size : L),
                         static_cast<u64>(Hkv), static_cast<u64>(paged ? paged->num_pages : B)};
    const u64 strides[3] = {static_cast<u64>(ks.l) * 2, static_cast<u64>(ks.h) * 2, static_cast<u64>(ks.b) * 2};
    const unsigned box[4] = {64, TILE_KEYS, 1, 1};
    if (!encode_tensor_map(&tmK, k, 4, dims, strides, box)) return cudaErrorInvalidValue;
  }
  {
    using u64 = unsigned long long;
    const u64 dims[2] = {static_cast<u64>(d), static_cast<u64>(B) * Hq * W};
    const u64 strides[1] = {static_cast<u64>(d) * 2};
    const unsigned box[2] = {64, static_cast<unsigned>(plan.npad)};
    if (!encode_tensor_map(&tmQ, q_obs, 2, dims, strides, box)) return cudaErrorInvalidValue;
  }
  score::ScoreArgs a = score_args(plan, L, W, Hkv, (lse_obs || never_ready) ? 1 : 0);
  a.wait_ns = wait_limit_setting();
  a.withhold = withhold ? 1 : 0;
  if (shard) {
    a.mask_n = shard->mask_n;
    a.stats_only = shard->lse_out ? 1 : 0;
  }
  a.page_table = paged ? paged->table : nullptr;
  a.pages_per_seq = paged ? paged->pages_per_seq : 0;
  a.page_size = paged ? paged->page_size : 1;
  a.c2 = static_cast<float>(1.4426950408889634 / sqrt(static_cast<double>(d)));
  a.partials = partials;
  a.lse2 = lse2;
  a.counters = counters;
  a.status = status;
  a.vote = vote;
  if (lse_obs) {
    const cudaError_t e =
        launch_pdl(lse_prep_kernel, dim3(plan.units), dim3(MAX_COLS), 0, stream, lse_obs, lse2,
                   counters, status, keep_status ? 1 : 0, plan.units, plan.sub_per_kv, plan.g,
                   plan.hpu, W, plan.ncols);
    if (e != cudaSuccess) return e;
    *launches += 1;
  }
  const int grid = score_grid();
  // a launch holds the items of so many waves; what has more (gigabytes of keys) takes a launch
  // after the other
  a.per = items_per_phase(a.upw, grid);
  const int most = score::MAX_RECORDS / (2 * a.per), waves = a.nwaves;
  if (most < 1) return cudaErrorInvalidValue;
  a.both_fold = !a.votes_only && !a.stats_only && shared_fold(plan, W, a.per, host_part);
  cudaError_t e = cudaSuccess;
  for (; a.wave0 < waves && e == cudaSuccess; a.wave0 += most) {
    a.nwaves = waves - a.wave0 < most ? waves - a.wave0 : most;
    e = score::run_scores_for(d, W, plan.npad, tmK, tmQ, a, score::NotRagged{}, grid, stream, launches);
  }
  if (e != cudaSuccess || !a.stats_only) return e;
  lse_finish_kernel<<<plan.units, MAX_COLS, 0, stream>>>(partials, counters, shard->lse_out, plan.units,
                                                        plan.maxseg, plan.sub_per_kv, plan.g, plan.hpu,
                                                        W, plan.ncols);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace snapkv
