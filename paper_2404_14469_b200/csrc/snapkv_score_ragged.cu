// Window scoring of a ragged batch: prompts of different lengths in one launch of the scoring
// kernel.  One prompt of a few thousand tokens is too short for the GPU (at 13K tokens and eight KV
// heads a call's scoring takes 26 us, 9 us of it arithmetic), and the calls of a batch used to follow
// one another with four launches each.  Here the sequences are waves of one launch: while one waits
// for its statistics to be complete the others' tiles are worked on.
#include "score_kernel.cuh"

namespace snapkv {

namespace {

// What the clear kernel and, with supplied normalisers, the conversion kernel of a single call do,
// for all sequences: status block to zero, partial slots marked as not written, or the normalisers
// into the per-unit rows.
struct PrepSeqs {
  int batch[RAGGED_MAX];
};
__global__ void ragged_prep_kernel(const float* __restrict__ lse_obs, const PrepSeqs seqs, float* __restrict__ lse2,
                                   int* __restrict__ counters, int* __restrict__ status, uint4* __restrict__ partials,
                                   long long slots16, int keep_status, int units_per_seq, int Hq, int sub_per_kv, int g,
                                   int hpu, int W, int ncols) {
  pdl_launch_dependents();
  pdl_wait();
  const int u = blockIdx.x, c = threadIdx.x;  // one block per unit, one thread per window column
  if (u == 0 && c < STATUS_BYTES / 4 && (!keep_status || c == STATUS_READY)) status[c] = 0;
  if (c == 0) counters[u] = lse_obs ? 1 : 0;  // supplied normalisers are ready
  if (!lse_obs) {  // neither a partial nor a folded row is there yet
    for (long long i = static_cast<long long>(u) * MAX_COLS + c; i < slots16; i += static_cast<long long>(gridDim.x) * MAX_COLS)
      partials[i] = make_uint4(NO_PARTIAL, NO_PARTIAL, NO_PARTIAL, NO_PARTIAL);
    return;
  }
  const int seq = u / units_per_seq, ul = u - seq * units_per_seq;
  const int kv = ul / sub_per_kv;
  const int hq0 = seqs.batch[seq] * Hq + kv * g + (ul - kv * sub_per_kv) * hpu;
  float out = 0.f;
  if (c < ncols) {
    const int hl = c / W, i = c - hl * W;
    out = -lse_obs[static_cast<size_t>(hq0 + hl) * W + i] * 1.4426950408889634f;
  }
  lse2[static_cast<size_t>(u) * MAX_COLS + c] = out;
}

// The sequences as the kernel gets them, without their tensor maps; returns the most units of a wave.
template <int MAPS>
int describe(const RaggedBatch& rb, bool votes_only, bool paged, score::RaggedSeqs<MAPS>* rs) {
  int upw = 1;
  rs->nseq = rb.count;
  rs->units_per_seq = rb.plan[0].units;
  rs->waves = 0;
  for (int i = 0; i < rb.count; ++i) {
    const ScorePlan& p = rb.plan[i];
    score::RaggedSeq& q = rs->s[i];
    q.L = rb.L[i];
    q.n = p.n_vote;
    q.upw = votes_only ? p.units : p.units_per_wave;  // votes alone: nothing couples the units
    q.nwaves = votes_only ? 1 : p.nwaves;
    rs->waves += q.nwaves;
    if (q.upw > upw) upw = q.upw;
    q.T1 = p.tiles_stats;
    q.T2 = p.tiles_vote;
    q.maxseg = p.maxseg;
    q.batch = rb.batch[i];
    q.rot = 53 * i;  // consecutive short sequences start on blocks a third of the GPU apart
    q.map = paged ? 0 : i;
    q.part0 = rb.part0[i];
    q.vote0 = rb.vote0[i];
  }
  return upw;
}

template <int MAPS>
cudaError_t launch(const RaggedBatch& rb, const void* q_obs, const void* k, const KVStrides& ks, int B, int Hq,
                   int Hkv, int d, int W, uint8_t* ws, cudaStream_t stream, int* launches, const float* lse_obs,
                   bool keep_status, const PagedKV* paged, bool withhold) {
  using u64 = unsigned long long;
  const ScorePlan& p0 = rb.plan[0];  // head grouping and columns are the same for all sequences
  const int units_per_seq = Hkv * p0.sub_per_kv;
  score::RaggedSeqs<MAPS> rs;
  const int upw = describe(rb, lse_obs != nullptr, paged != nullptr, &rs);
  const u64 strides[3] = {static_cast<u64>(ks.l) * 2, static_cast<u64>(ks.h) * 2, static_cast<u64>(ks.b) * 2};
  const unsigned box[4] = {64, TILE_KEYS, 1, 1};
  for (int i = 0; i < rb.count && !paged; ++i) {
    const u64 dims[4] = {static_cast<u64>(d), static_cast<u64>(rb.L[i]), static_cast<u64>(Hkv), 1};
    if (!encode_tensor_map(&rs.maps[i], static_cast<const uint8_t*>(k) + rb.k_off[i] * 2, 4, dims, strides, box))
      return cudaErrorInvalidValue;
  }
  if (paged) {
    const u64 dims[4] = {static_cast<u64>(d), static_cast<u64>(paged->page_size), static_cast<u64>(Hkv),
                         static_cast<u64>(paged->num_pages)};
    if (!encode_tensor_map(&rs.maps[0], k, 4, dims, strides, box)) return cudaErrorInvalidValue;
  }
  CUtensorMap tmQ;
  {
    const u64 dims[2] = {static_cast<u64>(d), static_cast<u64>(B) * Hq * W};
    const u64 qstr[1] = {static_cast<u64>(d) * 2};
    const unsigned qbox[2] = {64, static_cast<unsigned>(p0.npad)};
    if (!encode_tensor_map(&tmQ, q_obs, 2, dims, qstr, qbox)) return cudaErrorInvalidValue;
  }
  score::ScoreArgs a = score_args(p0, rb.L[0], W, Hkv, lse_obs ? 1 : 0);
  a.wait_ns = wait_limit_setting();
  a.withhold = withhold ? 1 : 0;
  a.page_table = paged ? paged->table : nullptr;
  a.pages_per_seq = paged ? paged->pages_per_seq : 0;
  a.page_size = paged ? paged->page_size : 1;
  a.c2 = static_cast<float>(1.4426950408889634 / sqrt(static_cast<double>(d)));
  a.counters = reinterpret_cast<int*>(ws + rb.off_counters);
  a.partials = reinterpret_cast<float*>(ws + rb.off_partials);
  a.lse2 = reinterpret_cast<float*>(ws + rb.off_lse);
  a.vote = reinterpret_cast<float*>(ws + rb.off_vote);
  a.status = reinterpret_cast<int*>(ws);
  PrepSeqs seqs = {};
  for (int i = 0; i < rb.count; ++i) seqs.batch[i] = rb.batch[i];
  cudaError_t e = launch_pdl(ragged_prep_kernel, dim3(rb.count * units_per_seq), dim3(MAX_COLS), 0, stream, lse_obs,
                             seqs, a.lse2, a.counters, a.status, reinterpret_cast<uint4*>(a.partials),
                             static_cast<long long>((rb.off_vote - rb.off_partials) / 16), keep_status ? 1 : 0,
                             units_per_seq, Hq, p0.sub_per_kv, p0.g, p0.hpu, W, p0.ncols);
  if (e != cudaSuccess) return e;
  *launches += 1;
  const int grid = score_grid();
  a.per = items_per_phase(upw, grid);
  if (rs.waves * 2 * a.per > score::MAX_RECORDS) return cudaErrorInvalidValue;  // (the callers' groups are small enough)
  return score::run_scores_for(d, W, p0.npad, tmQ, tmQ, a, rs, grid, stream, launches);
}

}  // namespace

int list_ragged_items(const RaggedBatch& rb, int W, int Hkv, int votes_only, int grid, int cta, int32_t* out,
                      int max_items) {
  score::RaggedSeqs<1> rs;
  describe(rb, votes_only != 0, true, &rs);
  const score::ScoreArgs a = score_args(rb.plan[0], rb.L[0], W, Hkv, votes_only);
  int count = 0;
  for (int p = 0; p < score::phase_count(a, rs); ++p) {
    const score::Phase ph = score::phase_at(a, rs, grid, p);
    const score::Share share = score::share_of(a, rs, ph, cta, grid);
    int m = 0;
    for (score::Item it = share.item(0); it.t0 < it.t1; it = share.item(++m), ++count) {
      if (count >= max_items) continue;
      int32_t* o = out + static_cast<size_t>(count) * 8;
      o[0] = it.unit; o[1] = it.t0; o[2] = it.t1; o[3] = ph.vote; o[4] = it.slot; o[5] = it.nseg;
      o[6] = ph.seq; o[7] = ph.ord;
    }
  }
  return count;
}

cudaError_t launch_ragged_scores(const RaggedBatch& rb, const void* q_obs, const void* k, const KVStrides& ks, int B,
                                 int Hq, int Hkv, int d, int W, uint8_t* ws, cudaStream_t stream, int* launches,
                                 const float* lse_obs, bool keep_status, const PagedKV* paged, bool withhold) {
  auto f = paged ? launch<1> : launch<RAGGED_MAX>;
  return f(rb, q_obs, k, ks, B, Hq, Hkv, d, W, ws, stream, launches, lse_obs, keep_status, paged, withhold);
}

}  // namespace snapkv
