// Pooling and per-head top-k (Listing 1's pool1d and topk; Eq. 2): one thread-block CLUSTER of 1
// to 16 CTAs per row, pooling radii up to 7, rows of up to 524288 positions.
//
// The votes come from L2 and are few (17 MB for 128 rows of 32K); what a row costs is the chain of
// steps that its threads take together.  So the chain is kept short:
//   1. a CTA's chunk of votes (plus the pooling halo) goes to shared memory with coalesced loads;
//      every thread pools its own EPT consecutive positions and keeps them, as order-preserving
//      32-bit keys, in registers for the rest of the kernel;
//   2. a small histogram of 256 pooled values sampled over the whole row, the same in every CTA,
//      gives the bins that lie four standard deviations to either side of the rank that ksel maps
//      to; they bound a window of keys which should hold the ksel-th largest;
//   3. the keys inside the window (a sixth of a row, a few per cent when ksel << n) are histogrammed
//      into 1024 bins, those above it counted; the CTAs of the cluster add up one another's
//      histograms through distributed shared memory, and all find the same bin;
//   4. that bin's few keys (about five for a row of 32K) are pushed, with the CTA's counts, into
//      every CTA's memory: each CTA ranks them by counting and knows the threshold, and how many
//      selected positions come before its chunk;
//   5. ordered compaction: a block scan, positions staged in shared memory, coalesced stores.
// The sample only guesses.  Counts are exact: when the ksel-th key turns out to lie outside the
// window the histogram is taken over the whole key range, and a bin with more keys than the list
// holds is refined by a further histogram; ties go to the lower position by construction.
// Two cluster barriers on the usual path (a byte-wise radix select took five), one histogram
// update for every sixth key.  Back to back in a graph: 4 rows of 992 in 4.7 us, 32 rows of 16352 in
// 9.1, 128 rows of 32736 in 13.8, 32 rows of 131008 in 17.  (Single launches back to back, when the kernel
// was new: 6.0, 11.6, 16.8 and 22.7; with one CTA per row, all keys in shared memory and five passes over them
// 12.4, 14.4, 20.6 and 49.9.)  Rows so long or so many that the clusters come in several rounds are
// filtered first (long_filter_kernel).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "launch.cuh"
#include "sm100_ptx.cuh"
#include "snapkv_internal.h"

namespace snapkv {

namespace {

constexpr int CL_RMAX = 7;           // largest pooling radius this kernel takes
constexpr int CL_MAX_CLUSTER = 16;   // above 8: non-portable cluster size
constexpr int CL_BINS = 1024;
constexpr int CL_SAMPLES = 256;
constexpr int CL_SAMPLE_BINS = 512;
constexpr int CL_LIST = 2048;        // candidates in all of a cluster's lists
constexpr int LONG_META = 256;       // words per row: threshold, whether it is done, keys listed per chunk
constexpr int LONG_THRESHOLD = 0, LONG_DONE = 1, LONG_COUNTS = 2;
constexpr uint32_t KEY_MIN = 0x80000000u;  // key of a vote of zero; below it: no position

__device__ __forceinline__ uint32_t float_to_key(float x) {
  const uint32_t b = __float_as_uint(x);
  return b ^ (static_cast<uint32_t>(static_cast<int32_t>(b) >> 31) | 0x80000000u);
}
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Tells L2 that a 128-byte line (global memory, 128-byte aligned) holds nothing worth keeping:
// a dirty line may then be dropped instead of written back.  Its contents are undefined afterwards.
__device__ __forceinline__ void discard_l2_line(const void* p) {
  asm volatile("discard.global.L2 [%0], 128;" ::"l"(__cvta_generic_to_global(p)) : "memory");
}

// Slot of position t of the staged chunk: four pad words after every 32, so that a thread reads
// its run (a multiple of 8 positions) as aligned 16-byte vectors and the runs of neighbouring
// threads fall into different banks.
__device__ __forceinline__ int slot(int t) { return t + ((t >> 5) << 2); }
constexpr int slots_for(int n) { return n + n / 8 + 8; }

// Exclusive prefix sum over the CTA's threads; *total_s holds the sum afterwards.  Two barriers.
template <int THREADS>
__device__ __forceinline__ uint32_t block_scan(uint32_t x, uint32_t* warp_sums_s, uint32_t* total_s) {
  constexpr int WARPS = THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sums_s[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < WARPS ? warp_sums_s[lane] : 0u;
    uint32_t winc = w;
#pragma unroll
    for (int o = 1; o < WARPS; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += y;
    }
    if (lane < WARPS) warp_sums_s[lane] = winc - w;
    if (lane == WARPS - 1) *total_s = winc;
  }
  __syncthreads();
  return warp_sums_s[warp] + inc - x;
}

struct OneLength {};
// Rows of one length that are sums of gsum consecutive vote rows.  A kind of its own: the sums need a second
// set of registers for the loads in flight, and kernels that never make one would spill for it (with 32 keys
// a thread 96 to 224 bytes where it is 0 to 88 without).
struct GroupedRows {};
// Rows seq * heads + h: head h of the batch's sequence batch[seq].  A batch's long and short rows may be
// two launches with CTAs of different sizes, side by side.  A CTA of the first one lets the second in
// once its own wait for the votes is over; the first CTA before that stores a flag (`ready`) with release
// semantics.  The second launch (`after`) reads the flag with acquire semantics and then the votes: what
// the first had visible is visible to it by that pair, not by the early start, which promises nothing.  A
// thread that does not find the flag set waits for the first launch to end.  Every CTA of the second
// launch waits for that before it ends itself, so the gather kernel, which waits for the second, finds both
// complete.
struct RaggedRows {
  int n[RAGGED_MAX], batch[RAGGED_MAX];
  int2 want[RAGGED_MAX];
  long long vote0[RAGGED_MAX];
  int heads;
  int* ready;  // zero when the first of two launches starts; nullptr: one launch
  bool after;
};

__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// A vote.  Rows of a ragged batch may be read by a kernel that starts while the one before it runs, so the
// load is an ordinary one, behind the acquire; others may take the read-only path.
template <typename ROWS>
__device__ __forceinline__ float ld_vote(const float* p) {
  if constexpr (std::is_same<ROWS, RaggedRows>::value) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
  } else {
    return __ldg(p);
  }
}

// Sliding pooling of eight positions: out[i] over a[i .. i + 2R].  The maximum is taken over
// doubling spans (three or four operations per position instead of 2R + 1; a maximum is the same
// in any order), the sum in ascending order.
template <int R, int PT>
__device__ __forceinline__ void pool8(const float* a, float (&out)[8], int r, int pool_type, float divisor) {
  if constexpr (PT == 0 && (R == 2 || R == 3 || R == 6)) {
    float m2[2 * R + 7], m4[2 * R + 5];
#pragma unroll
    for (int i = 0; i < 2 * R + 7; ++i) m2[i] = fmaxf(a[i], a[i + 1]);
#pragma unroll
    for (int i = 0; i < 2 * R + 5; ++i) m4[i] = fmaxf(m2[i], m2[i + 2]);
    if constexpr (R == 6) {
      float m8[13];
#pragma unroll
      for (int i = 0; i < 13; ++i) m8[i] = fmaxf(m4[i], m4[i + 4]);
#pragma unroll
      for (int i = 0; i < 8; ++i) out[i] = fmaxf(fmaxf(m8[i], m8[i + 5]), 0.f);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) out[i] = fmaxf(fmaxf(m4[i], m4[i + 2 * R - 3]), 0.f);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float p = 0.f;  // votes are >= 0: zero is neutral for max and is the padding of avg
#pragma unroll
      for (int t = 0; t <= 2 * R; ++t)
        if (PT >= 0 || (t - R >= -r && t - R <= r))
          p = (PT >= 0 ? PT == 0 : pool_type == 0) ? fmaxf(p, a[i + t]) : p + a[i + t];
      if (PT < 0 && divisor != 0.f) p = p / divisor;
      out[i] = p;
    }
  }
}

// R, PT >= 0: the pooling radius is exactly R and the type PT (0 max, 1 avg), no per-tap tests.
// PT = -1: radius r <= R and pool_type are run-time values, and with `divisor` != 0 average pooling
// divides the window sum by it (otherwise rows are ranked by the sum, which orders the same way up
// to rounding).  `want`: the sample ranks (from the top) that bound the window.  ROWS: OneLength (gsum = 1),
// GroupedRows, or RaggedRows when the rows come from sequences of different lengths (gsum = 1, n and want are
// not used then).
template <int THREADS, int EPT, int R, int PT, typename ROWS>
__global__ void __launch_bounds__(THREADS, THREADS == 1024 ? 1 : 1024 / THREADS)
pool_topk_cluster_kernel(const float* __restrict__ vote, int n, int gsum, int r, int pool_type, float divisor,
                         int ksel, int2 want, int32_t* __restrict__ out_idx, int ctas, int discard_votes,
                         const uint32_t* __restrict__ meta, const __grid_constant__ ROWS rows) {
  // With 16 and 32 keys a thread the instructions per key count (72 with 32 keys, 58 now: the schedulers issued in
  // 55 to 60 % of the cycles), so whole chunks skip the checks of the row's end, the keys are compared
  // with the bin once, and the positions are picked by set bits (128 rows of 32736: 3 us less).  With
  // eight it is the chain of steps: there the forms that need the fewest steps in a row stay.
  constexpr int CHUNK = THREADS * EPT;
  constexpr int BPT = CL_BINS / THREADS;      // bins a thread owns in the scans
  extern __shared__ __align__(16) uint32_t stage[];  // votes of the chunk, later the selected positions
  __shared__ float halo[2][CL_RMAX + 1];      // CL_RMAX positions before the chunk and behind it
  __shared__ __align__(16) uint32_t hist[2][CL_BINS + 4];  // word CL_BINS: keys above the window
  __shared__ __align__(16) uint32_t samp_hist[CL_SAMPLE_BINS];
  __shared__ uint32_t samp_min[CL_SAMPLES / 32], samp_max[CL_SAMPLES / 32];
  __shared__ __align__(8) uint2 list[CL_LIST];           // {key, position}, a region per CTA of the cluster
  __shared__ __align__(8) uint2 totals[CL_MAX_CLUSTER];  // per CTA: keys above the bin, keys inside it
  __shared__ uint32_t warp_sums[32];
  __shared__ uint32_t scan_total, sel_bin, sel_above, sel_count, win_hi, win_lo, n_list, n_gt;
  __shared__ uint32_t thr_key, thr_eq, thr_all, before_gt, before_eq;

  const uint32_t rank = blockIdx.x % ctas;
  const int row = blockIdx.x / ctas;
  const float* vrow;
  int32_t* orow;
  uint32_t C = ctas;
  if constexpr (std::is_same<ROWS, RaggedRows>::value) {
    const int seq = row / rows.heads, h = row - seq * rows.heads;
    n = rows.n[seq];
    want = rows.want[seq];
    vrow = vote + rows.vote0[seq] + static_cast<size_t>(h) * n;
    orow = out_idx + (static_cast<size_t>(rows.batch[seq]) * rows.heads + h) * ksel;
    // CTAs behind the end of a short row leave at once: cluster barriers do not count them
    C = min(C, static_cast<uint32_t>((n + CHUNK - 1) / CHUNK));
    if (rank >= C) {
      if (rows.after) pdl_wait();
      return;
    }
  } else {
    vrow = vote + static_cast<size_t>(row) * gsum * n;
    orow = out_idx + static_cast<size_t>(row) * ksel;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = static_cast<int>(rank) * CHUNK;  // first position of this CTA's chunk
  if constexpr (std::is_same<ROWS, RaggedRows>::value) {
    if (!rows.after || ld_acquire(rows.ready) == 0) pdl_wait();
    if (rows.ready != nullptr && !rows.after) {
      if (blockIdx.x == 0 && tid == 0) st_release(rows.ready, 1);
      pdl_launch_dependents();
    }
  } else {
    pdl_wait();
  }
  if (meta != nullptr && meta[static_cast<size_t>(row) * LONG_META + LONG_DONE]) return;
  if (C > 1) cluster_arrive();  // waited for before the first access to a peer's memory

  // ---- 1. the sample (pooled values at 256 positions spread over the whole row), the chunk and its
  // halo: all loads are issued before the first value is used.  Positions outside the row are zero.
  // A group's votes are summed in ascending head order.
  float tap[2 * R + 1];
  const int js = static_cast<int>((static_cast<long long>(tid) * n + n / 2) / CL_SAMPLES);
  if (tid < CL_SAMPLES) {
#pragma unroll
    for (int t = 0; t <= 2 * R; ++t) {
      const int j = js + t - R;
      tap[t] = static_cast<unsigned>(j) < static_cast<unsigned>(n) ? ld_vote<ROWS>(vrow + j) : 0.f;
    }
  }
  float h_val = 0.f;
  int h_at = -1;  // the halo position this thread fetches
  if (tid >= THREADS - 2 * CL_RMAX) {
    const int i = tid - (THREADS - 2 * CL_RMAX);
    const int j = i < CL_RMAX ? c0 - CL_RMAX + i : c0 + CHUNK + i - CL_RMAX;
    if (static_cast<unsigned>(j) < static_cast<unsigned>(n)) {
      h_at = j;
      h_val = ld_vote<ROWS>(vrow + j);
    }
  }
  // Of each further head of a group the sample, the halo and the first eight keys of a thread are requested
  // before any is added: one round trip a head where a thread has eight, not one for the sample and one
  // for the chunk.  With 32 keys and a wide sample the registers do not hold both (96 and 196 bytes of
  // spills with radius 6 and with any radius): there the sample is summed before the chunk is loaded.
  constexpr bool GROUPED = std::is_same<ROWS, GroupedRows>::value;
  constexpr bool TOGETHER = EPT < 32 || R <= 3;
  if constexpr (GROUPED && !TOGETHER) {
    for (int g = 1; g < gsum; ++g) {
      const float* src = vrow + static_cast<size_t>(g) * n;
      if (tid < CL_SAMPLES) {
#pragma unroll
        for (int t = 0; t <= 2 * R; ++t) {
          const int j = js + t - R;
          if (static_cast<unsigned>(j) < static_cast<unsigned>(n)) tap[t] += __ldg(src + j);
        }
      }
      if (h_at >= 0) h_val += __ldg(src + h_at);
    }
  }
  {
    float x[EPT];
    if (EPT > 8 && c0 + CHUNK <= n) {
#pragma unroll
      for (int u = 0; u < EPT; ++u) x[u] = ld_vote<ROWS>(vrow + c0 + tid + THREADS * u);
    } else {
#pragma unroll
      for (int u = 0; u < EPT; ++u) {
        const int j = c0 + tid + THREADS * u;
        x[u] = j < n ? ld_vote<ROWS>(vrow + j) : 0.f;
      }
    }
    for (int g = 1; GROUPED && g < gsum; ++g) {
      const float* src = vrow + static_cast<size_t>(g) * n;
      if constexpr (TOGETHER) {
        float t2[2 * R + 1], y[8], h2 = 0.f;
        if (tid < CL_SAMPLES) {
#pragma unroll
          for (int t = 0; t <= 2 * R; ++t) {
            const int j = js + t - R;
            t2[t] = static_cast<unsigned>(j) < static_cast<unsigned>(n) ? __ldg(src + j) : 0.f;
          }
        }
        if (h_at >= 0) h2 = __ldg(src + h_at);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int j = c0 + tid + THREADS * u;
          y[u] = j < n ? __ldg(src + j) : 0.f;
        }
        if (tid < CL_SAMPLES) {
#pragma unroll
          for (int t = 0; t <= 2 * R; ++t) tap[t] += t2[t];
        }
        h_val += h2;
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] += y[u];
      }
#pragma unroll
      for (int u = TOGETHER ? 8 : 0; u < EPT; ++u) {
        const int j = c0 + tid + THREADS * u;
        if (j < n) x[u] += __ldg(src + j);
      }
    }
#pragma unroll
    for (int u = 0; u < EPT; ++u) stage[slot(tid + THREADS * u)] = __float_as_uint(x[u]);
  }
  if (tid >= THREADS - 2 * CL_RMAX) {
    const int i = tid - (THREADS - 2 * CL_RMAX);
    halo[i >= CL_RMAX][i >= CL_RMAX ? i - CL_RMAX : i] = h_val;
  }
  uint32_t s_key = 0u;
  if (tid < CL_SAMPLES) {
    float p = 0.f;
#pragma unroll
    for (int t = 0; t <= 2 * R; ++t)
      if (PT >= 0 || (t - R >= -r && t - R <= r))
        p = (PT >= 0 ? PT == 0 : pool_type == 0) ? fmaxf(p, tap[t]) : p + tap[t];
    if (PT < 0 && divisor != 0.f) p = p / divisor;
    s_key = float_to_key(p);
    const uint32_t lo = __reduce_min_sync(0xffffffffu, s_key), hi = __reduce_max_sync(0xffffffffu, s_key);
    if (lane == 0) {
      samp_min[warp] = lo;
      samp_max[warp] = hi;
    }
  }
  for (int b = tid; b < CL_SAMPLE_BINS; b += THREADS) samp_hist[b] = 0u;
  for (int b = tid; b < CL_BINS + 4; b += THREADS) hist[0][b] = 0u;
  if (tid == 0) {
    sel_bin = ~0u;
    n_list = n_gt = before_gt = before_eq = 0u;
  }
  __syncthreads();

  // ---- 2. the window, from a histogram of the sample: the bins that hold the sample ranks four
  // standard deviations to either side of the rank that ksel maps to
  uint32_t smin = ~0u, smax = 0u;
  if (tid < CL_SAMPLES) {
#pragma unroll
    for (int w = 0; w < CL_SAMPLES / 32; ++w) {
      smin = min(smin, samp_min[w]);
      smax = max(smax, samp_max[w]);
    }
  }
  const int sshift = max(0, 23 - __clz(smax - smin));  // (range >> sshift) < CL_SAMPLE_BINS
  if (tid < CL_SAMPLES) atomicAdd(&samp_hist[(s_key - smin) >> sshift], 1u);
  __syncthreads();
  if (warp == 0) {  // lane t owns the 16 bins CL_SAMPLE_BINS - 16 t - 1 and down
    static_assert(CL_SAMPLE_BINS == 512, "16 bins per lane");
    const uint32_t want_hi = static_cast<uint32_t>(max(1, want.x + 1));
    const uint32_t want_lo = static_cast<uint32_t>(min(CL_SAMPLES, want.y + 1));
    uint32_t c[16], sum = 0u;
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(samp_hist + CL_SAMPLE_BINS - 16 * (lane + 1) + i);
      c[i] = v.x; c[i + 1] = v.y; c[i + 2] = v.z; c[i + 3] = v.w;
      sum += v.x + v.y + v.z + v.w;
    }
    uint32_t above = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, above, o);
      if (lane >= o) above += y;
    }
    above -= sum;
#pragma unroll
    for (int i = 15; i >= 0; --i) {
      const uint32_t edge = smin + (static_cast<uint32_t>(CL_SAMPLE_BINS - 16 * (lane + 1) + i) << sshift);
      if (above < want_hi && want_hi <= above + c[i]) win_hi = min(edge + ((1u << sshift) - 1u), smax);
      if (above < want_lo && want_lo <= above + c[i]) win_lo = want.y >= CL_SAMPLES ? KEY_MIN : edge;
      above += c[i];
    }
  }

  // ---- pooling: thread owns positions c0 + base .. c0 + base + EPT - 1
  const int base = tid * EPT;
  uint32_t key[EPT];
  {
    auto own8 = [&](int i, float* dst) {  // positions base + i .. + 7 of the chunk
#pragma unroll
      for (int q = 0; q < 8; q += 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(stage + slot(base + i + q));
        dst[q] = __uint_as_float(v.x);
        dst[q + 1] = __uint_as_float(v.y);
        dst[q + 2] = __uint_as_float(v.z);
        dst[q + 3] = __uint_as_float(v.w);
      }
    };
    auto at = [&](int t) {  // position t of the chunk or its halo
      return t < 0 ? halo[0][CL_RMAX + t] : (t >= CHUNK ? halo[1][t - CHUNK] : __uint_as_float(stage[slot(t)]));
    };
    // a[]: the R values before the current block of eight, the block, the next block
    float a[R + 16];
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = at(base - R + i);
    own8(0, a + R);
#pragma unroll
    for (int sb = 0; sb < EPT; sb += 8) {
      if (sb + 8 < EPT) {
        own8(sb + 8, a + R + 8);
      } else {
#pragma unroll
        for (int i = 0; i < R; ++i) a[R + 8 + i] = at(base + EPT + i);
      }
      float p[8];
      pool8<R, PT>(a, p, r, pool_type, divisor);
#pragma unroll
      for (int i = 0; i < 8; ++i) key[sb + i] = EPT > 8 || c0 + base + sb + i < n ? float_to_key(p[i]) : 0u;
#pragma unroll
      for (int i = 0; i < R + 8; ++i) a[i] = a[i + 8];
    }
    if (EPT > 8 && c0 + base + EPT > n) {  // the row ends among them
#pragma unroll
      for (int i = 0; i < EPT; ++i) key[i] = c0 + base + i < n ? key[i] : 0u;
    }
  }
  __syncthreads();

  // ---- 3. histogram rounds: the usual path takes one.  Keys lo .. lo + width take part, `top`
  // counts those above.
  uint32_t lo = win_lo, width = win_hi - win_lo;
  int shift = max(0, 22 - __clz(width));  // (width >> shift) < CL_BINS
  uint32_t krem = static_cast<uint32_t>(ksel);
  const uint32_t cap = min(CL_LIST / C, static_cast<uint32_t>(CL_SAMPLES));  // a thread per entry
  bool guess = true;
  uint32_t bin_lo = 0u, bin_w = 0u, in_bin = 0u;
#pragma unroll 1
  for (int round = 0;; ++round) {
    uint32_t* h = hist[round & 1];
    if (round > 0) {
      for (int b = tid; b < CL_BINS + 4; b += THREADS) h[b] = 0u;
      if (tid == 0) sel_bin = ~0u;
      __syncthreads();
    }
    uint32_t top = 0u;
    const uint32_t hi = lo + width;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      const uint32_t rel = key[i] - lo;  // wraps for keys below lo
      if (rel <= width) atomicAdd(&h[rel >> shift], 1u);
      top += key[i] > hi;
    }
    if (guess) {
      top = __reduce_add_sync(0xffffffffu, top);
      if (lane == 0 && top) atomicAdd(&h[CL_BINS], top);
    }
    if (C > 1) {
      if (round == 0) cluster_wait();
      cluster_arrive();  // the cluster's barrier stands in for the CTA's
      cluster_wait();
    } else {
      __syncthreads();
    }
    // thread t owns the bins CL_BINS - 1 - BPT t and down; thread 0 also the keys above the window
    uint32_t c[BPT], sum = 0u;
    top = 0u;
    {
      const int b0 = CL_BINS - BPT * (tid + 1);
#pragma unroll
      for (int u = 0; u < BPT; ++u) c[u] = 0u;
      if (C == 1) {
#pragma unroll
        for (int u = 0; u < BPT; ++u) c[u] = h[b0 + u];
        if (tid == 0) top = h[CL_BINS];
      } else {
        // the peers' reads are in flight four at a time
#pragma unroll 1
        for (uint32_t p0 = 0; p0 < C; p0 += 4) {
          uint32_t x[4][BPT];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t addr = peer_addr(h + b0, min(p0 + q, C - 1));
            if constexpr (BPT == 4)
              asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                           : "=r"(x[q][0]), "=r"(x[q][1]), "=r"(x[q][2]), "=r"(x[q][3]) : "r"(addr) : "memory");
            else if constexpr (BPT == 2)
              asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(x[q][0]), "=r"(x[q][1]) : "r"(addr) : "memory");
            else
              asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x[q][0]) : "r"(addr) : "memory");
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < BPT; ++u) c[u] += p0 + q < C ? x[q][u] : 0u;
        }
        if (warp == 0) {
          uint32_t x = 0u;
          if (static_cast<uint32_t>(lane) < C)
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(x) : "r"(peer_addr(h + CL_BINS, lane)) : "memory");
          x = __reduce_add_sync(0xffffffffu, x);
          if (lane == 0) top = x;
        }
      }
#pragma unroll
      for (int u = 0; u < BPT; ++u) sum += c[u];
    }
    uint32_t above = block_scan<THREADS>(sum + top, warp_sums, &scan_total) + top;
#pragma unroll
    for (int u = BPT - 1; u >= 0; --u) {
      if (above < krem && krem <= above + c[u]) {
        sel_bin = static_cast<uint32_t>(CL_BINS - BPT * (tid + 1) + u);
        sel_above = above;
        sel_count = c[u];
      }
      above += c[u];
    }
    __syncthreads();
    const uint32_t b = sel_bin;
    if (b == ~0u) {
      // Above the guessed window or below it: the whole range decides, and all of it, so that a bin is
      // found whatever the votes are (the 0 of the positions outside the row is its lowest key, and
      // those positions come last).
      guess = false;
      lo = 0u;
      width = ~0u;
      shift = 22;
      __syncthreads();  // everybody has read sel_bin before it is written again
      continue;
    }
    guess = false;
    krem -= sel_above;
    in_bin = sel_count;
    bin_lo = lo + (b << shift);
    bin_w = min((1u << shift) - 1u, lo + width - bin_lo);  // keys behind the window's end count as above it
    if (shift == 0 || in_bin <= cap) break;
    lo = bin_lo;
    width = bin_w;
    shift = max(0, shift - 10);
    __syncthreads();
  }
  const bool listed = shift > 0;  // else every key of the bin equals bin_lo

  // ---- 4. the bin's keys and this CTA's counts go to every CTA of the cluster
  uint32_t m_gt = 0u, m_in = 0u;  // this thread's keys above the bin and inside it (EPT <= 32)
  {
    const uint32_t bin_hi = bin_lo + bin_w;
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      if constexpr (EPT > 8) {
        if (key[i] >= bin_lo) m_in |= 1u << i;
        if (key[i] > bin_hi) m_gt |= 1u << i;
      } else {
        m_in |= static_cast<uint32_t>(key[i] - bin_lo <= bin_w) << i;
        if (C > 1) m_gt |= static_cast<uint32_t>(key[i] > bin_hi) << i;
      }
    }
    if (EPT > 8) m_in &= ~m_gt;
    if (C > 1) {  // the keys above the bin matter to the CTAs behind this one
      const uint32_t gt = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(__popc(m_gt)));
      if (lane == 0 && gt) atomicAdd(&n_gt, gt);
    }
    if (listed) {
      for (uint32_t m = m_in; m; m &= m - 1) {  // a few keys per row: the register is picked by comparison
        const int bit = __ffs(m) - 1;
        uint32_t k = key[0];
#pragma unroll
        for (int i = 1; i < EPT; ++i) k = i == bit ? key[i] : k;
        const uint32_t at = rank * cap + atomicAdd(&n_list, 1u);
        for (uint32_t p = 0; p < C; ++p) st_peer2(peer_addr(&list[at], p), k, static_cast<uint32_t>(c0 + base + bit));
      }
    } else {
      const uint32_t in = __reduce_add_sync(0xffffffffu, static_cast<uint32_t>(__popc(m_in)));
      if (lane == 0 && in) atomicAdd(&n_list, in);
    }
  }
  __syncthreads();
  if (tid < static_cast<int>(C)) st_peer2(peer_addr(&totals[rank], tid), n_gt, n_list);
  if (C > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  if (discard_votes) {
    // Every CTA of the row has its votes, and nobody reads them again: drop the whole 128-byte
    // lines inside the row from L2, so that they are not written back to HBM while the gather
    // kernel needs the bandwidth.  Lines that the row shares with its neighbours stay.
    const uintptr_t b0 = (reinterpret_cast<uintptr_t>(vrow) + 127) & ~static_cast<uintptr_t>(127);
    const uintptr_t b1 = reinterpret_cast<uintptr_t>(vrow + static_cast<size_t>(gsum) * n) & ~static_cast<uintptr_t>(127);
    for (uintptr_t a = b0 + (static_cast<uintptr_t>(rank) * THREADS + tid) * 128; a < b1;
         a += static_cast<uintptr_t>(C) * THREADS * 128)
      discard_l2_line(reinterpret_cast<const void*>(a));
  }
  if (listed) {
    // entry e of the lists: rank it among all (keys only), find the threshold
    uint32_t my_key = 0u, my_cta = C;
    if (static_cast<uint32_t>(tid) < in_bin) {
      uint32_t e = tid;
      my_cta = 0u;
      while (e >= totals[my_cta].y) e -= totals[my_cta++].y;
      my_key = list[my_cta * cap + e].x;
      uint32_t gt = 0u, eq = 0u;
      for (uint32_t p = 0; p < C; ++p)
        for (uint32_t i = 0; i < totals[p].y; ++i) {
          const uint32_t k = list[p * cap + i].x;
          gt += k > my_key;
          eq += k == my_key;
        }
      if (gt < krem && krem <= gt + eq) {
        thr_key = my_key;
        thr_eq = krem - gt;
        thr_all = eq;
      }
    }
    __syncthreads();
    if (my_cta < rank) {
      if (my_key > thr_key) atomicAdd(&before_gt, 1u);
      if (my_key == thr_key) atomicAdd(&before_eq, 1u);
    }
  } else if (tid == 0) {
    thr_key = bin_lo;
    thr_eq = krem;
    thr_all = in_bin;
  }
  if (tid < static_cast<int>(rank)) {
    atomicAdd(&before_gt, totals[tid].x);
    if (!listed) atomicAdd(&before_eq, totals[tid].y);
  }
  __syncthreads();

  // ---- 5. ordered compaction: keys above the threshold, plus the lowest positions equal to it
  const uint32_t T = thr_key, need_eq = thr_eq, gt0 = before_gt, eq0 = before_eq;
  const bool all_eq = need_eq == thr_all;  // every key equal to the threshold is kept (the usual case)
  uint32_t m_keep = EPT > 8 ? m_gt : 0u, m_eq = 0u;
  if (EPT == 8 || m_in) {  // (the threshold is a key of the bin)
    const uint32_t T_keep = all_eq ? T : T + 1u;
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      if (key[i] >= T_keep) m_keep |= 1u << i;
    if (!all_eq) {
#pragma unroll
      for (int i = 0; i < EPT; ++i) m_eq |= static_cast<uint32_t>(key[i] == T) << i;
    }
  }
  static_assert(CHUNK < 65536, "two 16-bit counts share one scan word");
  const uint32_t packed = block_scan<THREADS>((static_cast<uint32_t>(__popc(m_keep)) << 16) | __popc(m_eq),
                                              warp_sums, &scan_total);
  const uint32_t kept0 = min(eq0, need_eq);  // equal positions kept before this chunk
  uint32_t eq_seen = eq0 + (packed & 0xffffu);
  uint32_t at = packed >> 16;
  if (!all_eq) {
    at += min(eq_seen, need_eq) - kept0;
    while (m_eq && eq_seen < need_eq) {  // the lowest ones
      m_keep |= m_eq & (0u - m_eq);
      m_eq &= m_eq - 1;
      ++eq_seen;
    }
  }
  // A loop over set bits takes nine instructions a position and is as long as the warp's fullest lane
  // makes it, the other form takes five for every key (and has nothing to find out first).
  if (EPT > 8 && 2 * __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(__popc(m_keep))) <= EPT) {
    for (; m_keep; m_keep &= m_keep - 1) stage[at++] = static_cast<uint32_t>(c0 + base + __ffs(m_keep) - 1);
  } else {
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      if ((m_keep >> i) & 1u) stage[at] = static_cast<uint32_t>(c0 + base + i);
      at += (m_keep >> i) & 1u;
    }
  }
  const uint32_t mine = (scan_total >> 16) + (all_eq ? 0u : min(eq0 + (scan_total & 0xffffu), need_eq) - kept0);
  __syncthreads();
  orow += gt0 + kept0;
  for (uint32_t i = tid; i < mine; i += THREADS) orow[i] = static_cast<int32_t>(stage[i]);
  if constexpr (std::is_same<ROWS, RaggedRows>::value) {
    if (rows.after) pdl_wait();
  }
}

// Long rows of which few positions are kept: a cluster that holds a row in registers needs so many
// SMs that few clusters run at once (12 CTAs for a row of 379968: 7 rows).  But almost all keys
// are out of the question, and a sample tells which:
//   1. long_sample_kernel: a lower bound of the ksel-th largest key, four standard deviations
//      below its rank among 2048 samples of the row;
//   2. long_filter_kernel: a CTA per 4096 positions pools them and lists the keys that reach the
//      bound, in order of position;
//   3. long_finish_kernel: a CTA per row selects among its list (some 2 % of the row).
// The counts are exact.  A row whose list does not hold ksel keys, or overflows, is left to the cluster
// kernel, which follows and skips the rows that are done.
// 32 rows of 379968, 4064 kept: 47 us (7 + 21 + 16 + 5 for the skipped clusters), 119 with clusters
// alone; 32 rows of 262144: 39 (67); 128 rows of 131008: 54 (86).  What bounds it is the filter's
// instructions (some thirty per position; the votes alone would take 8 us) and, in the last kernel, the
// chain of steps that one CTA per row takes.
constexpr int LONG_SAMPLES = 2048;
constexpr int LONG_LIST = 16384;     // listed keys of a row that the last kernel takes
constexpr int LONG_THREADS = 512, LONG_CHUNK = LONG_THREADS * 8;
constexpr int LONG_PER_SM = 3;       // CTAs of the filter kernel on an SM
constexpr int LONG_BINS = 2048;

struct RankScratch {
  uint32_t hist[LONG_BINS], warp_sums[32], total, sel_bin, sel_above, sel_count;
};

// One histogram round of 1024 threads over the keys lo .. lo + width: narrows lo, width to the bin
// that holds the krem-th largest of them, takes the keys above the bin off krem and returns how many
// keys the bin holds.  The keys must hold krem in that range.
template <int EPT>
__device__ __forceinline__ uint32_t rank_round(const uint32_t (&key)[EPT], RankScratch& rs, uint32_t& lo,
                                               uint32_t& width, uint32_t& krem, int run = EPT) {
  const int shift = max(0, 21 - __clz(width));  // (width >> shift) < LONG_BINS
  for (int b = threadIdx.x; b < LONG_BINS; b += 1024) rs.hist[b] = 0u;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    if (i >= run) break;  // (the first `run` keys, the same in all threads)
    const uint32_t rel = key[i] - lo;  // wraps for keys below lo
    if (rel <= width) atomicAdd(&rs.hist[rel >> shift], 1u);
  }
  __syncthreads();
  const int b1 = LONG_BINS - 1 - 2 * static_cast<int>(threadIdx.x);  // this thread's bins, from the highest down
  const uint32_t n1 = rs.hist[b1], n0 = rs.hist[b1 - 1];
  const uint32_t above = block_scan<1024>(n0 + n1, rs.warp_sums, &rs.total);
  if (above < krem && krem <= above + n1 + n0) {
    const bool upper = krem <= above + n1;
    rs.sel_bin = upper ? b1 : b1 - 1;
    rs.sel_above = upper ? above : above + n1;
    rs.sel_count = upper ? n1 : n0;
  }
  __syncthreads();
  const uint32_t end = lo + width, bin = rs.sel_bin, count = rs.sel_count;
  krem -= rs.sel_above;
  lo += bin << shift;
  width = min((1u << shift) - 1u, end - lo);
  __syncthreads();  // all have read the results before the next round writes them
  return count;
}

// `want`: the bound is the lower edge of the bin, two rounds of 2048 bins deep, that holds the want-th
// largest sample.
template <int R, int PT>
__global__ void __launch_bounds__(1024) long_sample_kernel(const float* __restrict__ vote, int n, int gsum, int r,
                                                           int pool_type, float divisor, int want,
                                                           uint32_t* __restrict__ meta) {
  __shared__ RankScratch rs;
  __shared__ uint32_t key_max, key_min;
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const float* vrow = vote + static_cast<size_t>(row) * gsum * n;
  if (tid == 0) {
    key_max = 0u;
    key_min = ~0u;
  }
  __syncthreads();
  pdl_wait();
  float tap[2][2 * R + 1];
  int js[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    js[i] = static_cast<int>((static_cast<long long>(tid + 1024 * i) * n + n / 2) / LONG_SAMPLES);
#pragma unroll
    for (int t = 0; t <= 2 * R; ++t) {
      const int j = js[i] + t - R;
      tap[i][t] = static_cast<unsigned>(j) < static_cast<unsigned>(n) ? __ldg(vrow + j) : 0.f;
    }
  }
  for (int g = 1; g < gsum; ++g)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int t = 0; t <= 2 * R; ++t) {
        const int j = js[i] + t - R;
        if (static_cast<unsigned>(j) < static_cast<unsigned>(n)) tap[i][t] += __ldg(vrow + static_cast<size_t>(g) * n + j);
      }
  uint32_t k[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float p = 0.f;
#pragma unroll
    for (int t = 0; t <= 2 * R; ++t)
      if (PT >= 0 || (t - R >= -r && t - R <= r))
        p = (PT >= 0 ? PT == 0 : pool_type == 0) ? fmaxf(p, tap[i][t]) : p + tap[i][t];
    if (PT < 0 && divisor != 0.f) p = p / divisor;
    k[i] = float_to_key(p);
  }
  const uint32_t hi = __reduce_max_sync(0xffffffffu, max(k[0], k[1])), low = __reduce_min_sync(0xffffffffu, min(k[0], k[1]));
  if (lane == 0) {
    atomicMax(&key_max, hi);
    atomicMin(&key_min, low);
  }
  __syncthreads();
  uint32_t lo = key_min, width = key_max - lo, krem = static_cast<uint32_t>(want);
  rank_round(k, rs, lo, width, krem);
  if (width > 0u) rank_round(k, rs, lo, width, krem);
  if (tid == 0) meta[static_cast<size_t>(row) * LONG_META + LONG_THRESHOLD] = max(lo, KEY_MIN);
}

// Persistent: the votes of a CTA's next chunk are on their way while it works on the present one.
// Few instructions per position are what counts here: the halo lies in front of and behind the chunk in
// the same array (so a thread reads its run and its neighbours' as aligned vectors), whole chunks
// skip the checks of the row's end, the pooled values are compared as numbers, and only warps that
// have something to list scan (32 rows of 379968: 31 us with a scan of the block, element-wise
// neighbours and a division per chunk, 21 so).
template <int R, int PT>
__global__ void __launch_bounds__(LONG_THREADS, LONG_PER_SM)
long_filter_kernel(const float* __restrict__ vote, int rows, int n, int gsum, int r, int pool_type, float divisor,
                   int nchunk, int cap, uint32_t* __restrict__ meta, uint2* __restrict__ list) {
  constexpr int PAD = 8;             // halo positions staged on either side
  constexpr int NV = (R + 3) / 4;    // vectors of neighbours read on either side
  constexpr int STEP = LONG_THREADS + LONG_THREADS / 8;  // slot(t + LONG_THREADS) - slot(t)
  static_assert(CL_RMAX <= PAD && LONG_THREADS % 32 == 0, "the halo holds the largest radius");
  __shared__ __align__(16) uint32_t stage[slots_for(LONG_CHUNK + 2 * PAD)];
  __shared__ uint32_t warp_sums[LONG_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* const put = stage + slot(tid + PAD);
  const int h_at = tid < PAD ? tid - PAD : LONG_CHUNK + tid - PAD;  // halo position of the first 2 * PAD threads
  float x[8], h = 0.f;
  uint32_t bound;
  auto fetch = [&](int row, int c0) {
    const bool have_h = tid < 2 * PAD && static_cast<unsigned>(c0 + h_at) < static_cast<unsigned>(n);
    const float* src = vote + static_cast<size_t>(row) * gsum * n + c0;
    const int left = n - c0 - tid;  // positions from this thread's first one to the row's end
    bound = __ldg(meta + static_cast<size_t>(row) * LONG_META + LONG_THRESHOLD);
    if (n - c0 >= LONG_CHUNK) {
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = __ldg(src + tid + LONG_THREADS * u);
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = LONG_THREADS * u < left ? __ldg(src + tid + LONG_THREADS * u) : 0.f;
    }
    if (tid < 2 * PAD) h = have_h ? __ldg(src + h_at) : 0.f;
    for (int g = 1; g < gsum; ++g) {
      src += n;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (LONG_THREADS * u < left) x[u] += __ldg(src + tid + LONG_THREADS * u);
      if (have_h) h += __ldg(src + h_at);
    }
  };
  pdl_wait();
  const int row_step = gridDim.x / nchunk, chunk_step = gridDim.x - row_step * nchunk;
  int next_row = blockIdx.x / nchunk, next_chunk = blockIdx.x - next_row * nchunk;
  if (next_row < rows) fetch(next_row, next_chunk * LONG_CHUNK);
#pragma unroll 1
  while (next_row < rows) {
    const int row = next_row, chunk = next_chunk;
    next_row += row_step;
    next_chunk += chunk_step;
    if (next_chunk >= nchunk) {
      next_chunk -= nchunk;
      ++next_row;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) put[STEP * u] = __float_as_uint(x[u]);
    if (tid < 2 * PAD) stage[slot(h_at + PAD)] = __float_as_uint(h);
    const float least = __uint_as_float(bound & 0x7fffffffu);  // (bounds are keys of values from zero on)
    __syncthreads();
    if (next_row < rows) fetch(next_row, next_chunk * LONG_CHUNK);
    float v[8 * NV + 8], p[8];
#pragma unroll
    for (int q = 0; q < 2 * NV + 2; ++q) {
      const uint4 y = *reinterpret_cast<const uint4*>(stage + slot(tid * 8 + PAD + 4 * (q - NV)));
      v[4 * q] = __uint_as_float(y.x);
      v[4 * q + 1] = __uint_as_float(y.y);
      v[4 * q + 2] = __uint_as_float(y.z);
      v[4 * q + 3] = __uint_as_float(y.w);
    }
    pool8<R, PT>(v + 4 * NV - R, p, r, pool_type, divisor);
    const int base = chunk * LONG_CHUNK + tid * 8;
    uint32_t m_in = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) m_in |= static_cast<uint32_t>(p[i] >= least) << i;
    if (base + 8 > n) m_in &= base < n ? (1u << (n - base)) - 1u : 0u;
    const uint32_t in = __popc(m_in), of_warp = __reduce_add_sync(0xffffffffu, in);
    if (lane == 0) warp_sums[warp] = of_warp;
    __syncthreads();  // (and stage is free)
    if (of_warp || warp == LONG_THREADS / 32 - 1) {
      uint32_t to = __reduce_add_sync(0xffffffffu, lane < warp ? warp_sums[lane] : 0u);
      if (warp == LONG_THREADS / 32 - 1 && lane == 0)
        meta[static_cast<size_t>(row) * LONG_META + LONG_COUNTS + chunk] = to + of_warp;
      uint32_t inc = in;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      to += inc - in;
      uint2* out = list + (static_cast<size_t>(row) * nchunk + chunk) * cap + to;
      int room = cap - static_cast<int>(to);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((m_in >> i) & 1u) {
          if (room-- > 0) *out = make_uint2(__float_as_uint(p[i]) | KEY_MIN, static_cast<uint32_t>(base + i));
          ++out;
        }
    }
  }
}

__global__ void __launch_bounds__(1024) long_finish_kernel(int ksel, int nchunk, int cap, uint32_t* __restrict__ meta,
                                                           const uint2* __restrict__ list,
                                                           int32_t* __restrict__ out_idx) {
  constexpr int EPT = LONG_LIST / 1024;
  constexpr uint32_t NONE = 0u;  // below every listed key
  extern __shared__ __align__(16) uint32_t keys_s[];
  uint32_t* pos_s = keys_s + slots_for(LONG_LIST);
  __shared__ RankScratch rs;
  __shared__ uint32_t first[LONG_META], overflow, key_max;
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  uint32_t* m = meta + static_cast<size_t>(row) * LONG_META;
  if (tid == 0) overflow = key_max = 0u;
  pdl_wait();
  __syncthreads();
  const uint32_t mine = tid < nchunk ? m[LONG_COUNTS + tid] : 0u;
  if (mine > static_cast<uint32_t>(cap)) overflow = 1u;
  const uint32_t before = block_scan<1024>(mine, rs.warp_sums, &rs.total);
  if (tid < nchunk) first[tid] = before;
  const uint32_t total = rs.total;
  __syncthreads();
  const bool ok = !overflow && total >= static_cast<uint32_t>(ksel) && total <= LONG_LIST;
  if (tid == 0) m[LONG_DONE] = ok;
  if (!ok) return;

  // the list, compacted; slots behind its end are NONE
  uint32_t top = 0u;
  const int run = static_cast<int>((total + 4095) / 4096) * 4;  // slots a thread owns, up to EPT
#pragma unroll 8
  for (int u = 0; u < run; ++u) {
    const uint32_t e = tid + 1024 * u;
    uint2 kp = make_uint2(NONE, 0u);
    if (e < total) {
      int c = 0;  // the last chunk whose first entry is at or before e
#pragma unroll
      for (int step = LONG_META / 4; step > 0; step >>= 1)
        if (c + step < nchunk && first[c + step] <= e) c += step;
      kp = __ldg(list + (static_cast<size_t>(row) * nchunk + c) * cap + (e - first[c]));
    }
    keys_s[slot(e)] = kp.x;
    pos_s[slot(e)] = kp.y;
    top = max(top, kp.x);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if (lane == 0) atomicMax(&key_max, top);
  __syncthreads();
  const int base = tid * run;
  uint32_t key[EPT];
#pragma unroll
  for (int i = 0; i < EPT; ++i) key[i] = NONE;
#pragma unroll
  for (int i = 0; i < EPT; i += 4) {
    if (i >= run) break;
    const uint4 v = *reinterpret_cast<const uint4*>(keys_s + slot(base + i));
    key[i] = v.x; key[i + 1] = v.y; key[i + 2] = v.z; key[i + 3] = v.w;
  }

  // until a bin is one key wide or all of it is kept (two rounds as a rule)
  uint32_t lo = m[LONG_THRESHOLD], width = key_max - lo, krem = static_cast<uint32_t>(ksel), all;
  do {
    all = rank_round(key, rs, lo, width, krem, run);
  } while (width > 0u && krem != all);
  const uint32_t T = lo;
  const bool all_eq = krem == all;  // every key from T on is kept
  uint32_t m_keep = 0u, m_eq = 0u;
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    m_keep |= static_cast<uint32_t>(key[i] > T || (all_eq && key[i] == T)) << i;
    m_eq |= static_cast<uint32_t>(!all_eq && key[i] == T) << i;
  }
  const uint32_t packed =
      block_scan<1024>((static_cast<uint32_t>(__popc(m_keep)) << 16) | __popc(m_eq), rs.warp_sums, &rs.total);
  uint32_t eq_seen = packed & 0xffffu, at = (packed >> 16) + min(eq_seen, krem);
  if (all_eq) at = packed >> 16;
  while (m_eq && eq_seen < krem) {  // of the equal keys the lowest positions
    m_keep |= m_eq & (0u - m_eq);
    m_eq &= m_eq - 1;
    ++eq_seen;
  }
  int32_t* orow = out_idx + static_cast<size_t>(row) * ksel;
#pragma unroll
  for (int i = 0; i < EPT; ++i)
    if ((m_keep >> i) & 1u) orow[at++] = static_cast<int32_t>(pos_s[slot(base + i)]);
}

struct ClusterShape {
  int threads, ept, ctas;  // threads per CTA, keys per thread, CTAs per row
  double us = 0.0;         // estimated time (of the shapes of 1024 threads)
};

// How many clusters of c CTAs of 1024 threads (one per SM) run at once on the current device, which is
// asked once: a B200 answers 148, 74, 45, 33, 26, 22, 15, 15, 15, 11 for c = 1 .. 10 and 7 for more.
// When the clusters come in rounds fewer find a place than on an empty device: 52 clusters of five
// take three rounds, eight of nine two.  So sizes above 8 count as 16, and up to 8 the SMs that the
// GPCs leave over (16 with clusters of three or four, 28 with larger ones) are not counted on.
int clusters_at_once(int c) {
  constexpr int MAX_DEV = 64;
  static std::mutex mu;
  static int fit[MAX_DEV][CL_MAX_CLUSTER + 1];
  static std::atomic<bool> known[MAX_DEV];
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return c <= 8 ? sm_count() / c : 0;
  if (!known[dev].load(std::memory_order_acquire)) {
    std::lock_guard<std::mutex> lock(mu);
    if (!known[dev].load(std::memory_order_relaxed)) {
      auto kernel = pool_topk_cluster_kernel<1024, 32, CL_RMAX, -1, OneLength>;
      constexpr int SMEM = slots_for(1024 * 32) * 4;
      const bool ok = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) == cudaSuccess;
      fit[dev][1] = sm_count();
      for (int i = 2; i <= CL_MAX_CLUSTER; ++i) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = i;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(i);
        cfg.blockDim = dim3(1024);
        cfg.dynamicSmemBytes = SMEM;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (!ok || cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
          n = i <= 8 ? 1 : 0;       // (a size that every device takes, or none)
          (void)cudaGetLastError();  // a refusal here is an answer, not an error of the call
        }
        fit[dev][i] = n;
      }
      known[dev].store(true, std::memory_order_release);
    }
  }
  if (c > 8) return fit[dev][CL_MAX_CLUSTER];
  const int in_rounds = (fit[dev][1] - (c <= 2 ? 0 : (c <= 4 ? 16 : 28))) / c;
  return fit[dev][c] < in_rounds ? fit[dev][c] : in_rounds;
}

// What a round of CTAs of 1024 threads takes, in us, by the keys a thread holds: rows that have a CTA to
// themselves, and rows that a cluster shares (0.35 us more for each CTA of it).  Measured in a graph, rows that
// fill the device, kernel size 7 (5: up to two less, 13: two more), an eighth of the positions kept: 8.3,
// 11.0 and 16.4 alone; clusters of two, three and four 10.4, 10.8, 11.3 with 8 keys, 12.4, 12.9, 13.9 with 16,
// 18.1, 18.1, 19.8 with 32.  So the last entry is two to three us high, and 91 to 132 rows of 33000 to 49000
// take three rounds with 16 keys (34) where two with 32 are shorter (31).  With 18.7 there they would take
// those, but rows that are filtered now would come to the clusters, whose time depends on the sample
// (64 rows of 115000: 31 to 35 filtered, 34 to 43 in clusters; 56 of 131008: 36 to 40, and 33 to 43).
struct RoundCost {
  int ept;
  double alone, shared;
};
constexpr RoundCost ROUND_COST[3] = {{8, 8.0, 10.2}, {16, 10.5, 12.5}, {32, 16.5, 20.0}};

// The shape with the smallest estimated time for rows of which the longest has n positions;
// rounds(chunk, c, fit): in how many rounds clusters of c CTAs, of which `fit` find a place at once, come
// when a CTA takes `chunk` positions.  No CTAs: the device holds no cluster that is large enough.
template <typename Rounds>
ClusterShape cheapest_shape(int n, Rounds&& rounds) {
  ClusterShape best = {1024, 32, 0, 1e30};
  for (const RoundCost& cost : ROUND_COST) {
    const int chunk = 1024 * cost.ept, c = (n + chunk - 1) / chunk;
    if (c > CL_MAX_CLUSTER) continue;
    const int fit = clusters_at_once(c);
    if (fit < 1) continue;
    const double us = static_cast<double>(rounds(chunk, c, fit)) * (c == 1 ? cost.alone : cost.shared + 0.35 * c);
    if (us < best.us) best = {1024, cost.ept, c, us};
  }
  return best;
}

// How rows of n positions are cut: the shape with the smallest estimated time.  Up to 4096
// positions small CTAs have the shortest chain, and clusters of them while every CTA has an SM to
// itself (79.6 against 84.2 us for the whole step of 32 rows of 16352).  Beyond, CTAs of 1024 threads
// (one per SM) with 8, 16 or 32 keys a thread take about 8, 10.5 and 16.5 us, 2 to 4 us more when a
// cluster shares a row, and come in rounds when they do not all find a place at once.  No CTAs: the
// device holds no cluster that is large enough.
ClusterShape cluster_shape(int rows, int n) {
  if (n <= 2048) return {256, 8, 1};
  const int small = (n + 4095) / 4096;
  if (small <= 8 && rows * small <= sm_count()) return {512, 8, small};
  return cheapest_shape(n, [&](int, int, int fit) { return (rows + fit - 1) / fit; });
}

// What a launch needs besides the shape.
struct SelectCall {
  const float* vote;
  int rows, n, gsum, r, pool_type;
  float divisor;
  int ksel;
  int32_t* out_idx;
  int discard;
  cudaStream_t stream;
  const uint32_t* meta = nullptr;  // rows marked done here are skipped
};

// Sample ranks four standard deviations to either side of the rank that ksel maps to.
int2 window_ranks(int ksel, int n) {
  const double frac = static_cast<double>(ksel) / n;
  const int delta = static_cast<int>(4.0 * sqrt(CL_SAMPLES * frac * (1.0 - frac))) + 2;
  const int mid = static_cast<int>(frac * CL_SAMPLES);
  return make_int2(mid - delta, mid + delta);
}

template <int THREADS, int EPT, int R, int PT, typename ROWS>
cudaError_t launch_one(const SelectCall& c, int ctas, const ROWS& rows) {
  auto kernel = pool_topk_cluster_kernel<THREADS, EPT, R, PT, ROWS>;
  constexpr int SMEM = slots_for(THREADS * EPT) * 4;
  static DeviceOnce once;
  if (!once.done()) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    once.set();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(c.rows) * ctas);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = c.stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, c.vote, c.n, c.gsum, c.r, c.pool_type, c.divisor, c.ksel,
                            window_ranks(c.ksel, c.n), c.out_idx, ctas, c.discard, c.meta, rows);
}

template <int THREADS, int EPT, typename ROWS>
cudaError_t launch_shape(const SelectCall& c, int ctas, const ROWS& rows) {
  const bool mx = c.pool_type == 0;
#define SNAPKV_CL(RR, PP) launch_one<THREADS, EPT, RR, PP, ROWS>(c, ctas, rows)
  if (c.divisor != 0.f) return SNAPKV_CL(CL_RMAX, -1);
  // the paper's kernel sizes 5, 7 and 13 have instantiations of their own
  if (c.r == 2) return mx ? SNAPKV_CL(2, 0) : SNAPKV_CL(2, 1);
  if (c.r == 3) return mx ? SNAPKV_CL(3, 0) : SNAPKV_CL(3, 1);
  if (c.r == 6) return mx ? SNAPKV_CL(6, 0) : SNAPKV_CL(6, 1);
  return SNAPKV_CL(CL_RMAX, -1);
#undef SNAPKV_CL
}

// The want-th of LONG_SAMPLES samples is the bound that rows of n are filtered with; 0: the list
// would be too long (or the whole row).
int long_want(int n, int ksel) {
  const double p = static_cast<double>(ksel) / n;
  const int want = static_cast<int>(LONG_SAMPLES * p + 4.0 * sqrt(LONG_SAMPLES * p * (1.0 - p))) + 2;
  const double most = (want + 4.0 * sqrt(static_cast<double>(want))) / LONG_SAMPLES * n;
  return most <= LONG_LIST ? want : 0;
}

template <int R, int PT>
cudaError_t launch_filter(const SelectCall& c, int want, int nchunk, int cap, uint32_t* meta, uint2* list) {
  cudaError_t e = launch_pdl(long_sample_kernel<R, PT>, dim3(c.rows), dim3(1024), 0, c.stream, c.vote, c.n, c.gsum,
                             c.r, c.pool_type, c.divisor, want, meta);
  if (e != cudaSuccess) return e;
  const long long chunks = static_cast<long long>(c.rows) * nchunk;
  const int most = LONG_PER_SM * sm_count();
  return launch_pdl(long_filter_kernel<R, PT>, dim3(static_cast<unsigned>(chunks < most ? chunks : most)),
                    dim3(LONG_THREADS), 0, c.stream, c.vote, c.rows, c.n, c.gsum, c.r, c.pool_type, c.divisor, nchunk, cap, meta, list);
}

// `list` holds rows * n * 4 bytes, `meta` LONG_META words per row.
cudaError_t launch_long(const SelectCall& c, int want, uint32_t* meta, uint2* list) {
  const int nchunk = (c.n + LONG_CHUNK - 1) / LONG_CHUNK;
  const int cap = c.n / 2 / nchunk;
  constexpr int SMEM = 2 * slots_for(LONG_LIST) * 4;
  static DeviceOnce once;
  if (!once.done()) {
    const cudaError_t e = cudaFuncSetAttribute(long_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return e;
    once.set();
  }
  const bool mx = c.pool_type == 0;
  auto f = c.divisor != 0.f ? launch_filter<CL_RMAX, -1>
           : c.r == 2       ? (mx ? launch_filter<2, 0> : launch_filter<2, 1>)
           : c.r == 3       ? (mx ? launch_filter<3, 0> : launch_filter<3, 1>)
           : c.r == 6       ? (mx ? launch_filter<6, 0> : launch_filter<6, 1>)
                            : launch_filter<CL_RMAX, -1>;
  const cudaError_t e = f(c, want, nchunk, cap, meta, list);
  if (e != cudaSuccess) return e;
  return launch_pdl(long_finish_kernel, dim3(c.rows), dim3(1024), SMEM, c.stream, c.ksel, nchunk, cap, meta, list,
                    c.out_idx);
}

template <typename ROWS>
cudaError_t launch_rows(const ClusterShape& s, const SelectCall& c, const ROWS& rows) {
  auto f = s.threads == 256 ? launch_shape<256, 8, ROWS>
           : s.threads == 512 ? launch_shape<512, 8, ROWS>
           : s.ept == 8 ? launch_shape<1024, 8, ROWS> : (s.ept == 16 ? launch_shape<1024, 16, ROWS> : launch_shape<1024, 32, ROWS>);
  return f(c, s.ctas, rows);
}

}  // namespace

bool select_cluster_applies(int rows, int n, int pool_kernel) {
  if ((pool_kernel >> 1) > CL_RMAX || n > CL_MAX_CLUSTER * 1024 * 32) return false;
  const int ctas = cluster_shape(rows, n).ctas;
  return ctas > 0 && static_cast<long long>(rows) * ctas < 2147483647ll;
}

cudaError_t launch_pool_topk_cluster(const float* vote, int rows, int n, int pool_kernel,
                                     int pool_type, int ksel, int32_t* out_idx, void* scratch,
                                     cudaStream_t stream, int* launches, int gsum, bool vote_is_scratch) {
  // rows beyond 131072 positions rank average-pooled votes by the mean, shorter ones by the sum
  const float divisor = n > 131072 && pool_type == 1 ? static_cast<float>(pool_kernel) : 0.f;
  SelectCall c = {vote, rows, n, gsum, pool_kernel >> 1, pool_type, divisor, ksel, out_idx,
                  vote_is_scratch ? 1 : 0, stream};
  const ClusterShape shape = cluster_shape(rows, n);
  // The filter's four launches take 24 us and 1.85 us per million votes (within 5 % from 32 rows of
  // 262144 to 128 of 131008); it is taken where that is clearly less than the rounds of the clusters.
  const double filter_us = 24.0 + 1.85e-6 * static_cast<double>(rows) * n;
  const int want = scratch != nullptr && filter_us < 0.9 * shape.us ? long_want(n, ksel) : 0;
  if (want) {
    uint8_t* p = static_cast<uint8_t*>(scratch);
    uint32_t* meta = reinterpret_cast<uint32_t*>(p + ((static_cast<size_t>(rows) * n * 4 + 255) & ~static_cast<size_t>(255)));
    const cudaError_t e = launch_long(c, want, meta, reinterpret_cast<uint2*>(p));
    if (e != cudaSuccess) return e;
    *launches += 3;
    c.meta = meta;
  }
  const cudaError_t e = gsum > 1 ? launch_rows(shape, c, GroupedRows{}) : launch_rows(shape, c, OneLength{});
  if (e != cudaSuccess) return e;
  *launches += 1;
  return cudaGetLastError();
}

// Shape for rows of a ragged batch, `heads` of each of the lengths n, the longest first (a cluster has
// as many CTAs as that one needs, those that a shorter row does not need leave at once): the smallest
// estimated time, as for rows of one length.  128 rows of 8046 to 23968 take one round of CTAs with 32
// keys a thread (16 us) where clusters of two with 16 keys a thread took two (22 us).
constexpr int RAGGED_SHORT = 4096;  // rows up to here take a CTA of 256 or 512 threads
static ClusterShape ragged_shape(const int* n, int count, int heads) {
  if (n[0] <= 2048) return {256, 8, 1};
  if (n[0] <= RAGGED_SHORT) return {512, 8, 1};
  return cheapest_shape(n[0], [&](int chunk, int c, int fit) {
    long long ctas = 0;
    for (int j = 0; j < count; ++j) ctas += static_cast<long long>(heads) * ((n[j] + chunk - 1) / chunk);
    const long long at_once = static_cast<long long>(fit) * c;
    return (ctas + at_once - 1) / at_once;
  });
}

// Whether the rows of a ragged batch, the longest of n_max positions, can share a launch.
bool ragged_select_applies(int n_max, int pool_kernel, int pool_type) {
  if ((pool_kernel >> 1) > CL_RMAX || n_max > CL_MAX_CLUSTER * 1024 * 32) return false;
  if (pool_type == 1 && n_max > 131072) return false;  // two ways of ranking in one launch
  return ragged_shape(&n_max, 1, 1).ctas > 0;
}

cudaError_t launch_ragged_select(const RaggedBatch& rb, const float* vote, int Hq, int W, int pool_kernel,
                                 int pool_type, int ksel, int32_t* out_idx, int* ready, cudaStream_t stream, int* launches) {
  // longest rows first: the last CTAs to start should be short ones
  int order[RAGGED_MAX];
  for (int i = 0; i < rb.count; ++i) {
    int at = i;
    for (; at > 0 && rb.L[order[at - 1]] < rb.L[i]; --at) order[at] = order[at - 1];
    order[at] = i;
  }
  // Where the long rows alone are estimated to take less time, because they come in fewer rounds or can
  // have more CTAs each, the short ones are a launch of their own behind them: a CTA of 1024 threads has an
  // SM to itself and takes 10 us however short its row is, and the small CTAs fit where the long rows' last
  // round leaves SMs over.  (Eight sequences of 822
  // to 24000: 143 us in one launch, 132 in two; sixteen of 300 to 20000 with 8 heads 104.7 and 97.0.
  // Four of 400 to 12283, which take one round either way: 52.4 and 53.4.)
  int n[RAGGED_MAX], longer = 0;
  for (int i = 0; i < rb.count; ++i) n[i] = rb.L[order[i]] - W;
  while (longer < rb.count && n[longer] > RAGGED_SHORT) ++longer;
  if (longer > 0 && longer < rb.count && ragged_shape(n, longer, Hq).us + 1.0 >= ragged_shape(n, rb.count, Hq).us) longer = 0;
  for (int first = 0; first < rb.count;) {
    const int last = first < longer ? longer : rb.count;
    RaggedRows rows = {};
    rows.heads = Hq;
    rows.ready = longer > 0 && longer < rb.count ? ready : nullptr;
    rows.after = first > 0;
    for (int i = first; i < last; ++i) {
      rows.n[i - first] = n[i];
      rows.batch[i - first] = rb.batch[order[i]];
      rows.want[i - first] = window_ranks(ksel, n[i]);
      rows.vote0[i - first] = rb.vote0[order[i]];
    }
    const ClusterShape shape = ragged_shape(rows.n, last - first, Hq);
    if (shape.ctas < 1) return cudaErrorInvalidValue;  // (callers ask ragged_select_applies)
    const SelectCall c = {vote, (last - first) * Hq, rows.n[0], 1, pool_kernel >> 1, pool_type, 0.f, ksel, out_idx, 1, stream};
    const cudaError_t e = launch_rows(shape, c, rows);
    if (e != cudaSuccess) return e;
    *launches += 1;
    first = last;
  }
  return cudaGetLastError();
}

}  // namespace snapkv
