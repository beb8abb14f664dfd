// Window scoring (Eq. 1; Listing 1's compute_attn and the sum over the window):
//   vote[h, j] = sum_i softmax_i(q_i . k / sqrt(d))[j],  j in [0, n)
// computed in two tensor-core passes over K inside ONE persistent kernel.
//
//  pass S (statistics)  S^T tile = Q_rep[128 x d] . K_tile[128 x d]^T : window rows on
//      TMEM lanes, keys on columns.  Each thread owns one window row and keeps a running
//      (max, sum of exp) over the keys it sees: an online softmax without shuffles.
//      When the unit has fewer than 128 window rows the rows are replicated along M and
//      each replica takes a different slice of the tile's keys, so all four epilogue
//      warps of a warpgroup stay busy.  Each CTA publishes one log2-sum-exp per window row
//      for the keys it saw (its "partial") in a slot of the unit that is its own flag.
//  pass V (votes)       S tile = K_tile[128 x d] . Q[ncols x d]^T : keys on TMEM lanes,
//      window rows on columns.  Once every slot of the unit has been written, the CTA folds
//      the partials, in slot order, into one log2-sum-exp per window row;
//      then each thread owns one key and adds exp2(s*c - lse) over the W columns of each
//      head: the sum over the window is a serial add per thread.
//
// Units (batch, KV head, head sub-group) are grouped into waves small enough for L2; the
// kernel walks the phases  S(0), S(1), V(0), S(2), V(1), ...  so that part of the second sweep
// over a wave's keys is served by L2 and the partials a vote phase needs were published
// a whole phase earlier.  Within a phase the wave's tiles are split evenly over the CTAs.
// One CTA per SM and no more CTAs than SMs, so all of them are resident and waiting on
// another CTA's partials cannot starve it.
//
// Warp roles: warp 0 issues TMA loads (K tiles into a ring of stages, Q per work item
// into two buffers), warp 1 issues tcgen05.mma into four TMEM accumulator buffers, warps
// 2-9 (two warpgroups) read the accumulators back with tcgen05.ld and do the fp32 softmax
// arithmetic; with 64 or more query columns per unit a second set of eight softmax warps
// (12-19) takes every other tile, each warpgroup of a set working on half of the columns:
// the epilogue is bound by instruction latency, and four warps per scheduler hide it where
// two do not.  Warps 10 and 11 are the book-keepers: warp 10 publishes the partial
// statistics the softmax warps leave in shared memory, warp 11 fetches and folds the
// partials of the coming vote items' units while the softmax warps are still busy.  The single-thread roles (TMA and MMA issue) are entered through elect.sync:
// the compiler then keeps descriptors and addresses in uniform registers, which cut the
// time per tcgen05.mma issue by about a third against a lane-index test.
//
// A batch of prompts of different lengths runs in the same launch: every sequence is a wave (or
// several) of its own behind the others', with its own lengths, tensor map and vote rows.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "launch.cuh"
#include "sm100_ptx.cuh"
#include "snapkv_internal.h"

namespace snapkv {

namespace score {

constexpr int STAGES = 4;
constexpr int NBUF = 4;               // TMEM accumulator buffers of 128 columns
constexpr int TMEM_COLS = 512;
constexpr int SUBTILE_BYTES = 128 * 128;  // 128 rows x 64 bf16, 128-byte swizzled
constexpr int EPI_WARPS = 8;           // softmax warps per set (two warpgroups)
// Warps: 0 producer, 1 MMA issuer, 2-9 softmax set 0, 10 publisher, 11 lse fetcher and, in
// split mode, 12-19 softmax set 1.
constexpr int threads_for(bool split) { return split ? 640 : 384; }
constexpr long long WAVE_BYTES = 64ll << 20;
constexpr int RAGGED_AHEAD = 64;      // tiles per block, the same for the sequences of a ragged batch
constexpr int MAX_RECORDS = 192;      // work items of a CTA that one launch can hold
constexpr int NPB = 2;                // buffers for partial statistics (book-keeper queue)
constexpr int NLB = 8;                // buffers for merged log-sum-exp rows
constexpr int FOLD = 8;               // partials folded at a time
constexpr int MERGE_SEGS = 32;        // partials staged in shared memory at a time (a multiple of FOLD)

struct ScoreArgs {
  int L, n, W, Hkv;
  int hpu, ncols, npad;
  int sub_per_kv, g;
  int units, upw, nwaves;   // units per wave, number of waves (of this launch, from wave0 on)
  int wave0;
  int per;                  // most work items of a CTA in one phase
  int T1, T2;               // tiles per unit in the statistics / vote pass
  int maxseg;               // partial slots per unit
  int mask_n;               // window row i sees keys j <= mask_n + i (n, or n minus a shard's first position)
  int stats_only;           // 1: statistics pass alone (a shard's partial log-sum-exp), no votes
  int votes_only;           // 1: lse2 and the counters are already set, no statistics pass
  int withhold;             // 1: nothing is published (self-test of the waits for it)
  int both_fold;            // 1: the publisher folds half of the columns (shared_fold)
  unsigned long long wait_ns;  // time limit of every device-side wait
  const int32_t* page_table;   // paged K: [batch][pages_per_seq] page numbers, else nullptr
  int pages_per_seq, page_size;
  float c2;                 // log2(e) / sqrt(d)
  float* partials;          // [units][maxseg][MAX_COLS] log2-sum-exp of one CTA's share
  float* lse2;              // [units][MAX_COLS] minus the log2-sum-exp per window row, when supplied
  int* counters;            // [units] partials of a statistics-only launch; above zero when lse2 was supplied
  int* status;
  float* vote;
};

template <int D>
struct Smem {
  static constexpr int SUBT = D / 64;
  static constexpr int Q_BYTES = SUBT * SUBTILE_BYTES;
  static constexpr int STAGE_BYTES = SUBT * SUBTILE_BYTES;
  static constexpr int OFF_Q = 0;                            // two Q buffers
  static constexpr int OFF_K = 2 * Q_BYTES;
  static constexpr int OFF_BAR = OFF_K + STAGES * STAGE_BYTES;
  // barriers: full[STAGES], empty[STAGES], tf[NBUF], te[NBUF], qfull[2], qempty[2], drain,
  // pfull[NPB], pempty[NPB] (partial statistics), lfull[NLB], lempty[NLB] (log-sum-exp)
  static constexpr int NBAR = 2 * STAGES + 2 * NBUF + 5 + 2 * NPB + 2 * NLB;
  static constexpr int OFF_MISC = OFF_BAR + ((NBAR * 8 + 15) & ~15);  // tmem ptr, abort flag, wait limit
  static constexpr int OFF_PART = OFF_MISC + 16;              // float2 [NPB][2 sets][8][32]
  static constexpr int OFF_LSE = OFF_PART + NPB * 16 * 32 * 8; // float [NLB][128]
  static constexpr int OFF_MERGE = OFF_LSE + NLB * 128 * 4;   // float [MERGE_SEGS][128]
  static constexpr int OFF_ITEMS = OFF_MERGE + MERGE_SEGS * 128 * 4;  // ItemRecord [MAX_RECORDS]
  static constexpr int OFF_ORDER = OFF_ITEMS + MAX_RECORDS * 16;      // uint16 [MAX_RECORDS]
  static constexpr int TOTAL = OFF_ORDER + MAX_RECORDS * 2;
  static_assert(OFF_PART % 16 == 0 && OFF_LSE % 16 == 0 && OFF_MERGE % 16 == 0,
                "float4 reads of the lse buffers, 16-byte copies into the merge buffer");
  static constexpr int DYN_BYTES = TOTAL + 1024;            // slack for 1024-byte alignment
};

// Wait of the abort path (the abort flag is already set, so it is not looked at): for a copy
// or an MMA that is in flight and will complete.
__device__ __forceinline__ bool mbar_wait_drain(uint32_t bar, uint32_t parity,
                                                unsigned long long limit_ns) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}

// Warp-wide wait for a warp that is off the critical path: backs off between polls so
// that it does not take issue slots from the softmax warps of its scheduler.
__device__ __forceinline__ bool mbar_wait_warp_relaxed(uint32_t bar, uint32_t parity,
                                                       volatile int* abort_flag, int code) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    __nanosleep(250);
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    int stop = 0;
    if ((threadIdx.x & 31) == 0) {
      if (*abort_flag != 0) stop = 1;
      else if (globaltimer_ns() - t0 > wait_limit_ns(abort_flag)) { *abort_flag = code; stop = 1; }
    }
    if (__shfl_sync(0xffffffffu, stop, 0)) return false;
  }
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_relaxed(float* p, float v) {
  asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
// N consecutive floats (N = 1, 2 or 4) in one load.
template <int N>
__device__ __forceinline__ void ld_relaxed(const float* p, float (&v)[N]) {
  static_assert(N == 1 || N == 2 || N == 4, "vector widths");
  if constexpr (N == 1)
    asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v[0]) : "l"(p) : "memory");
  else if constexpr (N == 2)
    asm volatile("ld.relaxed.gpu.global.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "l"(p) : "memory");
  else
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "l"(p)
                 : "memory");
}

template <int N>
__device__ __forceinline__ void lds(uint32_t addr, float (&v)[N]) {
  if constexpr (N == 1)
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[0]) : "r"(addr) : "memory");
  else if constexpr (N == 2)
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(addr) : "memory");
  else
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void sts4(uint32_t addr, float x) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "f"(x) : "memory");
}

// 16 bytes from global memory (past L1) to shared memory, asynchronously.
__device__ __forceinline__ void copy16_async(uint32_t dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Adds partials (log2-sum-exp each) to a running maximum M (at least -1e30) and sum S of
// exp2(. - M), in order.  The maxima come first, so that the exponentials do not wait for one
// another: only the sums are a chain, one fused multiply-add per partial.  Of the two factors
// exp2(M - Mn) and exp2(p - Mn), Mn = max(M, p), one is exactly 1: one exponential per partial.
__device__ __forceinline__ void fold_partials(const float (&pv)[FOLD], float& M, float& S) {
  float scale[FOLD], term[FOLD];
#pragma unroll
  for (int i = 0; i < FOLD; ++i) {
    const bool up = pv[i] > M;
    const float e = ex2_approx(-fabsf(pv[i] - M));
    scale[i] = up ? e : 1.f;
    term[i] = up ? 1.f : e;
    M = fmaxf(M, pv[i]);
  }
#pragma unroll
  for (int i = 0; i < FOLD; ++i) S = fmaf(S, scale[i], term[i]);
}

// One piece of work: tiles [t0, t1) of one unit in one pass.  `seq` and `flip` matter to ragged
// batches alone: the sequence, and which set of softmax warps takes the first tile.
struct Item {
  int unit, t0, t1, vote, slot, nseg, seq, flip;
};
// The same in shared memory: unit | seq << 24 | flip << 31, tiles, slot | nseg << 16.
struct ItemRecord {
  uint32_t what;
  int t0, t1;
  uint32_t seg;
};

// The sequences of a ragged batch, passed by value with the launch (in constant memory, no copies
// to the device, safe to capture in a graph).
struct RaggedSeq {
  int L, n;            // prompt length, prefix length
  int upw, nwaves;     // units per wave, waves
  int T1, T2;          // tiles per unit in the statistics / vote pass
  int maxseg;          // partial slots per unit
  int batch;           // index in the caller's batch
  int rot;             // which block takes the first share of its tiles
  int map;             // its K tensor map
  long long part0;     // first partial slot
  long long vote0;     // first vote
};
template <int MAPS>
struct RaggedSeqs {
  CUtensorMap maps[MAPS];
  RaggedSeq s[RAGGED_MAX];
  int nseq, units_per_seq;
  int waves;           // of all sequences
};
struct NotRagged {};

// Quotients of tile arithmetic, in 32 bits whenever the dividend fits.
__host__ __device__ __forceinline__ uint32_t quotient(unsigned long long x, uint32_t y) {
  return (x >> 32) == 0 ? static_cast<uint32_t>(x) / y : static_cast<uint32_t>(x / y);
}

// The share of one CTA in one phase: the phase's TT = nu * T tiles (units u0 .. u0+nu-1, T tiles
// each) are cut into G consecutive shares, the CTA playing part `cr` owning tiles
// [cr*TT/G, (cr+1)*TT/G); a share that crosses a unit boundary is one item per unit.
struct Share {
  uint32_t lo, hi;
  int u0, nu, T, T1, cr, G;

  __host__ __device__ __forceinline__ Share(int cr_, int G_, int u0_, int nu_, int T_, int T1_)
      : u0(u0_), nu(nu_), T(T_), T1(T1_), cr(cr_), G(G_) {
    const unsigned long long TT = static_cast<unsigned long long>(nu) * static_cast<uint32_t>(T);
    lo = quotient(static_cast<uint32_t>(cr) * TT, G);
    hi = quotient(static_cast<uint32_t>(cr + 1) * TT, G);
  }
  // Item m of the share, which ends where its unit does; an empty one (t0 = t1) behind the last.
  __host__ __device__ __forceinline__ Item item(int m) const {
    Item it = {};
    const uint32_t ul = lo / static_cast<uint32_t>(T) + static_cast<uint32_t>(m);
    const uint32_t pos = m == 0 ? lo : ul * static_cast<uint32_t>(T);
    if (pos >= hi) return it;
    it.unit = u0 + static_cast<int>(ul);
    it.t0 = static_cast<int>(pos - ul * static_cast<uint32_t>(T));
    const uint32_t t1 = static_cast<uint32_t>(it.t0) + (hi - pos);
    it.t1 = t1 < static_cast<uint32_t>(T) ? static_cast<int>(t1) : T;
    it.flip = static_cast<int>((pos - lo) & 1);  // tiles of this phase that this block has had before
    // where this CTA's partial of the unit goes and how many partials the unit gets follow from
    // the statistics-pass partition of the unit's wave
    const uint32_t T1u = static_cast<uint32_t>(T1), TT1 = static_cast<uint32_t>(nu) * T1u;
    if (TT1 >= static_cast<uint32_t>(G)) {  // every CTA has tiles: a unit's owners are consecutive CTAs
      // the CTA whose share contains tile x: the largest c with c*TT1/G <= x
      auto owner = [&](uint32_t x) {
        return static_cast<int>(quotient((x + 1ull) * static_cast<uint32_t>(G) + TT1 - 1, TT1)) - 1;
      };
      const int first = owner(ul * T1u);
      it.slot = cr - first;
      it.nseg = owner(ul * T1u + T1u - 1) - first + 1;
    } else {  // fewer tiles than CTAs: one tile per owner, one partial per tile
      it.slot = it.t0;
      it.nseg = T1;
    }
    return it;
  }
};

// One phase: a wave (of a sequence) in one of the sweeps.  `ord` counts the waves of the launch.
struct Phase {
  int seq, wave, vote, ord;
};

// Phase p of the launch.  Statistics run WAVE_LAG waves ahead of votes: S(0) S(1) V(0) S(2) V(1) ...
__host__ __device__ __forceinline__ Phase phase_at(const ScoreArgs& a, NotRagged, int, int p) {
  int s = a.votes_only ? a.nwaves : 0, v = 0;
  Phase ph = {0, 0, 0, 0};
  for (int i = 0; i <= p; ++i) {
    ph.vote = !(s < a.nwaves && (a.stats_only || s - v < WAVE_LAG));
    ph.ord = ph.vote ? v++ : s++;
  }
  ph.wave = a.wave0 + ph.ord;
  return ph;
}
__host__ __device__ __forceinline__ int phase_count(const ScoreArgs& a, NotRagged) {
  return (a.votes_only || a.stats_only) ? a.nwaves : 2 * a.nwaves;
}
// CTA `cta`'s share of a phase.  TT is seldom a multiple of G, so some CTAs get one tile less than
// the others; which ones moves on by one CTA from phase to phase, so that over the phases of a
// launch no CTA carries the longer share every time.
__host__ __device__ __forceinline__ Share share_of(const ScoreArgs& a, NotRagged, const Phase& ph, int cta, int G) {
  const int u0 = ph.wave * a.upw;
  return Share((cta + 2 * ph.wave + ph.vote) % G, G, u0, a.upw < a.units - u0 ? a.upw : a.units - u0,
               ph.vote ? a.T2 : a.T1, a.T1);
}
__host__ __device__ __forceinline__ int tiles_before(const ScoreArgs&, NotRagged, const Phase&, int, int) { return 0; }

// The same for a ragged batch.  Each sequence is cut as a call of its own would cut it (the same
// shares, partials and order of additions, so its results do not depend on the batch), and the
// waves of the sequences follow one another with the statistics at least WAVE_LAG waves and
// RAGGED_AHEAD tiles per block ahead: the hand-over of a wave's statistics takes some microseconds,
// the tiles of a short sequence less than one.  (Waiting costs more than reading the keys again
// from HBM: eight sequences of 822 to 24000 positions took 175 us with 10 tiles, 155 with 16,
// 145 with 64 and 147 without a limit.)  Block c plays the part of block (c + rot) % G of
// such a call, so that short sequences occupy different blocks; tiles_before restores the parity
// with which that block would have met a statistics item's first tile.
template <int MAPS>
__host__ __device__ __forceinline__ Phase phase_at(const ScoreArgs& a, const RaggedSeqs<MAPS>& rs, int G, int p) {
  int s_seq = a.votes_only ? rs.nseq : 0, s_wave = 0, v_seq = 0, v_wave = 0, s_ord = 0, v_ord = 0, tiles = 0;
  Phase ph = {0, 0, 0, 0};
  for (int i = 0; i <= p; ++i) {
    ph.vote = !(s_seq < rs.nseq && (s_ord - v_ord < WAVE_LAG || tiles < RAGGED_AHEAD * G));
    ph.seq = ph.vote ? v_seq : s_seq;
    ph.wave = ph.vote ? v_wave : s_wave;
    ph.ord = ph.vote ? v_ord++ : s_ord++;
    const RaggedSeq& q = rs.s[ph.seq];
    const int left = rs.units_per_seq - ph.wave * q.upw;
    const int wave_tiles = (q.T1 < 1 << 16 ? q.T1 : 1 << 16) * (q.upw < left ? q.upw : left);
    int& wave = ph.vote ? v_wave : s_wave;
    tiles += ph.vote ? -wave_tiles : wave_tiles;
    if (++wave == q.nwaves) {
      wave = 0;
      ++(ph.vote ? v_seq : s_seq);
    }
  }
  return ph;
}
template <int MAPS>
__host__ __device__ __forceinline__ int phase_count(const ScoreArgs& a, const RaggedSeqs<MAPS>& rs) {
  return a.votes_only ? rs.waves : 2 * rs.waves;
}
template <int MAPS>
__host__ __device__ __forceinline__ Share share_of(const ScoreArgs&, const RaggedSeqs<MAPS>& rs, const Phase& ph, int cta, int G) {
  const RaggedSeq& q = rs.s[ph.seq];
  const int u0 = ph.wave * q.upw, left = rs.units_per_seq - u0;
  return Share((cta + q.rot + 2 * ph.wave + ph.vote) % G, G, u0, q.upw < left ? q.upw : left, ph.vote ? q.T2 : q.T1,
               q.T1);
}
template <int MAPS>
__host__ __device__ __forceinline__ int tiles_before(const ScoreArgs& a, const RaggedSeqs<MAPS>& rs, const Phase& ph, int cta, int G) {
  int before = 0;  // in earlier phases of the sequence
  if (!ph.vote)
    for (int e = 0; e < ph.wave; ++e)
      for (int v = 0; v < (e + WAVE_LAG <= ph.wave ? 2 : 1); ++v) {
        const Share earlier = share_of(a, rs, Phase{ph.seq, e, v, 0}, cta, G);
        before += static_cast<int>(earlier.hi - earlier.lo);
      }
  return before;
}

// NCH = npad / 32: how many 32-column chunks of the accumulator a thread reads per tile.
// SEQS: NotRagged, or the RaggedSeqs of a batch (tmK is not used then).
template <int D, int NCH, bool SPLIT, typename SEQS>
__global__ void __launch_bounds__(threads_for(SPLIT), 1)
score_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ,
             const ScoreArgs a, const __grid_constant__ SEQS rs) {
  constexpr bool RAGGED = !std::is_same<SEQS, NotRagged>::value;
  using SM = Smem<D>;
  constexpr int SUBT = SM::SUBT;
  constexpr int NPAD = NCH * 32;
  constexpr int REPS = 128 / NPAD;
  constexpr int NSET = SPLIT ? 2 : 1;  // sets of softmax warps
  // In split mode the fetcher folds the columns in two halves, and the publisher takes one of them.
  constexpr int HALVES = SPLIT && !RAGGED ? 2 : 1;
  const bool both_fold = HALVES == 2 && a.both_fold;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t k_s = sbase + SM::OFF_K;
  const uint32_t bar0 = sbase + SM::OFF_BAR;
  auto q_s = [&](int b) { return sbase + SM::OFF_Q + b * SM::Q_BYTES; };
  auto stage_addr = [&](int s, int sb) { return k_s + s * SM::STAGE_BYTES + sb * SUBTILE_BYTES; };
  auto bar_full = [&](int s) { return bar0 + 8u * s; };
  auto bar_empty = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto bar_tf = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
  auto bar_te = [&](int b) { return bar0 + 8u * (2 * STAGES + NBUF + b); };
  auto bar_qf = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 * NBUF + b); };
  auto bar_qe = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 * NBUF + 2 + b); };
  const uint32_t bar_drain = bar0 + 8u * (2 * STAGES + 2 * NBUF + 4);
  constexpr int BAR_P = 2 * STAGES + 2 * NBUF + 5;
  auto bar_pf = [&](int b) { return bar0 + 8u * (BAR_P + b); };
  auto bar_pe = [&](int b) { return bar0 + 8u * (BAR_P + NPB + b); };
  auto bar_lf = [&](int b) { return bar0 + 8u * (BAR_P + 2 * NPB + b); };
  auto bar_le = [&](int b) { return bar0 + 8u * (BAR_P + 2 * NPB + NLB + b); };
  volatile uint32_t* tmem_ptr_s = reinterpret_cast<volatile uint32_t*>(smem + SM::OFF_MISC);
  volatile int* abort_s = reinterpret_cast<volatile int*>(smem + SM::OFF_MISC + 4);
  float2* part_s = reinterpret_cast<float2*>(smem + SM::OFF_PART);
  float* lse_s = reinterpret_cast<float*>(smem + SM::OFF_LSE);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int cta = blockIdx.x;
  const int G = gridDim.x;

  if (threadIdx.x == 0) {
    // (the descriptors come with the launch: no need to wait for the previous kernel)
    if constexpr (!RAGGED) tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmQ);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(bar_tf(b), 1);
      mbar_init(bar_te(b), EPI_WARPS);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_qf(b), 1);
      mbar_init(bar_qe(b), 1);
    }
    for (int b = 0; b < NPB; ++b) {
      mbar_init(bar_pf(b), EPI_WARPS * NSET);
      mbar_init(bar_pe(b), 1);
    }
    for (int b = 0; b < NLB; ++b) {
      mbar_init(bar_lf(b), both_fold ? 2 : 1);
      mbar_init(bar_le(b), EPI_WARPS * NSET);
    }
    mbar_init(bar_drain, 1);
    *abort_s = 0;
    *reinterpret_cast<volatile unsigned long long*>(abort_s + 1) = a.wait_ns;
    mbar_fence_init();
  }
  // The work items of this CTA, one per thread: `per` records for each wave in each sweep and
  // the order of the phases.  (Walking the list cost a single thread 2500 cycles of divisions an
  // item, in every role: a ragged batch of short prompts did little else.)
  ItemRecord* items_s = reinterpret_cast<ItemRecord*>(smem + SM::OFF_ITEMS);
  uint16_t* order_s = reinterpret_cast<uint16_t*>(smem + SM::OFF_ORDER);
  const int nphase = phase_count(a, rs);
  // (warps 0 and 1 are busy with the barriers and the tensor memory)
  for (int i = static_cast<int>(threadIdx.x) - 64; i >= 0 && i < nphase * a.per; i += threads_for(SPLIT) - 64) {
    const int m = i / nphase, p = i - m * nphase;
    const Phase ph = phase_at(a, rs, G, p);
    if (m == 0) order_s[p] = static_cast<uint16_t>(2 * ph.ord + ph.vote);
    const Share share = share_of(a, rs, ph, cta, G);
    const int before = tiles_before(a, rs, ph, cta, G);
    const Item it = share.item(m);
    items_s[(2 * ph.ord + ph.vote) * a.per + m] =
        ItemRecord{static_cast<uint32_t>(it.unit) | static_cast<uint32_t>(ph.seq) << 24 |
                       static_cast<uint32_t>((it.flip + before) & 1) << 31,
                   it.t0, it.t1, static_cast<uint32_t>(it.slot) | static_cast<uint32_t>(it.nseg) << 16};
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_ptr_s)), TMEM_COLS);
    tmem_relinquish();
  }
  // everything above touched only this CTA's shared memory and TMEM; from here on the
  // kernel reads and writes global memory, so the previous kernel must be complete
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_s;

  // Item m of phase 2 * wave + sweep.
  auto item_at = [&](int phase, int m) {
    const ItemRecord r = items_s[phase * a.per + m];
    Item it;
    it.unit = static_cast<int>(r.what & 0xffffffu);
    it.seq = RAGGED ? static_cast<int>(r.what >> 24 & 0x7fu) : 0;
    it.flip = static_cast<int>(r.what >> 31);
    it.t0 = r.t0;
    it.t1 = r.t1;
    it.vote = phase & 1;
    it.slot = static_cast<int>(r.seg & 0xffffu);
    it.nseg = static_cast<int>(r.seg >> 16);
    return it;
  };
  // Calls f(item) for the CTA's items in schedule order until it returns false.
  auto each_item = [&](auto&& f) {
    for (int p = 0, m = 0; p < nphase;) {
      const Item it = item_at(order_s[p], m);
      if (it.t0 < it.t1 && !f(it)) break;
      if (++m == a.per) {
        m = 0;
        ++p;
      }
    }
  };
  auto first_head = [&](const Item& it, int* ukv) {
    *ukv = it.unit / a.sub_per_kv;
    const int sub = it.unit - *ukv * a.sub_per_kv;
    if constexpr (RAGGED) *ukv += rs.s[it.seq].batch * a.Hkv;
    return *ukv * a.g + sub * a.hpu;  // flat over the batch
  };
  auto unit_of = [&](const Item& it) {  // index of the unit's counter and supplied normalisers
    if constexpr (RAGGED) return it.seq * rs.units_per_seq + it.unit;
    else return it.unit;
  };
  auto slots_of = [&](const Item& it) -> float* {  // the unit's partials
    if constexpr (RAGGED)
      return a.partials + (rs.s[it.seq].part0 + static_cast<long long>(it.unit) * rs.s[it.seq].maxseg) * MAX_COLS;
    else
      return a.partials + static_cast<size_t>(it.unit) * a.maxseg * MAX_COLS;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (elect_one()) {
      const uint64_t pol_first = l2_policy_evict_first();
      int git = 0;      // tiles issued so far (ring position)
      int nitem = 0;    // items started so far (Q buffer position)
      each_item([&](const Item& it) {
        int ukv;
        const int qrow0 = first_head(it, &ukv) * a.W;
        const CUtensorMap* mapK = &tmK;
        if constexpr (RAGGED) mapK = &rs.maps[rs.s[it.seq].map];
        const int qb = nitem & 1;
        if (!mbar_wait_thread(bar_qe(qb), ((nitem >> 1) & 1) ^ 1, abort_s, WAIT_Q_FULL)) return false;
        if (it.vote) {
          mbar_expect_tx(bar_qf(qb), SUBT * NPAD * 128);
          for (int sb = 0; sb < SUBT; ++sb)
            tma_load_2d(q_s(qb) + sb * SUBTILE_BYTES, &tmQ, bar_qf(qb), sb * 64, qrow0);
        } else {
          mbar_expect_tx(bar_qf(qb), SUBT * 128 * 128);
          for (int rep = 0; rep < REPS; ++rep)
            for (int sb = 0; sb < SUBT; ++sb)
              tma_load_2d(q_s(qb) + sb * SUBTILE_BYTES + rep * NPAD * 128, &tmQ, bar_qf(qb),
                          sb * 64, qrow0);
        }
        ++nitem;
        const int kb = ukv / a.Hkv, kh = ukv - kb * a.Hkv;  // the K map is (d, L, Hkv, B); ragged: B = 1
        for (int t = it.t0; t < it.t1; ++t, ++git) {
          const int s = git % STAGES;
          const uint32_t ph = (git / STAGES) & 1;
          if (!mbar_wait_thread(bar_empty(s), ph ^ 1, abort_s, WAIT_PRODUCER_EMPTY)) return false;
          mbar_expect_tx(bar_full(s), SM::STAGE_BYTES);
          int key0 = t * TILE_KEYS;
          int kslab = RAGGED ? 0 : kb;  // outermost coordinate of the K map: the batch, or the page of the pool
          if (a.page_table) {
            // a page holds a whole number of tiles: the tile's 128 keys sit in one page
            const int pg = key0 / a.page_size;
            kslab = __ldg(a.page_table + static_cast<size_t>(kb) * a.pages_per_seq + pg);
            key0 -= pg * a.page_size;
          }
          // the vote pass is the last reader of a key tile: its lines may leave L2 first,
          // which keeps the next wave's statistics-pass lines resident instead
          for (int sb = 0; sb < SUBT; ++sb) {
            if (it.vote)
              tma_load_4d_hint(stage_addr(s, sb), mapK, bar_full(s), sb * 64, key0, kh, kslab, pol_first);
            else
              tma_load_4d(stage_addr(s, sb), mapK, bar_full(s), sb * 64, key0, kh, kslab);
          }
        }
        return true;
      });
      if (*abort_s != 0) {
        // let every copy in flight land before the CTA's shared memory goes away
        for (int b = 0; b < 2; ++b) {
          int last = -1;
          for (int i = b; i < nitem; i += 2) last = i;
          if (last >= 0) mbar_wait_drain(bar_qf(b), (last >> 1) & 1, a.wait_ns);
        }
        for (int s = 0; s < STAGES; ++s) {
          int last = -1;
          for (int i = s; i < git; i += STAGES) last = i;
          if (last >= 0) mbar_wait_drain(bar_full(s), (last / STAGES) & 1, a.wait_ns);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // One key tile per instruction.  Two tiles as one 128 x 256 x 16 instruction complete together:
    // both sets of softmax warps then wait for the tensor pipe at the same time and the
    // exponentials stand still; tile by tile they take turns (78.3 -> 76.7 us on the 16K MHA
    // workload; the gain on the 32K GQA one is within its spread).
    if (elect_one()) {
      const uint32_t idesc_s = umma_idesc_bf16(128, 128);
      const uint32_t idesc_v = umma_idesc_bf16(128, NPAD);
      int git = 0, nitem = 0;
      each_item([&](const Item& it) {
        const int qb = nitem & 1;
        if (!mbar_wait_thread(bar_qf(qb), (nitem >> 1) & 1, abort_s, WAIT_Q_FULL)) return false;
        ++nitem;
        const uint64_t qd0 = umma_desc_k128(q_s(qb));
        const int nt = it.t1 - it.t0;
        for (int k = 0; k < nt; ++k, ++git) {
          const int s = git % STAGES;
          const uint32_t ph = (git / STAGES) & 1;
          const int buf = git & (NBUF - 1);
          const uint32_t ub = (git / NBUF) & 1;
          if (!mbar_wait_thread(bar_full(s), ph, abort_s, WAIT_MMA_FULL)) return false;
          if (!mbar_wait_thread(bar_te(buf), ub ^ 1, abort_s, WAIT_MMA_TMEM_EMPTY)) return false;
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + buf * 128;
          // One descriptor per operand and tile; the eight K-slices of the tile differ from it
          // by constants (the start-address field counts 16-byte units and the operands sit
          // below 256 KB, so adding to the low word never carries into another field).  The
          // issuing thread is a single in-order instruction stream: every instruction saved
          // per tcgen05.mma shortens the time between two of them.
          const uint64_t kd0 = umma_desc_k128(stage_addr(s, 0));
          constexpr uint64_t K_SB = SUBTILE_BYTES >> 4;  // next 64 elements of d
          constexpr uint64_t Q_SB = SUBTILE_BYTES >> 4;
          if (it.vote) {
#pragma unroll
            for (int sb = 0; sb < SUBT; ++sb)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                tc_mma_bf16(d_tmem, kd0 + (sb * K_SB + kk * 2), qd0 + (sb * Q_SB + kk * 2), idesc_v,
                            (sb | kk) != 0);
          } else {
#pragma unroll
            for (int sb = 0; sb < SUBT; ++sb)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                tc_mma_bf16(d_tmem, qd0 + (sb * Q_SB + kk * 2), kd0 + (sb * K_SB + kk * 2), idesc_s,
                            (sb | kk) != 0);
          }
          tc_commit(bar_empty(s));
          tc_commit(bar_tf(buf));
        }
        tc_commit(bar_qe(qb));  // the item's MMAs are the last readers of its Q buffer
        return true;
      });
      if (*abort_s != 0) {
        tc_commit(bar_drain);
        mbar_wait_drain(bar_drain, 0, a.wait_ns);
      }
    }
  } else if (warp < 2 + EPI_WARPS || warp >= 4 + EPI_WARPS) {
    // ------------------------------------------------------------ softmax warps
    // SPLIT: both warpgroups work on every tile, each on half of the accumulator columns
    // (CPT columns per thread); the -lse values of a vote item then fit in registers.
    // Otherwise the warpgroups alternate tiles and take all NPAD columns.
    constexpr int CPT = SPLIT ? NPAD / 2 : NPAD;
    constexpr int VCH = CPT / 32;
    // SPLIT also has two sets of softmax warps: set 0 takes the even tiles (by ring position)
    // and set 1 the odd ones, so four warps per scheduler hide each other's latencies.
    const int set = warp >= 4 + EPI_WARPS ? 1 : 0;
    const int wg = ((set ? warp - (4 + EPI_WARPS) : warp - 2) >> 2);
    const int q = warp & 3;  // TMEM lane quarter this warp may read
    const uint32_t lane_sel = static_cast<uint32_t>(32 * q) << 16;
    const int rrow = 32 * q + lane;  // TMEM lane
    const int rep = rrow / NPAD;
    const int qcol = rrow - rep * NPAD;
    const int wrow = qcol % a.W;
    int jmax = min(a.L - 1, a.mask_n + wrow);  // last key window row wrow sees
    int jfree = min(a.L - 1, a.mask_n);        // keys up to here are seen by every row
    const int coff = SPLIT ? wg * CPT : 0;               // first accumulator column of this thread
    const bool w16 = (a.W & 15) == 0;
    const int gpw = a.W >> 4;  // 16-column groups per head (when W is a multiple of 16)
    const uint32_t te_arrivals = SPLIT ? 1 : 2;          // the barrier expects 8 per tile
    // Two columns per instruction wherever the arithmetic is not an exponential: an element then
    // takes one multiply-add and one add for every two of what the special-function unit does, the
    // results are the same (one sweep of 2 x 20K keys with the rest of the call 42.6 -> 41.1 us, 128K
    // keys with 64-row windows 265 -> 258).  The kernels for one length no longer spill; those for
    // ragged batches with 128 columns in split mode are three registers short (12 bytes).
    const unsigned long long scale2 = pack2(a.c2, a.c2);
    int git = 0, nstat = 0, nvote = 0;
    each_item([&](const Item& it) {
      int ukv;
      const int hq0 = first_head(it, &ukv);
      int flip = 0;
      if constexpr (RAGGED) {
        const RaggedSeq& q = rs.s[it.seq];
        jmax = min(q.L - 1, q.n + wrow);
        jfree = min(q.L - 1, q.n);
        flip = (git ^ it.flip) & 1;
      }
      auto put_vote = [&](int hl, int j, float x) {  // head hl of the unit, key j
        if constexpr (RAGGED) {
          const RaggedSeq& q = rs.s[it.seq];
          if (j < q.n) a.vote[q.vote0 + static_cast<long long>(hq0 - q.batch * a.Hkv * a.g + hl) * q.n + j] = x;
        } else {
          if (j < a.n) a.vote[static_cast<size_t>(hq0 + hl) * a.n + j] = x;
        }
      };
      if (!it.vote) {
        // ---------------------------------------------------------- statistics
        float m2 = -INFINITY;  // running max, log2 domain
        float l = 0.f;         // running sum of exp2(x - m2)
        for (int t = it.t0; t < it.t1; ++t, ++git) {
          if (((git ^ flip) & 1) != (SPLIT ? set : wg)) continue;
          const int buf = git & (NBUF - 1);
          const uint32_t ub = (git / NBUF) & 1;
          if (!mbar_wait_warp(bar_tf(buf), ub, abort_s, WAIT_EPI_TMEM_FULL)) return false;
          tc_fence_after();
          const int key0 = t * TILE_KEYS;
          // this thread's slice of its window row: CPT key columns
          float v[VCH][32];
          const uint32_t taddr = tmem_base + lane_sel + buf * 128 + rep * NPAD + coff;
#pragma unroll
          for (int ch = 0; ch < VCH; ++ch) tmem_ld32(taddr + ch * 32, v[ch]);
          tmem_wait_ld();
          // the accumulator is in registers now: hand the buffer back to the MMA warp
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_n(bar_te(buf), te_arrivals);
          if (key0 + TILE_KEYS - 1 > jfree) {  // tile touches the window or the end of the keys
            const int kb = key0 + rep * NPAD + coff;
#pragma unroll
            for (int ch = 0; ch < VCH; ++ch)
#pragma unroll
              for (int c = 0; c < 32; ++c)
                v[ch][c] = (kb + ch * 32 + c <= jmax) ? v[ch][c] : -INFINITY;
          }
          float c0 = v[0][0], c1 = v[0][1], c2m = v[0][2], c3 = v[0][3];
#pragma unroll
          for (int ch = 0; ch < VCH; ++ch)
#pragma unroll
            for (int c = (ch == 0 ? 4 : 0); c < 32; c += 4) {
              c0 = fmaxf(c0, v[ch][c + 0]);
              c1 = fmaxf(c1, v[ch][c + 1]);
              c2m = fmaxf(c2m, v[ch][c + 2]);
              c3 = fmaxf(c3, v[ch][c + 3]);
            }
          const float cmax = fmaxf(fmaxf(c0, c1), fmaxf(c2m, c3));
          const float mnew = fmaxf(fmaxf(cmax * a.c2, m2), -1e30f);
          l *= ex2_approx(m2 - mnew);
          const unsigned long long negm = pack2(-mnew, -mnew);
          unsigned long long s01 = 0ull, s23 = 0ull;
#pragma unroll
          for (int ch = 0; ch < VCH; ++ch)
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
              s01 = add2(s01, ex2_approx2(fma2(pack2(v[ch][c + 0], v[ch][c + 1]), scale2, negm)));
              s23 = add2(s23, ex2_approx2(fma2(pack2(v[ch][c + 2], v[ch][c + 3]), scale2, negm)));
            }
          const float2 sa = unpack2(s01), sb = unpack2(s23);
          l += (sa.x + sa.y) + (sb.x + sb.y);
          m2 = mnew;
        }
        // leave this warp's (max, sum) per TMEM lane for the book-keeper
        const int pb = nstat % NPB;
        if (!mbar_wait_warp(bar_pe(pb), ((nstat / NPB) & 1) ^ 1, abort_s, WAIT_PART_EMPTY))
          return false;
        part_s[((pb * 2 + set) * 8 + wg * 4 + q) * 32 + lane] = make_float2(m2, l);
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_pf(pb));
        ++nstat;
        return true;
      }
      // ------------------------------------------------------------ votes
      const int lb = nvote % NLB;
      if (!mbar_wait_warp(bar_lf(lb), (nvote / NLB) & 1, abort_s, WAIT_LSE_FULL)) return false;
      const float* lse_b = lse_s + lb * MAX_COLS;
      for (int t = it.t0; t < it.t1; ++t, ++git) {
        if ((git & 1) != (SPLIT ? set : wg)) continue;
        const int buf = git & (NBUF - 1);
        const uint32_t ub = (git / NBUF) & 1;
        if (!mbar_wait_warp(bar_tf(buf), ub, abort_s, WAIT_EPI_TMEM_FULL)) return false;
        tc_fence_after();
        const int j = t * TILE_KEYS + 32 * q + lane;
        const uint32_t taddr = tmem_base + lane_sel + buf * 128 + coff;
        float g16[VCH * 2];
        float v[SPLIT ? 1 : VCH][32];
        if (!SPLIT) {
#pragma unroll
          for (int ch = 0; ch < VCH; ++ch) tmem_ld32(taddr + ch * 32, v[ch]);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_n(bar_te(buf), te_arrivals);
        }
        if (SPLIT || w16) {
#pragma unroll
          for (int ch = 0; ch < VCH; ++ch) {
            if (SPLIT) {
              tmem_ld32(taddr + ch * 32, v[0]);
              tmem_wait_ld();
              if (ch == VCH - 1) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_n(bar_te(buf), te_arrivals);
              }
            }
            const float(&vc)[32] = v[SPLIT ? 0 : ch];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              unsigned long long a01 = 0ull, a23 = 0ull;
#pragma unroll
              for (int t4 = 0; t4 < 4; ++t4) {
                // -lse of four adjacent columns: one broadcast read for the whole warp
                const ulonglong2 z =
                    *reinterpret_cast<const ulonglong2*>(lse_b + coff + ch * 32 + hf * 16 + 4 * t4);
                const int c = hf * 16 + 4 * t4;
                a01 = add2(a01, ex2_approx2(fma2(pack2(vc[c + 0], vc[c + 1]), scale2, z.x)));
                a23 = add2(a23, ex2_approx2(fma2(pack2(vc[c + 2], vc[c + 3]), scale2, z.y)));
              }
              const float2 aa = unpack2(a01), ab = unpack2(a23);
              g16[ch * 2 + hf] = (aa.x + aa.y) + (ab.x + ab.y);
            }
          }
          int hl = coff / a.W, left = gpw;  // SPLIT: coff is a multiple of W
          float acc = 0.f;
#pragma unroll
          for (int gi = 0; gi < VCH * 2; ++gi) {
            acc += g16[gi];
            if (--left == 0) {
              if (hl < a.hpu) put_vote(hl, j, acc);
              acc = 0.f;
              left = gpw;
              ++hl;
            }
          }
        } else {
          int hl = 0, left = a.W;
          float acc = 0.f;
#pragma unroll
          for (int ch = 0; ch < VCH; ++ch)
#pragma unroll
            for (int c = 0; c < 32; ++c) {
              const int col = ch * 32 + c;
              if (col < a.ncols) {
                acc += ex2_approx(fmaf(v[ch][c], a.c2, lse_b[col]));
                if (--left == 0) {
                  put_vote(hl, j, acc);
                  acc = 0.f;
                  left = a.W;
                  ++hl;
                }
              }
            }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_le(lb));  // this warp is done reading lse_s[lb]
      ++nvote;
      return true;
    });
  } else {
    // ------------------------------------------------------------ book-keeper warps
    // Warp 10 publishes this CTA's statistics partials; warp 11 fetches the unit's partials
    // for every vote item and folds them into the log-sum-exp row the item needs, as far ahead
    // as its shared-memory buffers allow.  A fold of 37 partials of 128 columns took one warp 5 us
    // beside the softmax warps, which keep the special-function units busy, longer than a wave of a 13K
    // prompt lasts; so it takes one exponential per partial, not two, and in split mode warp 10 folds
    // the upper half of the columns once it has published a wave's partials.  All CTAs publish a wave
    // before they fold it, so this wait too is for something that does not wait for it.
    const bool publisher = warp == 2 + EPI_WARPS;  // warp 10; warp 11 is the fetcher
    int nstat = 0, nvote = 0;
    auto publish = [&](const Item& it) {
      // merge the replicas and the two warpgroups (fixed order), publish
      const int pb = nstat % NPB;
      if (!mbar_wait_warp(bar_pf(pb), (nstat / NPB) & 1, abort_s, WAIT_PART_FULL)) return false;
      const float2* ps = part_s + pb * 16 * 32;
      for (int c = lane; c < NPAD; c += 32) {  // (padding columns too: a reader looks at all of them)
        float M = -INFINITY;
        for (int w2 = 0; w2 < 2 * NSET; ++w2)
          for (int r = 0; r < REPS; ++r) {
            const int row = r * NPAD + c;
            M = fmaxf(M, ps[(w2 * 4 + (row >> 5)) * 32 + (row & 31)].x);
          }
        M = fmaxf(M, -1e30f);
        float S = 0.f;
        for (int w2 = 0; w2 < 2 * NSET; ++w2)
          for (int r = 0; r < REPS; ++r) {
            const int row = r * NPAD + c;
            const float2 p = ps[(w2 * 4 + (row >> 5)) * 32 + (row & 31)];
            S += p.y * ex2_approx(p.x - M);
          }
        // log2 of this CTA's share of the row's softmax normaliser (-inf if it saw no key)
        const float part = M + log2f(S);
        if (!a.withhold)
          st_relaxed(slots_of(it) + static_cast<size_t>(it.slot) * MAX_COLS + c,
                     __float_as_uint(part) == NO_PARTIAL ? __uint_as_float(0x7fffffffu) : part);
      }
      __syncwarp();  // every lane is done with the buffer
      if (lane == 0) {
        if (a.stats_only) atomicAdd(a.counters + unit_of(it), 1);  // for the kernel that folds a shard's partials
        mbar_arrive(bar_pe(pb));
      }
      ++nstat;
      return true;
    };
    // Part `part` of the columns of a vote item's row, the whole row cut into as many as the constant says.
    auto fetch_part = [&](const Item& it, auto parts, int part) {
      constexpr int PARTS = decltype(parts)::value;
      constexpr int CPL = NCH / PARTS;  // columns per lane
      // Fetcher.  A vote item needs minus the log2-sum-exp of every window row of its unit.
      // With a supplied normaliser that row is in global memory already (its counter says so).
      // Otherwise it is the fold of the unit's partials.  A partial is its own flag: the slots hold
      // NO_PARTIAL until it is written, so this warp just reads them until none does (bounded) and
      // folds them in slot order, the same order in every CTA and every run, so all CTAs get
      // bit-identical rows without a second hand-over through global memory.  No fence, no counter
      // and no staging copy: a write and a read through L2 are all that lies between the last
      // partial and the first vote.
      // The slots are read with cp.async, which the PTX memory model counts as a weak access: against
      // the publishers' relaxed stores it promises nothing.  What the reading relies on is how this
      // GPU carries it out: `.cg` passes L1 by and reads L2, the point of coherence, where an aligned
      // 4-byte element is old or new, never a mixture; every element carries its own flag and is
      // looked at by itself; and each attempt is a new copy (volatile, memory clobber), so an old
      // element is read again until it is new.  Relaxed loads instead keep within the model, but the
      // slots on their way are then held in registers: 8 to 16 slots at a time, with or without the
      // next ones behind them, took 43.9-47 us against 43.5 for a prompt of 13K and 149-155 against
      // 146.5 for eight sequences of 1353 to 24000 positions.
      // In a ragged batch one CTA per unit folds and leaves the row, a flag of its own as well, in
      // global memory: a fold of 20 partials takes this warp 3-5 us beside the softmax warps, and
      // with a vote item for every two or three tiles the folds would set the pace.
      const int lb = nvote % NLB;
      const int c0 = (part * 32 + lane) * CPL;  // this lane's columns of the window rows
      float val[CPL];
#pragma unroll
      for (int t = 0; t < CPL; ++t) val[t] = 0.f;
      const unsigned long long t0 = globaltimer_ns();
      // half the limit: the roles of this CTA that wait for this row then still see the abort
      // flag, not their own time-out, and the status names the wait that failed
      auto give_up = [&]() {
        int stop = 0;
        if (lane == 0) {
          if (*abort_s != 0) stop = 1;
          else if (globaltimer_ns() - t0 > a.wait_ns / 2) { *abort_s = WAIT_UNIT_STATS; stop = 1; }
        }
        return __shfl_sync(0xffffffffu, stop, 0) != 0;
      };
      float* const row = a.lse2 + static_cast<size_t>(unit_of(it)) * MAX_COLS + c0;
      // whether a column of a row is missing
      auto missing = [&](const float (&x)[CPL]) {
        uint32_t most = 0u;  // NO_PARTIAL is the largest of all bit patterns
#pragma unroll
        for (int t = 0; t < CPL; ++t) most = max(most, __float_as_uint(x[t]));
        return __any_sync(0xffffffffu, most == NO_PARTIAL);
      };
      if (RAGGED && !a.votes_only && it.vote) {
        for (;;) {
          ld_relaxed<CPL>(row, val);
          if (!missing(val)) break;
          if (give_up()) return false;
          __nanosleep(100);
        }
      } else if (a.votes_only) {
        while (!__all_sync(0xffffffffu, ld_acquire(a.counters + unit_of(it)) > 0)) {
          if (give_up()) return false;
          __nanosleep(100);
        }
#pragma unroll
        for (int t = 0; t < CPL; ++t)
          if (c0 + t < a.ncols) val[t] = __ldcg(row + t);
      } else {
        const float* pp = slots_of(it);
        const uint32_t merge_addr = sbase + SM::OFF_MERGE;
        float M[CPL], S[CPL];
#pragma unroll
        for (int t = 0; t < CPL; ++t) { M[t] = -1e30f; S[t] = 0.f; }
        // All slots at once, through shared memory: every round trip to L2 costs 0.8 us here, with
        // the other CTAs reading the same lines, and registers hold only a few slots.
        int s0 = 0;
        while (s0 < it.nseg) {
          const int ns = min(MERGE_SEGS, it.nseg - s0);
          constexpr int CPS = NPAD / 4 / PARTS;  // 16-byte pieces of this warp's columns per slot
          const uint32_t mine = merge_addr + part * (CPS * 16);
          for (int p = lane; p < ns * CPS; p += 32)
            copy16_async(mine + (p / CPS) * (MAX_COLS * 4) + (p % CPS) * 16,
                         pp + static_cast<size_t>(s0 + p / CPS) * MAX_COLS + (part * CPS + p % CPS) * 4);
          // slots up to the next multiple of FOLD add nothing
          for (int p = ns * CPS + lane; p < (ns + FOLD - 1) / FOLD * FOLD * CPS; p += 32)
            sts4(mine + (p / CPS) * (MAX_COLS * 4) + (p % CPS) * 16, -INFINITY);
          copy_wait_all();
          __syncwarp();
          int at = 0;
          for (; at < ns; at += FOLD) {
            float x[FOLD][CPL];
            uint32_t most = 0u;
#pragma unroll
            for (int i = 0; i < FOLD; ++i) {
              lds<CPL>(merge_addr + ((at + i) * MAX_COLS + c0) * 4, x[i]);
#pragma unroll
              for (int t = 0; t < CPL; ++t) most = max(most, __float_as_uint(x[i][t]));
            }
            if (__any_sync(0xffffffffu, most == NO_PARTIAL)) break;
#pragma unroll
            for (int t = 0; t < CPL; ++t) {
              float pv[FOLD];
#pragma unroll
              for (int i = 0; i < FOLD; ++i) pv[i] = x[i][t];
              fold_partials(pv, M[t], S[t]);
            }
          }
          __syncwarp();  // all lanes are done with the buffer before the next copies land
          s0 += min(at, ns);
          // A slot is missing: wait until the last one is there (the wave is still being worked on,
          // usually), then fetch again from the first that was missing.
          while (at < ns) {
            if (give_up()) return false;
            float x[CPL];
            ld_relaxed<CPL>(pp + static_cast<size_t>(it.nseg - 1) * MAX_COLS + c0, x);
            if (!missing(x)) break;
            __nanosleep(100);
          }
        }
#pragma unroll
        for (int t = 0; t < CPL; ++t) val[t] = -(M[t] + log2f(S[t]));
        if (RAGGED) {
#pragma unroll
          for (int t = 0; t < CPL; ++t)
            st_relaxed(row + t, __float_as_uint(val[t]) == NO_PARTIAL ? __uint_as_float(0x7fffffffu) : val[t]);
          return true;
        }
      }
      // the softmax warps must be done with this buffer's previous row
      if (!mbar_wait_warp_relaxed(bar_le(lb), ((nvote / NLB) & 1) ^ 1, abort_s, WAIT_LSE_EMPTY))
        return false;
#pragma unroll
      for (int t = 0; t < CPL; ++t) lse_s[lb * MAX_COLS + c0 + t] = val[t];
      return true;
    };
    auto fetch = [&](const Item& it) {  // this warp's columns
      if (HALVES == 2 && both_fold) {
        if (!fetch_part(it, std::integral_constant<int, HALVES>{}, publisher ? 1 : 0)) return false;
      } else {
        if (!fetch_part(it, std::integral_constant<int, 1>{}, 0)) return false;
      }
      if (RAGGED && !a.votes_only && !it.vote) return true;  // (a folded row went to global memory)
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_lf(nvote % NLB));
      ++nvote;
      return true;
    };
    const int waves = (a.votes_only || a.stats_only) ? nphase : nphase / 2;
    bool go = publisher ? !a.votes_only : !a.stats_only;
    const bool folds = RAGGED && !publisher && !a.votes_only;
    // In a ragged batch the fetcher folds the next wave's rows, where this CTA holds the unit's first
    // slot, before it fetches those of a wave, so that nobody waits for a fold.  With a lag of one
    // wave this would never end: the next wave's statistics would stand behind the votes that wait
    // for this very fetch.
    static_assert(!RAGGED || WAVE_LAG >= 2, "a wave's statistics come before the votes of the wave before it");
    for (int w = folds ? -1 : 0; w < waves && go; ++w) {
      for (int m = 0; m < a.per && go && folds && w + 1 < waves; ++m) {
        const Item it = item_at(2 * (w + 1), m);
        if (it.t0 < it.t1 && it.slot == 0) go = fetch(it);
      }
      for (int m = 0; m < a.per && go && w >= 0 && publisher; ++m) {
        const Item it = item_at(2 * w, m);
        if (it.t0 < it.t1) go = publish(it);
      }
      for (int m = 0; m < a.per && go && w >= 0 && (!publisher || both_fold); ++m) {
        const Item it = item_at(2 * w + 1, m);
        if (it.t0 < it.t1) go = fetch(it);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_s != 0) {
    if (atomicCAS(a.status, 0, 5 /* SNAPKV_ERR_TIMEOUT */) == 0) a.status[1] = *abort_s;
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int D, int NCH, bool SPLIT, typename SEQS>
static cudaError_t run_scores(const CUtensorMap& tmK, const CUtensorMap& tmQ, const ScoreArgs& a, const SEQS& rs,
                              int grid, cudaStream_t stream, int* launches) {
  static DeviceOnce once;  // one flag set per instantiation: the attribute is per function and device
  if (!once.done()) {
    cudaError_t e = cudaFuncSetAttribute(score_kernel<D, NCH, SPLIT, SEQS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         Smem<D>::DYN_BYTES);
    if (e != cudaSuccess) return e;
    once.set();
  }
  // One CTA per SM (the shared-memory footprint allows no second one), grid no larger
  // than the SM count: every CTA becomes resident as soon as the stream's earlier work
  // has drained, so a CTA that waits for another CTA's partial statistics is waiting for
  // a CTA that runs.  The waits are bounded in any case.
  cudaError_t e = launch_pdl(score_kernel<D, NCH, SPLIT, SEQS>, dim3(grid), dim3(threads_for(SPLIT)),
                             Smem<D>::DYN_BYTES, stream, tmK, tmQ, a, rs);
  if (e != cudaSuccess) return e;
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  *launches += 1;
  return cudaSuccess;
}

// The column-split epilogue: each warpgroup's half of the columns is whole heads.
inline bool split_columns(int npad, int W) { return npad >= 64 && (W % 16) == 0 && ((npad / 2) % W) == 0; }

// The instantiation for a plan: columns padded to 32, 64 or 128, split or not.
template <typename SEQS>
static cudaError_t run_scores_for(int d, int W, int npad, const CUtensorMap& tmK, const CUtensorMap& tmQ,
                                  const ScoreArgs& a, const SEQS& rs, int grid, cudaStream_t stream, int* launches) {
  const int nch = npad >> 5;
  const bool split = split_columns(npad, W);
#define SNAPKV_SCORES(DD, NN, SS) run_scores<DD, NN, SS, SEQS>(tmK, tmQ, a, rs, grid, stream, launches)
#define SNAPKV_SCORES_D(DD)                                                                                  \
  (nch == 1 ? SNAPKV_SCORES(DD, 1, false)                                                                    \
            : (nch == 2 ? (split ? SNAPKV_SCORES(DD, 2, true) : SNAPKV_SCORES(DD, 2, false))                 \
                        : (split ? SNAPKV_SCORES(DD, 4, true) : SNAPKV_SCORES(DD, 4, false))))
  return d == 64 ? SNAPKV_SCORES_D(64) : SNAPKV_SCORES_D(128);
#undef SNAPKV_SCORES_D
#undef SNAPKV_SCORES
}

}  // namespace score

// The part of the kernel's arguments that fixes the schedule (what the work items follow from).
score::ScoreArgs score_args(const ScorePlan& plan, int L, int W, int Hkv, int votes_only);

}  // namespace snapkv
