// One generation step's attention over the compressed cache (Sec. 5.1.2: decoding on the
// compressed keys and values).  Per (batch, query head): out = softmax(q . K^T / sqrt(d)) V over
// the `rows` rows of the head's compressed cache.
//
// Bound by HBM: the cache is read once, whatever the number of query heads that share a cache
// head.  One thread-block CLUSTER per cache head, its CTAs taking contiguous shares of the rows:
//   * every warp streams its own row tiles (16 rows of d = 128, 32 of d = 64: 8 KB of K and V) by
//     TMA into a ring of stages of its own.  Loads run ahead without holding registers (128 KB and
//     more in flight per SM), and no barrier joins the warps: with plain loads each warp waited
//     for every step's data, at 4.85 TB/s;
//   * both products run on mma.sync with the cache as the 16-row operand: S = K.Q^T has 16 keys on
//     M and the group's query heads on N, O^T = V^T.P^T has 16 output dimensions on M and the heads
//     on N.  S takes bf16 operands as they are.  The fp32 probability is split into three bf16
//     terms whose sum is the fp32 value to its last bits; the eight columns of one instruction
//     hold the three terms of two heads, or two terms of four, or one of eight, so that 16 cache
//     rows of d = 128 take 16, 24 or 32 instructions for groups of up to 2, 4 and 8 heads (they
//     issue every five cycles per SM here; heads on M took 48).  On the fp32 pipes a group of four
//     costs 55 instructions a row;
//   * softmax is online, in the log2 domain, fp32;
//   * the partial results (maximum, sum, unnormalised output) of the CTAs are merged through
//     distributed shared memory, in rank order: no second kernel, no scratch, same bits every run.
//     Every CTA writes the slices it owes into its peers' memory before the one cluster barrier
//     and reads its own memory behind it (1.7 us less than barrier, remote reads, barrier).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "../../include/snapkv.h"
#include "launch.cuh"
#include "sm100_ptx.cuh"
#include "snapkv_internal.h"

namespace snapkv {
namespace {

constexpr int DEC_STAGE_BYTES = 8192;        // K and V of one row tile
constexpr int DEC_HEADS = 8;                 // query heads per CTA
constexpr int DEC_MAX_CLUSTER = 16;          // above 8: non-portable cluster size

// CTA shapes.  With one CTA per SM, eight warps with two stages each read fastest (268 MB in
// 42.7 us; 46.0 us with three stages, 47.7 us as two CTAs of four warps).  When there are more
// cache heads than SMs the CTAs come in rounds, and two smaller CTAs per SM hide one another's
// start and end (512 heads of 1024 rows: 44.4 us against 50.3 us).
struct DecWide { static constexpr int WARPS = 8, STAGES = 2, CTAS = 1; };
struct DecPair { static constexpr int WARPS = 4, STAGES = 3, CTAS = 2; };

constexpr int tile_rows(int D) { return DEC_STAGE_BYTES / (4 * D); }

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
__device__ __forceinline__ uint32_t peer_smem(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer_f(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Transpose of an 8x8 matrix of 16-bit elements spread over the warp as an mma fragment.
__device__ __forceinline__ uint32_t transpose8(uint32_t x) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
  return r;
}

// The first NT bf16 terms of x (each the rounding of what the terms before it leave), two
// elements at a time (packed pairs for an mma operand).
template <int NT>
__device__ __forceinline__ void split_bf16(float x, float y, uint32_t (&t)[NT]) {
#pragma unroll
  for (int i = 0; i < NT; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    t[i] = *reinterpret_cast<const uint32_t*>(&h);
    x -= __low2float(h);
    y -= __high2float(h);
  }
}

// Warp-wide wait for a copy of this warp's ring; false when the time limit has passed.
__device__ __forceinline__ bool wait_copy(uint32_t bar, uint32_t parity, unsigned long long limit_ns) {
  for (int i = 0; i < 256; ++i)
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if (__shfl_sync(0xffffffffu, globaltimer_ns() - t0 > limit_ns ? 1 : 0, 0)) return false;
  }
}

// Grid: (CTAs per cluster, B * Hc, groups of DEC_HEADS query heads).  NH: 2, 4 or 8, at least the
// query heads of a CTA; column n of an instruction belongs to head n % NH and, in the product
// with V, carries term n / NH of its probabilities (then, in further instructions, the terms
// 8 / NH later).
template <int D, int NH, typename SHAPE>
__global__ void __launch_bounds__(SHAPE::WARPS * 32, SHAPE::CTAS)
decode_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
              const __nv_bfloat16* __restrict__ q, int g, int rows, float c2, unsigned long long limit_ns,
              float* __restrict__ out, float* __restrict__ out_lse) {
  constexpr int DEC_WARPS = SHAPE::WARPS, DEC_STAGES = SHAPE::STAGES, DEC_THREADS = DEC_WARPS * 32;
  constexpr int ROWS = tile_rows(D);      // cache rows per stage
  constexpr int HALVES = D / 64;          // 64-element (128-byte) column blocks of a row
  constexpr int KS = D / 16;              // k-steps of S, and pairs of 8-column tiles of the output
  constexpr int BOX = ROWS * 128;         // bytes of one column block of a tile
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[DEC_WARPS][DEC_STAGES];
  __shared__ float w_m[DEC_WARPS][DEC_HEADS], w_l[DEC_WARPS][DEC_HEADS];
  // what the cluster's CTAs leave here: maximum and sum per head, and this CTA's output slice
  __shared__ float in_m[DEC_MAX_CLUSTER][DEC_HEADS], in_l[DEC_MAX_CLUSTER][DEC_HEADS];
  __shared__ float in_acc[DEC_HEADS * D + DEC_MAX_CLUSTER];
  pdl_launch_dependents();
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;   // mma fragment coordinates
  const int C = gridDim.x, rank = blockIdx.x, head = blockIdx.y;
  const int h0 = blockIdx.z * DEC_HEADS, gc = min(DEC_HEADS, g - h0);
  const uint32_t ring = smem_u32(smem) + warp * (DEC_STAGES * DEC_STAGE_BYTES);
  const uint32_t bar = smem_u32(&bars[warp][0]);

  // this CTA's tiles of the head, and this warp's: every DEC_WARPS-th of them
  const int T = (rows + ROWS - 1) / ROWS;
  const int t_begin = static_cast<int>(static_cast<long long>(rank) * T / C) + warp;
  const int t_end = static_cast<int>(static_cast<long long>(rank + 1) * T / C);
  auto issue = [&](int t, int s) {  // one lane: K and V of tile t into stage s
    const uint32_t dst = ring + s * DEC_STAGE_BYTES, b = bar + 8u * s;
    mbar_expect_tx(b, DEC_STAGE_BYTES);
#pragma unroll
    for (int h = 0; h < HALVES; ++h) {
      tma_load_3d(dst + h * BOX, &tmK, b, h * 64, t * ROWS, head);
      tma_load_3d(dst + (HALVES + h) * BOX, &tmV, b, h * 64, t * ROWS, head);
    }
  };
  if (C > 1) cluster_arrive();  // waited for before the first write into a peer's memory
  if (lane == 0) {
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
    for (int s = 0; s < DEC_STAGES; ++s) mbar_init(bar + 8u * s, 1);
    mbar_fence_init();
    fence_proxy_async();
  }
  __syncwarp();
  pdl_wait();  // everything above touched this CTA's shared memory only
  if (lane == 0)
    for (int s = 0; s < DEC_STAGES; ++s)
      if (t_begin + s * DEC_WARPS < t_end) issue(t_begin + s * DEC_WARPS, s);

  // Q as the B operand: column gid is head h0 + gid % NH (zero beyond gc)
  uint32_t qb[KS][2];
  {
    const int h = gid % NH;
    const __nv_bfloat16* qh = q + (static_cast<size_t>(head) * g + h0 + h) * D + 2 * tig;
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i)
        qb[k][i] = h < gc ? __ldg(reinterpret_cast<const uint32_t*>(qh + k * 16 + i * 8)) : 0u;
  }
  float acc[KS][4];  // dimensions 16 j + gid (+ 8) of columns 2 tig, 2 tig + 1
#pragma unroll
  for (int j = 0; j < KS; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
  constexpr int NT = (3 * NH + 7) / 8;          // instructions with V per 16 keys and dimensions
  const int term0 = (2 * tig) / NH;             // this lane's columns carry terms term0, term0 + 8 / NH, ...
  float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // of columns 2 tig + {0, 1}; l: this lane's keys
  bool failed = false;
  // ldmatrix: lane addresses a row of one of four 8x8 blocks, 16-byte chunks XORed with the row
  // as the 128-byte swizzle of the copies left them
  const int lrow_k = lane & 15, lchunk_k = lane >> 4;
  const int lrow_v = (lane & 7) + ((lane >> 4) << 3), lchunk_v = (lane >> 3) & 1;
  int n = 0;
  for (int t = t_begin; t < t_end; t += DEC_WARPS, ++n) {
    const int s = n % DEC_STAGES;
    if (!wait_copy(bar + 8u * s, (n / DEC_STAGES) & 1, limit_ns)) {
      failed = true;
      break;
    }
    const uint32_t kb = ring + s * DEC_STAGE_BYTES, vb = kb + HALVES * BOX;
#pragma unroll
    for (int sub = 0; sub < ROWS / 16; ++sub) {
      const int key0 = t * ROWS + sub * 16;
      const int rk = sub * 16 + lrow_k, rv = sub * 16 + lrow_v;
      float sc[2][4];  // two chains, even and odd k-steps
#pragma unroll
      for (int i = 0; i < 4; ++i) sc[0][i] = sc[1][i] = 0.f;
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t a[4];
        ldsm_x4(kb + (k >> 2) * BOX + rk * 128 + ((((k & 3) * 2 + lchunk_k) ^ (rk & 7)) << 4), a);
        mma_16816(sc[k & 1], a[0], a[1], a[2], a[3], qb[k][0], qb[k][1]);
      }
      float p[4];  // keys gid (0, 1) and gid + 8 (2, 3) of the lane's two columns
#pragma unroll
      for (int i = 0; i < 4; ++i)
        p[i] = key0 + gid + (i >> 1) * 8 < rows ? (sc[0][i] + sc[1][i]) * c2 : -INFINITY;
      float mx[2] = {fmaxf(p[0], p[2]), fmaxf(p[1], p[3])};
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        mx[0] = fmaxf(mx[0], __shfl_xor_sync(0xffffffffu, mx[0], o));
        mx[1] = fmaxf(mx[1], __shfl_xor_sync(0xffffffffu, mx[1], o));
      }
      if (__any_sync(0xffffffffu, mx[0] > m[0] || mx[1] > m[1])) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float mn = fmaxf(m[c], mx[c]);
          const float corr = m[c] == -INFINITY ? 0.f : exp2f(m[c] - mn);  // (nothing summed yet: 0)
          l[c] *= corr;
#pragma unroll
          for (int j = 0; j < KS; ++j) {
            acc[j][c] *= corr;
            acc[j][c + 2] *= corr;
          }
          m[c] = mn;
        }
      }
      // (a subtile past the head's last row, possible for 32-row tiles, has no key: p = 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = m[i & 1] == -INFINITY ? 0.f : exp2f(p[i] - m[i & 1]);
      l[0] += p[0] + p[2];
      l[1] += p[1] + p[3];
      uint32_t lo[3], hi[3];  // terms of keys gid and gid + 8
      split_bf16<3>(p[0], p[1], lo);
      split_bf16<3>(p[2], p[3], hi);
      uint32_t b[NT][2];      // P^T as the B operand: keys 2 tig, + 1 (and 8 further on) of column gid
#pragma unroll
      for (int i = 0; i < NT; ++i) {
        const int term = term0 + i * (8 / NH);
        b[i][0] = transpose8(term == 0 ? lo[0] : (term == 1 ? lo[1] : (term == 2 ? lo[2] : 0u)));
        b[i][1] = transpose8(term == 0 ? hi[0] : (term == 1 ? hi[1] : (term == 2 ? hi[2] : 0u)));
      }
#pragma unroll
      for (int j = 0; j < KS; ++j) {
        uint32_t a[4];
        ldsm_x4_trans(vb + (j >> 2) * BOX + rv * 128 + ((((j & 3) * 2 + lchunk_v) ^ (rv & 7)) << 4), a);
#pragma unroll
        for (int i = 0; i < NT; ++i) mma_16816(acc[j], a[0], a[1], a[2], a[3], b[i][0], b[i][1]);
      }
    }
    __syncwarp();  // every lane has read the stage
    if (lane == 0 && t + DEC_STAGES * DEC_WARPS < t_end) issue(t + DEC_STAGES * DEC_WARPS, s);
  }
  if (failed) {  // never leave with copies in flight; the outputs of this head become NaN
    for (int i = 1; i < DEC_STAGES; ++i)
      if (t_begin + (n + i) * DEC_WARPS < t_end)
        wait_copy(bar + 8u * ((n + i) % DEC_STAGES), ((n + i) / DEC_STAGES) & 1, limit_ns);
    l[0] = l[1] = NAN;
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    l[0] += __shfl_xor_sync(0xffffffffu, l[0], o);
    l[1] += __shfl_xor_sync(0xffffffffu, l[1], o);
  }
  // the columns of one head (its terms) are NH apart: NH / 2 lanes
#pragma unroll
  for (int o = NH / 2; o < 4; o <<= 1)
#pragma unroll
    for (int j = 0; j < KS; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[j][i] += __shfl_xor_sync(0xffffffffu, acc[j][i], o);

  // ---- merge the warps, then the CTAs of the cluster, both in order; the ring is idle by now
  __syncthreads();
  float* part = reinterpret_cast<float*>(smem);  // [warp][head][D]
  static_assert(DEC_HEADS * 128 * 4 <= DEC_STAGES * DEC_STAGE_BYTES, "a warp's partial fits its ring");
  if (tig < NH / 2) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int h = 2 * tig + c;
      if (gid == 0) {
        w_m[warp][h] = m[c];
        w_l[warp][h] = l[c];
      }
#pragma unroll
      for (int j = 0; j < KS; ++j) {
        part[(warp * DEC_HEADS + h) * D + 16 * j + gid] = acc[j][c];
        part[(warp * DEC_HEADS + h) * D + 16 * j + gid + 8] = acc[j][c + 2];
      }
    }
  }
  if (C > 1) cluster_wait();  // every CTA of the cluster runs: its memory may be written
  __syncthreads();
  const int per = (gc * D + C - 1) / C;  // outputs each CTA finishes; slices of in_acc, by source rank
  for (int e = threadIdx.x; e < gc * D; e += DEC_THREADS) {
    const int h = e / D;  // the same in all lanes (D is a multiple of 32): lane w weighs warp w's partial
    const float wm = w_m[lane % DEC_WARPS][h];
    float M = wm;
#pragma unroll
    for (int o = 1; o < DEC_WARPS; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float f = wm == -INFINITY ? 0.f : exp2f(wm - M);
    const float fl = f * w_l[lane % DEC_WARPS][h];
    float o = 0.f, L = 0.f;
#pragma unroll
    for (int w = 0; w < DEC_WARPS; ++w) {
      o += part[w * DEC_HEADS * D + e] * __shfl_sync(0xffffffffu, f, w);
      L += __shfl_sync(0xffffffffu, fl, w);
    }
    const int r = e / per, at = rank * per + (e - r * per);
    if (C > 1) st_peer_f(peer_smem(&in_acc[at], r), o);
    else in_acc[at] = o;
    if (e % D < 32 && lane < C) {  // one warp per head tells every CTA
      if (C > 1) {
        st_peer_f(peer_smem(&in_m[rank][h], lane), M);
        st_peer_f(peer_smem(&in_l[rank][h], lane), L);
      } else {
        in_m[0][h] = M;
        in_l[0][h] = L;
      }
    }
  }
  if (C > 1) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  for (int i = threadIdx.x; i < per; i += DEC_THREADS) {
    const int e = rank * per + i;
    if (e >= gc * D) break;
    const int h = e / D;
    float M = -INFINITY, o = 0.f, L = 0.f;
    for (int r = 0; r < C; ++r) M = fmaxf(M, in_m[r][h]);
    for (int r = 0; r < C; ++r) {
      const float f = in_m[r][h] == -INFINITY ? 0.f : exp2f(in_m[r][h] - M);
      o += in_acc[r * per + i] * f;
      L += in_l[r][h] * f;
    }
    const size_t bh = static_cast<size_t>(head) * g + h0 + h;
    out[bh * D + e % D] = o / L;
    if (out_lse && e % D == 0) out_lse[bh] = (M + log2f(L)) * 0.6931471805599453f;
  }
}

// CTAs per cache head: the cluster size with the smallest estimated time.  Clusters that find no
// place at once (`active`: clusters of a size that fit the GPU) come in rounds, each with a fixed
// part of about 3.5 us (start, first copies, merge).  Within a round a warp spends 0.35-0.8 us on a
// tile, more the more warps of its SM are at work; over all rounds the cache comes in at 6.8 TB/s
// at best.  (All measured; 24 heads of 2777 rows: 11.3 us with clusters of 4, 17.2 us with
// clusters of 6, of which 24 do not fit at once.)
int decode_cluster(long long heads, int tiles, int warps, int most, const int* active) {
  const double hbm_us = static_cast<double>(heads) * tiles * DEC_STAGE_BYTES / 6.8e6;
  int best = 1;
  double best_cost = 1e30;
  for (int c = 1; c <= most && (c == 1 || c <= tiles); ++c) {
    if (active[c] < 1) continue;
    const int per_cta = (tiles + c - 1) / c, per_warp = (per_cta + warps - 1) / warps;
    const double rounds = static_cast<double>((heads + active[c] - 1) / active[c]);
    const double tile_us = 0.35 + 0.06 * (per_cta < warps ? per_cta : warps);
    const double work = rounds * per_warp * tile_us;
    const double cost = (work > hbm_us ? work : hbm_us) + 3.5 * rounds;
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

template <int D, int NH, typename SHAPE>
cudaError_t launch_decode_shape(const void* q, const void* ck, const void* cv, int B, int Hq, int Hc, int rows,
                                float* out, float* out_lse, cudaStream_t stream) {
  constexpr int SMEM = SHAPE::WARPS * SHAPE::STAGES * DEC_STAGE_BYTES + 1024;  // slack for the ring's alignment
  auto kernel = decode_kernel<D, NH, SHAPE>;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(SHAPE::WARPS * 32);
  cfg.dynamicSmemBytes = SMEM;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  // how many clusters of each size the device holds at once, asked once per device
  constexpr int MAX_DEV = 16;
  static std::mutex mu;
  static int active[MAX_DEV][DEC_MAX_CLUSTER + 1];
  static std::atomic<bool> known[MAX_DEV];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= MAX_DEV) return cudaErrorInvalidDevice;
  if (!known[dev].load(std::memory_order_acquire)) {
    std::lock_guard<std::mutex> lock(mu);
    if (!known[dev].load(std::memory_order_relaxed)) {  // (another thread may have done it meanwhile)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
      active[dev][1] = SHAPE::CTAS * sm_count();
      for (int c = 2; c <= DEC_MAX_CLUSTER; ++c) {
        cfg.gridDim = dim3(c);
        attr[0].val.clusterDim.x = c;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&active[dev][c], kernel, &cfg) != cudaSuccess) {
          active[dev][c] = 0;
          (void)cudaGetLastError();  // a refusal here is an answer, not an error of the call
        }
      }
      known[dev].store(true, std::memory_order_release);
    }
  }
  CUtensorMap tmK, tmV;
  const unsigned long long dims[3] = {static_cast<unsigned long long>(D), static_cast<unsigned long long>(rows),
                                      static_cast<unsigned long long>(B) * Hc};
  const unsigned long long strides[2] = {D * 2ull, static_cast<unsigned long long>(rows) * D * 2ull};
  const unsigned box[3] = {64, static_cast<unsigned>(tile_rows(D)), 1};
  if (!encode_tensor_map(&tmK, ck, 3, dims, strides, box) || !encode_tensor_map(&tmV, cv, 3, dims, strides, box))
    return cudaErrorInvalidValue;
  const int g = Hq / Hc, chunks = (g + DEC_HEADS - 1) / DEC_HEADS;
  const int tiles = (rows + tile_rows(D) - 1) / tile_rows(D);
  const long long heads = static_cast<long long>(B) * Hc * chunks;
  const int C = decode_cluster(heads, tiles, SHAPE::WARPS, DEC_MAX_CLUSTER, active[dev]);
  const float c2 = static_cast<float>(1.4426950408889634 / sqrt(static_cast<double>(D)));
  cfg.gridDim = dim3(C, static_cast<unsigned>(B) * Hc, chunks);
  cfg.stream = stream;
  attr[0].val.clusterDim.x = C;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, tmK, tmV, static_cast<const __nv_bfloat16*>(q), g, rows, c2,
                            wait_limit_setting(), out, out_lse);
}

template <int D, int NH>
cudaError_t launch_decode_nh(const void* q, const void* ck, const void* cv, int B, int Hq, int Hc, int rows,
                             float* out, float* out_lse, cudaStream_t stream) {
  const long long heads = static_cast<long long>(B) * Hc * ((Hq / Hc + DEC_HEADS - 1) / DEC_HEADS);
  auto f = heads > sm_count() ? launch_decode_shape<D, NH, DecPair> : launch_decode_shape<D, NH, DecWide>;
  return f(q, ck, cv, B, Hq, Hc, rows, out, out_lse, stream);
}

template <int D>
cudaError_t launch_decode(const void* q, const void* ck, const void* cv, int B, int Hq, int Hc, int rows,
                          float* out, float* out_lse, cudaStream_t stream) {
  const int g = Hq / Hc;
  auto f = g <= 2 ? launch_decode_nh<D, 2> : (g <= 4 ? launch_decode_nh<D, 4> : launch_decode_nh<D, 8>);
  return f(q, ck, cv, B, Hq, Hc, rows, out, out_lse, stream);
}

}  // namespace
}  // namespace snapkv

// The step needs no scratch any more; the size and the check of the argument stay as part of the
// interface.
extern "C" size_t snapkv_decode_workspace_size(int B, int Hq, int rows, int d) {
  if (B < 1 || Hq < 1 || rows < 1 || (d != 64 && d != 128)) return 0;
  const size_t heads = static_cast<size_t>(B) * Hq;
  return (heads * (d + 2) * sizeof(float) + 255) / 256 * 256;
}

extern "C" snapkv_status_t snapkv_decode_attention(const void* q_cur, const void* cache_k,
                                                   const void* cache_v, int B, int Hq, int Hc,
                                                   int rows, int d, float* out, float* out_lse,
                                                   void* workspace, size_t workspace_bytes,
                                                   void* stream) {
  using namespace snapkv;
  if (B < 1 || Hq < 1 || Hc < 1 || rows < 1 || Hq % Hc != 0) return SNAPKV_ERR_INVALID_ARG;
  if (d != 64 && d != 128) return SNAPKV_ERR_UNSUPPORTED;
  if (!q_cur || !cache_k || !cache_v || !out) return SNAPKV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(q_cur) & 15) || (reinterpret_cast<uintptr_t>(cache_k) & 15) ||
      (reinterpret_cast<uintptr_t>(cache_v) & 15) || (reinterpret_cast<uintptr_t>(out) & 3) ||
      (reinterpret_cast<uintptr_t>(out_lse) & 3))
    return SNAPKV_ERR_INVALID_ARG;
  const long long heads = static_cast<long long>(B) * Hq;
  if (heads > 65535) return SNAPKV_ERR_UNSUPPORTED;
  const size_t need = static_cast<size_t>(heads) * (d + 2) * sizeof(float);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need)
    return SNAPKV_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const cudaError_t e = d == 128 ? launch_decode<128>(q_cur, cache_k, cache_v, B, Hq, Hc, rows, out, out_lse, s)
                                 : launch_decode<64>(q_cur, cache_k, cache_v, B, Hq, Hc, rows, out, out_lse, s);
  return e == cudaSuccess ? SNAPKV_OK : SNAPKV_ERR_CUDA;
}
