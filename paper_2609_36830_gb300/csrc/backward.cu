// Backward of the fused LM head and of the clipped surrogate (what the unchanged
// policy update needs after the log-probs: gradients with respect to the hidden
// states and the vocabulary matrix), without ever holding the logits of more
// than one chunk of rows.
//
// For the rows in the loss, in chunks of up to kChunkRows compacted rows:
//   1. gemm_kernel<EPI_G>:    z = H_c W^T recomputed on the tensor cores; the
//                             epilogue writes G = (g / tau) (onehot(y) - softmax(z / tau))
//                             in bf16, using the forward's log-sum-exp, in 64-column
//                             blocks: G[v / 64][row][v % 64], so that both later
//                             GEMMs read it in long contiguous runs (a K step of
//                             dH is one 16 KB run, a K step of dW 8 KB);
//   2. gemm_kernel<EPI_ROWS>: dH_c = G W (A = G K-major, B = W read MN-major),
//                             fp32 rows scattered back to their original row.  The
//                             tiles that would not fill a last round are split
//                             along K (tail_split) into partial tiles, which
//                             reduce_tail_kernel adds in a fixed order;
//   3. gemm_kernel<EPI_ACC>:  dW += G^T H_c (A = G and B = H_c, both read
//                             MN-major), fp32 accumulation in place; the first
//                             chunk stores, so dW needs no clearing.
// The GEMM is one warp-specialised tcgen05 kernel on CTA pairs: in each CTA
// warp 0 issues TMA for the CTA's own A tile and its own half of the B tile (one
// instruction of several lanes a stage)
// into a 4-stage ring (128-byte swizzle), both CTAs' bytes completing on the
// even CTA's barrier; warp 1 of the even CTA issues tcgen05.mma.cta_group::2
// (M 256 = 128 rows per CTA, N 256 = 128 columns from each CTA, K 16; the
// instruction descriptor's major bits select K- or MN-major operand layouts);
// warps 2-5 of each CTA drain its two TMEM accumulators.  Every CTA loads only
// its own tiles.  Every wait is bounded.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "pace_block.cuh"
#include "pace_internal.cuh"
#include "pace_loss.cuh"
#include "pace_rows.cuh"
#include "pace_tma.cuh"

namespace pace {
namespace {

constexpr int GBM = 128;
constexpr int GBN = 256;
constexpr int GBK = 64;
constexpr int GSTAGES = 4;
constexpr int kGemmThreads = 192;
constexpr uint32_t kGStageA = GBM * GBK * 2;  // 16 KB
constexpr uint32_t kGStageB = GBN / 2 * GBK * 2;  // 16 KB: this CTA's half of the B tile
constexpr uint32_t kGStageBytes = kGStageA + kGStageB;
constexpr uint32_t kGTmemCols = 2 * GBN;
// Two staging tiles of 32 rows x 128 bytes per epilogue warp, then the barriers.
constexpr uint32_t kGOutTile = 32 * 128;
constexpr uint32_t kGOutBytes = 4 * 2 * kGOutTile;
constexpr size_t kGSmemBytes = 1024 + GSTAGES * kGStageBytes + kGOutBytes + 256;
constexpr int64_t kChunkRows = 32768;         // rows of G held at once (bf16 M x V)
constexpr int kGroupM = 38;                   // M tiles per raster group
// The clusters meet (wait_round) about every kPaceSteps K steps, at a round
// boundary: meeting costs 1-2 us, the time of a few K steps, and the clusters drift
// slowly.  Whole calls meeting at every round / 512 / 4096 steps / never: 2,582 rows
// of the H 2048 head 3.31 / 3.22 / 3.18-3.30 / 3.18-3.23 ms, two 32k chunks of the
// H 1024 / V 50,001 head 14.92 / 14.76 / 14.68 / 14.65 ms, 21k rows of the H 3584 head
// 42.2 / 42.1 / 42.0 / 42.3 ms.
constexpr int kPaceSteps = 4096;
constexpr int kMaxKSplits = 8;                // parts a tail tile is split into at most
constexpr int kMaxGemmClusters = 76;          // clusters launched at most (bounds the partial tiles)

enum { EPI_G = 0, EPI_ROWS = 1, EPI_ACC = 2 };
enum { TRIM_NONE = 0, TRIM_M = 1, TRIM_K = 2 };

struct GemmArgs {
  int64_t M, N, K;
  int64_t m_tiles, n_tiles;
  int raster_n_fast;            // 1: N tile fastest; 0: groups of kGroupM M tiles, M fastest
  int trim;                     // TRIM_M / TRIM_K: that extent is cut, on the device, to the
                                // chunk's rows in the loss rounded up to GBM (TRIM_NONE: as given)
  // EPI_G
  int64_t chunk_row0;           // compact row of the chunk's first row
  const long long* n_valid;     // rows in the loss (device)
  const int32_t* rowidx;        // compact -> original row
  const int32_t* targets;
  const float* lse;             // forward log-sum-exp per original row
  const float* dlp;             // dLoss/dlp per original row
  float scale_log2;             // log2(e) / tau
  float inv_tau;
  int64_t g_cols;               // bf16 G in 64-column blocks [g_cols / 64][g_pitch][64]: V rounded
                                // up to 64 (columns >= V hold zeros)
  int64_t g_pitch;              // rows per 64-column block (tm_c stores 32-row boxes of it)
  // A operand from the blocked G (a_pitch > 0: rows per 64-column block); 0: plain matrix
  int64_t a_pitch;
  int32_t V;
  // EPI_ROWS
  float* rows_out;              // fp32 [orig rows][ldo]
  int64_t ldo;
  // partial tiles of the tail, or null: fp32 [part * items + item][2 GBM][GBN]
  float* part;
  // EPI_ACC
  float* acc_out;               // fp32 [M][ldo]
  int acc_first;                // 1: store (the first chunk), 0: add
  unsigned* round_ctr;          // pacing counter, zeroed before the launch (or null)
  int32_t* status;
};

// Work items are (pair of M tiles, N tile); the two CTAs of a cluster take the
// two M tiles of a pair and share every B tile through the 2-CTA MMA, each
// loading its own half of it.
__device__ __forceinline__ void item_of(const GemmArgs& p, int64_t m_tiles, int64_t item,
                                        int64_t* mp, int64_t* n) {
  const int64_t pairs = (m_tiles + 1) / 2;
  if (p.raster_n_fast) {
    *mp = item / p.n_tiles;
    *n = item % p.n_tiles;
    return;
  }
  const int64_t gp = kGroupM / 2;  // pairs per raster group
  const int64_t per_group = gp * p.n_tiles;
  const int64_t g = item / per_group;
  const int64_t r = item % per_group;
  const int64_t g0 = g * gp;
  const int64_t gm = (pairs - g0) < gp ? (pairs - g0) : gp;
  *mp = g0 + r % gm;
  *n = r / gm;
}

// The last, partial round of items items on n_clusters clusters: its tail items are
// split along K into `splits` parts each, so that together they fill the clusters
// for 1 / splits of a round instead of leaving most of them idle for a whole one
// (the dH of a micro-batch, 88 tiles on 76 clusters, took two rounds and takes
// 1 + 1/6).  Whole rounds are not split, so the partial tiles stay below kMaxKSplits
// a cluster.  splits = 1: no split pays (a full round, a short K).
struct TailSplit {
  int64_t full;  // items before the tail
  int tail;      // items of the tail
  int splits;
};

// Parts that a tile of nkb K steps may be split into: each has at least 32 of them.
__host__ __device__ inline int max_k_splits(int nkb) {
  return nkb / 32 < kMaxKSplits ? nkb / 32 : kMaxKSplits;
}

__host__ __device__ inline TailSplit tail_split(int64_t items, int n_clusters, int nkb) {
  TailSplit s;
  s.full = items / n_clusters * n_clusters;
  s.tail = static_cast<int>(items - s.full);
  s.splits = 1;
  int best = nkb;  // the tail's K steps
  const int most = max_k_splits(nkb);
  for (int k = 2; k <= kMaxKSplits; ++k) {  // (constant bounds: the divisions' latencies overlap)
    const int rounds = (s.tail * k + n_clusters - 1) / n_clusters;
    const int steps = rounds * ((nkb + k - 1) / k);
    if (k <= most && steps < best) {
      best = steps;
      s.splits = k;
    }
  }
  return s;
}

// 128-byte-swizzled operand tiles.  K-major: rows of 64 K elements (128 B),
// 8-row groups 1024 B apart; a 16-deep K step is +32 B.  MN-major: 64 MN
// elements per 128-byte row, one row per k; boxes of 64 (MN) x 64 (K) stacked
// along MN 8 KB apart (leading byte offset), 8-k groups 1024 B apart (stride
// byte offset); a 16-deep K step is +2048 B.
__device__ __forceinline__ uint64_t operand_desc(uint32_t saddr, bool mn_major) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(mn_major ? (8192u >> 4) : 1u) << 16;
  d |= static_cast<uint64_t>(1024u >> 4) << 32;
  d |= static_cast<uint64_t>(1u) << 46;
  d |= static_cast<uint64_t>(2u) << 61;
  return d;
}

// M = 256: the pair's two 128-row tiles.
__host__ __device__ constexpr uint32_t idesc_bf16(bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) |
         ((b_mn ? 1u : 0u) << 16) | ((static_cast<uint32_t>(GBN) >> 3) << 17) |
         ((static_cast<uint32_t>(2 * GBM) >> 4) << 24);
}

// Two floats as bf16 (round to nearest even), the first in the low half.
__device__ __forceinline__ uint32_t bf16x2_rn(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

template <bool A_MN, bool B_MN, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                const __grid_constant__ CUtensorMap tm_c, GemmArgs p) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + GSTAGES * kGStageBytes + kGOutBytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + GSTAGES;
  uint64_t* tmem_full = bars + 2 * GSTAGES;
  uint64_t* tmem_empty = tmem_full + 2;
  uint64_t* mma_done = tmem_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t crank = cluster_ctarank();
  const bool leader = crank == 0;
  // The host sizes a chunk by its row capacity; the rows of it that are in the
  // loss are known only on the device (the compaction's count).  Tiles past
  // them hold zero rows: M (G, dH) or K (dW) is cut to the count rounded up to
  // GBM, the same value in every CTA, so every early exit below is uniform.
  int64_t M = p.M, K = p.K, m_tiles = p.m_tiles;
  if (p.trim != TRIM_NONE) {
    int64_t v = static_cast<int64_t>(*p.n_valid) - p.chunk_row0;
    const int64_t cap = p.trim == TRIM_M ? p.M : p.K;
    v = v < 0 ? 0 : (v > cap ? cap : v);
    v = (v + GBM - 1) / GBM * GBM;
    if (v > cap) v = cap;
    if (p.trim == TRIM_M) {
      M = v;
      m_tiles = (v + GBM - 1) / GBM;
    } else {
      K = v;
    }
  }
  const int64_t base_items = (m_tiles + 1) / 2 * p.n_tiles;
  const int64_t cid = blockIdx.x / 2, n_clusters = gridDim.x / 2;
  const int nkb_all = static_cast<int>((K + GBK - 1) / GBK);
  // uniform over the grid, and before the pair's collective TMEM allocation
  if (nkb_all == 0 || base_items == 0) {
    if (EPI == EPI_ACC && p.acc_first)  // no rows in the loss: dW = 0
      for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
           i < p.M * p.N / 4; i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        reinterpret_cast<float4*>(p.acc_out)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    return;
  }
  TailSplit ts{base_items, 0, 1};
  if (EPI == EPI_ROWS && p.part)
    ts = tail_split(base_items, static_cast<int>(n_clusters), nkb_all);
  const int64_t n_items = ts.splits > 1 ? ts.full + static_cast<int64_t>(ts.tail) * ts.splits
                                        : base_items;
  // item t's tile and K steps [k0, k1); a tail item's part (-1: the whole K)
  auto work_of = [&](int64_t t, int* k0, int* k1, int* part) -> int64_t {
    *k0 = 0;
    *k1 = nkb_all;
    *part = -1;
    if (EPI != EPI_ROWS || ts.splits == 1 || t < ts.full) return t;
    const int u = static_cast<int>(t - ts.full);
    *part = u / ts.tail;
    *k0 = nkb_all * *part / ts.splits;
    *k1 = nkb_all * (*part + 1) / ts.splits;
    return ts.full + u % ts.tail;
  };
  const int pace_rounds = max(1, kPaceSteps / nkb_all);

  if (threadIdx.x == 0) {
    for (int s = 0; s < GSTAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tmem_full[b], 1);
      mbar_init(&tmem_empty[b], 2 * 4);  // one arrival per epilogue warp of the pair
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  cluster_sync();  // both CTAs run and their barriers exist
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, kGTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();  // both CTAs' tensor memory is allocated before any MMA writes it
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  constexpr uint32_t kIdesc = idesc_bf16(A_MN, B_MN);
  const uint32_t peer_abort = cluster_addr(const_cast<int*>(abort_flag), crank ^ 1u);
  auto give_up = [&]() {
    if (!*abort_flag) report(p.status, PACE_ERR_TIMEOUT);
    *abort_flag = 1;
    st_cluster_u32(peer_abort, 1u);
  };

  if (warp == 0) {
    // The whole warp produces: a stage's boxes (one or two 64-wide ones per operand) are
    // one TMA instruction of lanes 0..n-1.  Issued one after the other by one lane, whole
    // calls took 3.03 against 2.96 ms (2,582 rows, H 2048 head) and 1.63 against 1.61
    // (8,248 rows, H 1024 / V 50,001); 21k rows of H 3584 the same (power-capped).
    if (lane == 0) {
      tma_prefetch_desc(&tm_a);
      tma_prefetch_desc(&tm_b);
    }
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    constexpr int kBoxesA = A_MN ? 2 : 1, kBoxes = kBoxesA + (B_MN ? 2 : 1);
    const bool is_a = lane < kBoxesA;
    const int half = is_a ? lane : lane - kBoxesA;  // which 64-wide box of an MN-major tile
    const void* desc = is_a ? static_cast<const void*>(&tm_a) : static_cast<const void*>(&tm_b);
    const uint32_t dst = (is_a ? 0u : kGStageA) + half * 8192u;
    uint32_t it = 0;
    bool ok = true;
    unsigned round = 0;  // this cluster's items so far
    for (int64_t t = cid; t < n_items && ok; t += n_clusters, ++round) {
      int64_t mp, nt;
      int kb0, kb1, part;
      item_of(p, m_tiles, work_of(t, &kb0, &kb1, &part), &mp, &nt);
      const int32_t m0 = static_cast<int32_t>((2 * mp + crank) * GBM);
      // this CTA's half of B: columns nh .. nh + 127
      const int32_t nh = static_cast<int32_t>(nt * GBN) + static_cast<int32_t>(crank) * (GBN / 2);
      // this lane's box: at K step kb it starts at (x + kb * dx, y + kb * dy)
      int32_t x, y, dx, dy;
      if (is_a && p.a_pitch > 0) {  // G in 64-wide blocks: the block is the inner dimension
        const int32_t ap = static_cast<int32_t>(p.a_pitch);
        x = 0;
        dx = 0;
        y = A_MN ? (m0 / 64 + half) * ap : m0;  // M = vocabulary: block, K rows; else K = vocabulary
        dy = A_MN ? GBK : ap;
      } else if (is_a ? A_MN : B_MN) {  // {64 MN, 64 K}
        x = (is_a ? m0 : nh) + 64 * half;
        dx = 0;
        y = 0;
        dy = GBK;
      } else {  // {64 K, 128 rows}
        x = 0;
        dx = GBK;
        y = is_a ? m0 : nh;
        dy = 0;
      }
      // the clusters start this round together (every round but the last is full)
      if (leader && lane == 0 && round > 0 && round % pace_rounds == 0 && p.round_ctr)
        wait_round(p.round_ctr, round * static_cast<unsigned>(n_clusters));
      __syncwarp();
      for (int kb = kb0; kb < kb1; ++kb, ++it) {
        const uint32_t s = it % GSTAGES, ph = (it / GSTAGES) & 1u;
        // one outcome for the warp
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&empty[s], ph ^ 1u, abort_flag))) {
          ok = false;
          break;
        }
        const uint32_t bar = cluster_addr(&full[s], 0);
        if (leader && lane == 0) mbar_arrive_expect_tx(&full[s], 2 * kGStageBytes);
        __syncwarp();  // the lanes' loads are one TMA instruction
        if (lane < kBoxes)
          tma_load_2d_pair(smem + s * kGStageBytes + dst, desc, bar, x + kb * dx, y + kb * dy, pol);
      }
      if (leader && lane == 0 && ok && p.round_ctr) atomicAdd(p.round_ctr, 1u);
    }
    if (lane == 0) {
      if (!ok) give_up();
      // every copy issued has landed before the CTA exits: the even CTA sees
      // both CTAs' bytes on its full barriers, the odd CTA its stages consumed
      const uint64_t lim = *abort_flag ? 1000000ull : kWaitLimitNs;
      for (uint32_t s = 0; s < GSTAGES && s < it; ++s) {
        const uint32_t last = it - 1 - ((it - 1 - s) % GSTAGES);
        if (leader)
          mbar_wait_bounded(&full[s], (last / GSTAGES) & 1u, nullptr, lim);
        else
          mbar_wait_bounded(&empty[s], (last / GSTAGES) & 1u, nullptr, lim);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      uint32_t it = 0, tc = 0;
      bool ok = true;
      for (int64_t t = cid; t < n_items && ok; t += n_clusters, ++tc) {
        int kb0, kb1, part;
        work_of(t, &kb0, &kb1, &part);
        const uint32_t acc = tc & 1u, acc_ph = (tc >> 1) & 1u;
        if (!mbar_wait_bounded_cluster(&tmem_empty[acc], acc_ph ^ 1u, abort_flag)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * GBN;
        for (int kb = kb0; kb < kb1; ++kb, ++it) {
          const uint32_t s = it % GSTAGES, ph = (it / GSTAGES) & 1u;
          if (!mbar_wait_bounded(&full[s], ph, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + s * kGStageBytes);
          const uint32_t sb = sa + kGStageA;
#pragma unroll
          for (int k = 0; k < GBK / 16; ++k) {
            const uint32_t ka = A_MN ? sa + k * 2048 : sa + k * 32;
            const uint32_t kbb = B_MN ? sb + k * 2048 : sb + k * 32;
            tc_mma_f16_pair(d_tmem, operand_desc(ka, A_MN), operand_desc(kbb, B_MN), kIdesc,
                            (kb > kb0 || k > 0) ? 1u : 0u);
          }
          tc_commit_pair(cluster_addr(&empty[s], 0));
          tc_commit_pair(cluster_addr(&empty[s], 1));
        }
        if (!ok) break;
        tc_commit_pair(cluster_addr(&tmem_full[acc], 0));
        tc_commit_pair(cluster_addr(&tmem_full[acc], 1));
      }
      if (!ok) give_up();
      tc_commit_pair(cluster_addr(mma_done, 0));
      mbar_wait_bounded(mma_done, 0, nullptr);
    }
  } else {
    const int quad = warp & 3;
    const int r_local = quad * 32 + lane;
    const uint32_t empty0 = cluster_addr(&tmem_empty[0], 0);
    const uint32_t empty1 = cluster_addr(&tmem_empty[1], 0);
    // Output tiles leave through shared memory: a lane writes its row's 128 bytes (in
    // the 128-byte swizzle, so the warp's 16-byte stores are conflict-free) and lane 0
    // hands the 32 x 128-byte tile to the TMA, two tiles in turn.  Whole 128-byte lines
    // go out, asynchronously, where a lane storing its own row piece by piece spread
    // every store over 32 lines: whole calls of 607 rows (H 2048 head) 1.24 -> 1.01 ms,
    // 2,582 rows 3.17 -> 3.03, two 32k chunks of H 1024 / V 50,001 12.5 -> 11.8, 21k
    // rows of H 3584 41.4 -> 40.8.
    unsigned char* out = smem + GSTAGES * kGStageBytes + (warp - 2) * 2 * kGOutTile;
    uint32_t n_out = 0;  // tiles handed out so far
    auto out_begin = [&]() -> unsigned char* {  // the next tile, once its last copy was read
      if (lane == 0) bulk_wait_read<1>();
      __syncwarp();
      return out + (n_out & 1u) * kGOutTile + lane * 128;
    };
    auto out_chunk = [&](unsigned char* row, int q, uint4 v) {  // 16-byte chunk q of the row
      *reinterpret_cast<uint4*>(row + ((q ^ (lane & 7)) << 4)) = v;
    };
    auto out_end = [&](int32_t x, int32_t y) {
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store_2d(&tm_c, out + (n_out & 1u) * kGOutTile, x, y);
        bulk_commit();
      }
      ++n_out;
    };
    uint32_t tc = 0;
    for (int64_t t = cid; t < n_items; t += n_clusters, ++tc) {
      int64_t mp, nt;
      int kb0, kb1, part;
      item_of(p, m_tiles, work_of(t, &kb0, &kb1, &part), &mp, &nt);
      const int64_t mt = 2 * mp + crank;
      const uint32_t acc = tc & 1u, acc_ph = (tc >> 1) & 1u;
      // one outcome for the whole warp (tcgen05.ld below is warp-collective)
      const bool got = __all_sync(0xffffffffu,
                                  mbar_wait_bounded(&tmem_full[acc], acc_ph, abort_flag));
      if (!got) {
        give_up();
        break;
      }
      tc_fence_after();
      const int64_t row = mt * GBM + r_local;  // row of C
      const int64_t n0 = nt * GBN;
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + acc * GBN;
      unsigned char* orow = nullptr;
      const int64_t row_w = mt * GBM + quad * 32;  // the warp's first row
      // per-row context
      bool row_ok = row < M;
      int32_t y = -1;
      float gscale = 0.0f, lse2 = 0.0f;
      int64_t orig = -1;
      if (EPI == EPI_G || EPI == EPI_ROWS) {
        const int64_t crow = p.chunk_row0 + row;
        const bool in_loss = row_ok && crow < static_cast<int64_t>(*p.n_valid);
        if (in_loss) orig = p.rowidx[crow];
        if (EPI == EPI_G && in_loss) {
          y = p.targets[orig];
          gscale = p.dlp[orig] * p.inv_tau;
          lse2 = p.lse[orig] * 1.4426950408889634f;
        }
        if (EPI == EPI_ROWS) row_ok = in_loss;
      }
#pragma unroll 1
      for (int c = 0; c < GBN; c += 32) {
        float v[32];
        tmem_ld_32x32b_x32(tbase + c, v);
        tmem_wait_ld();
        const int64_t col0 = n0 + c;
        if (EPI == EPI_G) {
          if (row_w < M && col0 < p.g_cols) {  // M is a multiple of 32: all its rows
            // G = (g / tau) (onehot - p), zero for rows outside the loss.  This epilogue
            // bounds the G GEMM at small H (a 256-column tile takes 5 us of MMAs at H
            // 1024), so per-column tests stay out of it: with them and rounding in
            // integer arithmetic, a chunk of 32k rows (H 1024, V 50,001) took 3.88 ms,
            // now 2.40; 8,248 rows 1.01 -> 0.62 ms; 2,582 rows of H 2048 1.08 -> 1.02.
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = ex2_approx(fmaf(v[i], p.scale_log2, -lse2));
            const uint32_t off = static_cast<uint32_t>(y - col0);
            if (off < 32u) {  // the target: 1 - p, kept as -(1 - p) for the product below
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (off == static_cast<uint32_t>(i)) v[i] = -(1.0f - v[i]);
            }
            if (col0 + 32 > p.V) {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (col0 + i >= p.V) v[i] = 0.0f;
            }
            uint32_t packed[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const uint32_t g = bf16x2_rn(-gscale * v[2 * i], -gscale * v[2 * i + 1]);
              packed[i] = gscale != 0.0f ? g : 0u;
            }
            // two chunks of 32 columns make one 64-column block's 128-byte rows
            if ((c & 32) == 0) orow = out_begin();
#pragma unroll
            for (int q = 0; q < 4; ++q)
              out_chunk(orow, (c & 32 ? 4 : 0) + q,
                        make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2],
                                   packed[4 * q + 3]));
            if (c & 32)
              out_end(0, static_cast<int32_t>((col0 >> 6) * p.g_pitch + row_w));
          }
        } else if (EPI == EPI_ROWS) {
          if (part >= 0) {  // a partial tile, whole (its rows outside the loss are not read)
            float4* d4 = reinterpret_cast<float4*>(
                p.part + ((t - ts.full) * (2 * GBM) + crank * GBM + r_local) * GBN + c);
#pragma unroll
            for (int q = 0; q < 8; ++q)
              d4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          } else if (row_ok) {
            float* dst = p.rows_out + orig * p.ldo + col0;
            if (col0 + 32 <= p.N) {
              float4* d4 = reinterpret_cast<float4*>(dst);
#pragma unroll
              for (int q = 0; q < 8; ++q)
                d4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            } else {
              for (int i = 0; i < 32 && col0 + i < p.N; ++i) dst[i] = v[i];
            }
          }
        } else {
          // N is a multiple of 64, so a chunk of 32 columns is inside or outside; rows
          // past M are clipped by the tensor map
          if (p.acc_first) {
            if (row_w < M && col0 < p.N) {
              orow = out_begin();
#pragma unroll
              for (int q = 0; q < 8; ++q)
                out_chunk(orow, q,
                          make_uint4(__float_as_uint(v[4 * q]), __float_as_uint(v[4 * q + 1]),
                                     __float_as_uint(v[4 * q + 2]), __float_as_uint(v[4 * q + 3])));
              out_end(static_cast<int32_t>(col0), static_cast<int32_t>(row_w));
            }
          } else if (row_ok && col0 < p.N) {  // (a TMA reduction would flush subnormals)
            float4* d4 = reinterpret_cast<float4*>(p.acc_out + row * p.ldo + col0);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              float4 o = d4[q];
              o.x += v[4 * q];
              o.y += v[4 * q + 1];
              o.z += v[4 * q + 2];
              o.w += v[4 * q + 3];
              d4[q] = o;
            }
          }
        }
      }
      // one arrival per warp on the even CTA's barrier, after every lane's loads
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc ? empty1 : empty0);
    }
    if (lane == 0) bulk_wait_all();  // the copies are done before the CTA's memory goes
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA frees its tensor memory or leaves while the pair's MMAs, copies
  // or arrivals may still reach it
  cluster_sync();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem_base, kGTmemCols);
  cluster_sync();  // the collective release is complete in both CTAs
}

// Adds the partial tiles of the tail of a dH GEMM (the same geometry as the GEMM's,
// from the same device-side count), part 0 first, and writes their rows in the loss:
// a warp per row of 256 columns.
__global__ void __launch_bounds__(256)
    reduce_tail_kernel(GemmArgs p, int n_clusters) {
  int64_t v = static_cast<int64_t>(*p.n_valid) - p.chunk_row0;
  v = v < 0 ? 0 : (v > p.M ? p.M : v);
  const int64_t m_tiles = (v + GBM - 1) / GBM;
  const int nkb = static_cast<int>((p.K + GBK - 1) / GBK);
  const TailSplit ts = tail_split((m_tiles + 1) / 2 * p.n_tiles, n_clusters, nkb);
  if (ts.splits == 1) return;
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < ts.tail * 2 * GBM; u += warps) {
    const int i = u / (2 * GBM), r = u % (2 * GBM);
    int64_t mp, nt;
    item_of(p, m_tiles, ts.full + i, &mp, &nt);
    const int64_t row = mp * (2 * GBM) + r;
    if (row >= v) continue;
    float* dst = p.rows_out + static_cast<int64_t>(p.rowidx[p.chunk_row0 + row]) * p.ldo;
    const int64_t n0 = nt * GBN;
    for (int c = lane * 4; c < GBN && n0 + c < p.N; c += 128) {  // N is a multiple of 64
      float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      for (int s = 0; s < ts.splits; ++s) {
        const float4 x = __ldcg(reinterpret_cast<const float4*>(
            p.part + ((static_cast<int64_t>(s) * ts.tail + i) * (2 * GBM) + r) * GBN + c));
        a.x += x.x;
        a.y += x.y;
        a.z += x.z;
        a.w += x.w;
      }
      *reinterpret_cast<float4*>(dst + n0 + c) = a;
    }
  }
}

// Zero the gathered rows from n_valid up to the next multiple of GBM (at most
// rows_end) of the compact buffer: dW reads whole GBM-row tiles of them, and the
// rows outside the loss must contribute exactly 0 (0 x garbage could be NaN).
__global__ void zero_tail_rows_kernel(uint4* __restrict__ buf, int64_t row_vecs,
                                      const long long* __restrict__ n_valid, int64_t rows_end) {
  const int64_t start = *n_valid;
  int64_t end = (start + GBM - 1) / GBM * GBM;
  if (end > rows_end) end = rows_end;
  const int64_t total = (end - start) * row_vecs;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    buf[start * row_vecs + i] = make_uint4(0, 0, 0, 0);
}

// dLoss/dlp per row of the clipped surrogate (oracle: oracle_surrogate_grad), 0
// outside the loss.  The scale (1 / rows in the loss, or 1 / (sequences x rows of
// the sequence)) is an fp64 quotient and a row's product with it is taken in fp64 and
// rounded to fp32 (quick_product does without where it can).
struct GradArgs {
  const int64_t* seq_offsets;
  const uint8_t* seq_accepted;
  const uint8_t* mask;
  const float* logprob;
  const float* behav;
  const float* adv;
  int64_t n_seq, n_rows;
  RowGeom geom;
  bool vec;
  float eps_low, eps_high, dual;
  const long long* block_in;  // TOKEN_MEAN: rows in the loss per block of the count
  const unsigned long long* seq_in;  // SEQ_MEAN: rows in the loss per sequence,
  const int* n_used;                 // sequences that have any
  float* dlp;
};

// x * scale rounded to fp64 and then to fp32, without the fp64 pipe, which a conversion,
// a product and a conversion back per row would keep busy for most of the kernel (derivative
// of 5.4M rows by graph replay 42.6 us that way, 23.0 so).  scale = s_hi + s_lo to 2^-49, and
// q + t is x * scale to 2^-45.  Where t moved by 2^-18 of itself both ways rounds to the same
// float, so does the product (after Ziv, ACM TOMS 17, 1991: |t| is at least 2^-26 |q| where
// q + t is near the middle of two floats); otherwise `sure` is false and the result is to be
// computed.  The partial products must not be subnormal: see products_fit.
__device__ __forceinline__ float quick_product(float x, float s_hi, float s_lo, bool* sure) {
  const float q = __fmul_rn(x, s_hi);
  const float t = __fmaf_rn(x, s_lo, __fmaf_rn(x, s_hi, -q));
  const float r = __fmaf_rn(t, 1.0f - 0x1p-18f, q);
  *sure = r == __fmaf_rn(t, 1.0f + 0x1p-18f, q);
  return r;
}

// A row's derivative is 0 or at least |a| e^-20 in magnitude, so its product with the scale is
// 0 or above 2^-90, which keeps every bit of the partial products in the normal range.
__device__ __forceinline__ bool products_fit(float a, float s_hi) {
  return (a == 0.0f || fabsf(a) >= 0x1p-20f) && s_hi >= 0x1p-40f;
}

// A sequence's advantage and, under SEQ_MEAN, its rows' scale.
struct AdvScale {
  float a;
  double scale;
};
struct AdvScaleOf {
  using Value = AdvScale;
  const float* adv;
  const unsigned long long* seq_in;
  double n_used;
  __device__ Value operator()(int64_t i) const {
    return {adv[i], 1.0 / (n_used * static_cast<double>(seq_in[i]))};
  }
};

// dl/dlp of a row.
__device__ __forceinline__ float term_derivative(const GradArgs& p, float lp, float bh, float a) {
  const float d = lp - bh;
  const float dc = fminf(fmaxf(d, -20.0f), 20.0f);
  const float rho = expf(dc);
  const float rc = fminf(fmaxf(rho, 1.0f - p.eps_low), 1.0f + p.eps_high);
  const float p1 = -a * rho, p2 = -a * rc;
  const float lm = fmaxf(p1, p2);
  float x = 0.0f;
  if (d > -20.0f && d < 20.0f && p1 >= p2) x = -a * rho;
  if (a < 0.0f && -p.dual * a < lm) x = 0.0f;
  return x;
}

__device__ __forceinline__ float scale_hi(double scale) { return static_cast<float>(scale); }
__device__ __forceinline__ float scale_lo(double scale) {
  return static_cast<float>(scale - static_cast<double>(scale_hi(scale)));
}

// TOKEN_MEAN: a tile's derivatives are computed at once, whatever its sequences.
__global__ void __launch_bounds__(kRowThreads, kRowMinBlocks) surrogate_grad_kernel(GradArgs p) {
  const int wid = threadIdx.x >> 5;
  const int64_t w0 = (static_cast<int64_t>(blockIdx.x) * kRowWarps + wid) * p.geom.per_warp;
  const int64_t w1 = w0 + p.geom.per_warp < p.geom.n_tiles ? w0 + p.geom.per_warp : p.geom.n_tiles;
  int64_t t0 = w0 * kRowTile;
  RowLoads cur, nxt;
  // the first rows' loads are in flight while the counts are added up
  if (w0 < w1) cur.load(p.logprob, p.behav, p.mask, t0, tile_end(t0, p.n_rows), p.vec);
  __shared__ double s_scale;
  long long mine = 0, total = 0;
  for (int i = threadIdx.x; i < p.geom.blocks; i += kRowThreads) mine += p.block_in[i];
  block_exclusive_scan<long long>(mine, &total);
  __shared__ float s_part[2];
  if (threadIdx.x == 0) {
    s_scale = 1.0 / static_cast<double>(total);
    s_part[0] = scale_hi(s_scale);
    s_part[1] = scale_lo(s_scale);
  }
  __syncthreads();
  const float s_hi = s_part[0], s_lo = s_part[1];
  if (w0 >= w1) return;
  PieceWalker<FloatOf> pw(p.seq_offsets, p.seq_accepted, FloatOf{p.adv}, p.n_seq, t0);
  for (int64_t w = w0; w < w1; ++w) {
    const int64_t t1 = tile_end(t0, p.n_rows);
    if (w + 1 < w1) nxt.load(p.logprob, p.behav, p.mask, t1, tile_end(t1, p.n_rows), p.vec);
    unsigned in = 0u, unsure = 0u;
    float adv[kRowsPerLane] = {};
    pw.walk(t0, t1, [&](int64_t, int64_t lo, int64_t hi, float a, int64_t) {
      const unsigned rows = piece_bits(t0, lo, hi) & cur.mask;
      in |= rows;
      if (!products_fit(a, s_hi)) unsure |= rows;
#pragma unroll
      for (int u = 0; u < kRowsPerLane; ++u) adv[u] = rows >> u & 1u ? a : adv[u];
    });
    if (__any_sync(0xffffffffu, in != 0u)) {
#pragma unroll
      for (int u = 0; u < kRowsPerLane; ++u) {
        const float x = term_derivative(p, cur.lp[u], cur.bh[u], adv[u]);
        bool sure;
        cur.lp[u] = quick_product(x, s_hi, s_lo, &sure);  // the derivative, once the row is used
        cur.bh[u] = x;
        if (!sure) unsure |= 1u << u;
      }
      unsure &= in;
      if (__any_sync(0xffffffffu, unsure != 0u)) {  // the vote keeps it a branch
#pragma unroll
        for (int u = 0; u < kRowsPerLane; ++u)
          if (unsure >> u & 1u)
            cur.lp[u] = static_cast<float>(static_cast<double>(cur.bh[u]) * s_scale);
      }
    }
    store_rows(p.dlp, t0, t1, p.vec, in, cur.lp);
    cur = nxt;
    t0 = t1;
  }
}

// SEQ_MEAN: a tile's pieces, with their advantages and the scales that lanes of the walker
// have divided for, go through shared memory; a lane then finds the piece of each of its
// rows.  (All lanes on every piece in turn, each with its own division, and the count's
// atomics one by one took 1 to 2 us a piece: 5,000 rows of 1,000 sequences 95 us a call,
// now 17; 300 rows of 8 19.1 and 12.5, 5.4M rows of 1,024 37.3 and 37.5.)
struct PieceScales {
  double scale[kRowTile];
  float a[kRowTile];
  uint16_t begin[kRowTile], end[kRowTile];  // rows in the tile
};

__global__ void __launch_bounds__(kRowThreads, kRowMinBlocks)
    surrogate_grad_seq_kernel(GradArgs p) {
  __shared__ PieceScales lists[kRowWarps];
  const int wid = threadIdx.x >> 5;
  PieceScales& list = lists[wid];
  const int64_t w0 = (static_cast<int64_t>(blockIdx.x) * kRowWarps + wid) * p.geom.per_warp;
  const int64_t w1 = w0 + p.geom.per_warp < p.geom.n_tiles ? w0 + p.geom.per_warp : p.geom.n_tiles;
  if (w0 >= w1) return;
  int64_t t0 = w0 * kRowTile;
  RowLoads cur, nxt;
  cur.load(p.logprob, p.behav, p.mask, t0, tile_end(t0, p.n_rows), p.vec);
  PieceWalker<AdvScaleOf> pw(p.seq_offsets, p.seq_accepted,
                             AdvScaleOf{p.adv, p.seq_in, static_cast<double>(*p.n_used)},
                             p.n_seq, t0);
  const int r0 = row_in_tile(0);
  for (int64_t w = w0; w < w1; ++w) {
    const int64_t t1 = tile_end(t0, p.n_rows);
    if (w + 1 < w1) nxt.load(p.logprob, p.behav, p.mask, t1, tile_end(t1, p.n_rows), p.vec);
    int n = pw.collect(t0, t1, [&](int i, int64_t, int64_t lo, int64_t hi, AdvScale v, int64_t) {
      if (i >= kRowTile) return;  // (overlapping offsets may make more pieces)
      list.scale[i] = v.scale;
      list.a[i] = v.a;
      list.begin[i] = static_cast<uint16_t>(lo - t0);
      list.end[i] = static_cast<uint16_t>(hi - t0);
    });
    n = n < kRowTile ? n : kRowTile;
    __syncwarp();
    int k = 0;  // the first piece that ends past the lane's first row
    for (int above = n; k < above;) {
      const int m = (k + above) >> 1;
      if (list.end[m] <= r0) k = m + 1;
      else above = m;
    }
    const int k0 = k;
    int begin = kRowTile, end = kRowTile;
    float a = 0.0f, s_hi = 0.0f, s_lo = 0.0f;
    bool fit = true;
    auto fetch = [&]() {
      const bool any = k < n;
      begin = any ? list.begin[k] : kRowTile;
      end = any ? list.end[k] : kRowTile;
      a = any ? list.a[k] : 0.0f;
      const double sc = any ? list.scale[k] : 0.0;
      s_hi = scale_hi(sc);
      s_lo = scale_lo(sc);
      fit = !any || products_fit(a, s_hi);
    };
    fetch();
    unsigned in = 0u, unsure = 0u;
#pragma unroll
    for (int u = 0; u < kRowsPerLane; ++u) {
      while (r0 + u >= end) {  // (past the last piece, end is past the tile)
        ++k;
        fetch();
      }
      if (r0 + u >= begin) in |= 1u << u;
      const float x = term_derivative(p, cur.lp[u], cur.bh[u], a);
      bool sure;
      cur.lp[u] = quick_product(x, s_hi, s_lo, &sure);
      cur.bh[u] = x;
      if (!sure || !fit) unsure |= 1u << u;
    }
    in &= cur.mask;
    unsure &= in;
    if (__any_sync(0xffffffffu, unsure != 0u)) {  // the vote keeps it a branch
      k = k0;
#pragma unroll
      for (int u = 0; u < kRowsPerLane; ++u) {
        if (!(unsure >> u & 1u)) continue;
        while (r0 + u >= list.end[k]) ++k;
        cur.lp[u] = static_cast<float>(static_cast<double>(cur.bh[u]) * list.scale[k]);
      }
    }
    store_rows(p.dlp, t0, t1, p.vec, in, cur.lp);
    __syncwarp();  // the list is rewritten
    cur = nxt;
    t0 = t1;
  }
}

// ---------------------------------------------------------------- host side

int gemm_clusters() {
  const int n = sm_count() / 2;
  return n < kMaxGemmClusters ? (n > 0 ? n : 1) : kMaxGemmClusters;
}

template <bool A_MN, bool B_MN, int EPI>
pace_status launch_gemm(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tc,
                        GemmArgs a, unsigned* round_ctr, cudaStream_t st) {
  constexpr int kMaxDevices = 64;
  static bool done[kMaxDevices] = {};  // shared-memory opt-in made on that device
  static std::mutex mu;
  int dev = 0;
  PACE_TRY_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return PACE_ERR_CUDA;
  {
    std::lock_guard<std::mutex> g(mu);
    if (!done[dev]) {
      PACE_TRY_CUDA(cudaFuncSetAttribute(gemm_kernel<A_MN, B_MN, EPI>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kGSmemBytes)));
      done[dev] = true;
    }
  }
  a.m_tiles = (a.M + GBM - 1) / GBM;
  a.n_tiles = (a.N + GBN - 1) / GBN;
  const int64_t items = (a.m_tiles + 1) / 2 * a.n_tiles;
  if (items == 0) return PACE_OK;
  // with partial tiles every cluster is launched: a short tail is spread over all
  const int64_t max_clusters = gemm_clusters();
  const int64_t grid = 2 * (items < max_clusters && !a.part ? items : max_clusters);
  PACE_TRY_CUDA(cudaMemsetAsync(round_ctr, 0, sizeof(unsigned), st));
  a.round_ctr = round_ctr;
  gemm_kernel<A_MN, B_MN, EPI><<<static_cast<unsigned>(grid), kGemmThreads, kGSmemBytes, st>>>(
      ta, tb, tc, a);
  PACE_TRY(last_launch_status());
  if (EPI == EPI_ROWS && a.part) {
    reduce_tail_kernel<<<static_cast<unsigned>(sm_count() * 4), 256, 0, st>>>(
        a, static_cast<int>(max_clusters));
    return last_launch_status();
  }
  return PACE_OK;
}

struct BwWs {
  LmWs lm;            // compaction + gathered rows (hidden_c)
  uint16_t* g;        // bf16 G of one chunk, 64-column blocks [ceil(V / 64)][chunk][64]
  unsigned* round_ctr;  // the GEMMs' pacing counter
  float* part;          // dH's partial tiles
};

int64_t chunk_rows(int64_t n_rows) {
  int64_t c = n_rows < kChunkRows ? n_rows : kChunkRows;
  return (c + GBM - 1) / GBM * GBM;
}

void carve_bw_ws(Carver& cv, int64_t n_rows, int64_t n_seq, int H, int V, BwWs* w) {
  carve_lm_ws(cv, n_rows, n_seq, H, true, &w->lm);
  const int64_t g_cols = (static_cast<int64_t>(V) + 63) / 64 * 64;
  w->g = cv.take<uint16_t>(static_cast<size_t>(chunk_rows(n_rows > 0 ? n_rows : 1)) * g_cols);
  w->round_ctr = cv.take<unsigned>(1);
  // a tail of R < kMaxGemmClusters tiles, and no more tiles than the rows have, in as many
  // parts as the vocabulary's K steps allow (none below 64 K steps: no tile is split then)
  const int64_t tiles = (chunk_rows(n_rows > 0 ? n_rows : 1) + 2 * GBM - 1) / (2 * GBM) *
                        ((H + GBN - 1) / GBN);
  const int64_t tail = tiles < kMaxGemmClusters ? tiles : kMaxGemmClusters - 1;
  const int parts = max_k_splits(static_cast<int>((V + GBK - 1) / GBK));
  w->part = parts > 1 ? cv.take<float>(static_cast<size_t>(tail) * parts * 2 * GBM * GBN) : nullptr;
}

}  // namespace
}  // namespace pace

using namespace pace;

namespace pace {
namespace {

struct SurBwWs {
  RowCounts counts;
  unsigned long long* seq_in;
  int* n_used;
  float* adv;
};

SurBwWs carve_sur_bw_ws(Carver& cv, int64_t n_rows, int64_t n_seq) {
  SurBwWs w;
  w.counts = carve_row_counts(cv, n_rows);
  w.seq_in = cv.take<unsigned long long>(n_seq > 0 ? n_seq : 1);
  w.n_used = cv.take<int>(1);
  w.adv = cv.take<float>(n_seq > 0 ? n_seq : 1);
  return w;
}

}  // namespace
}  // namespace pace

extern "C" size_t pace_surrogate_backward_workspace_size(int64_t n_rows, int64_t n_seq) {
  if (n_rows < 0 || n_seq < 0) return 0;
  Carver cv;
  carve_sur_bw_ws(cv, n_rows, n_seq);
  return cv.used;
}

extern "C" pace_status pace_surrogate_backward(const PaceBatch* batch, const float* logprob,
                                               const PaceLossArgs* loss, float* dlp,
                                               void* workspace, size_t workspace_bytes,
                                               int32_t* status_dev, void* stream) {
  PACE_TRY(check_batch(batch));
  PACE_TRY(check_loss_args(batch, loss));
  if (batch->n_rows > 0 && (!logprob || !dlp)) return PACE_ERR_INVALID_ARG;
  if (!workspace || !aligned(workspace, 256)) return PACE_ERR_WORKSPACE;
  Carver cv(workspace, workspace_bytes);
  const SurBwWs ws = carve_sur_bw_ws(cv, batch->n_rows, batch->n_seq);
  if (!cv.fits()) return PACE_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  if (batch->n_seq == 0) {
    if (batch->n_rows > 0)
      PACE_TRY_CUDA(cudaMemsetAsync(dlp, 0, static_cast<size_t>(batch->n_rows) * 4, st));
    return PACE_OK;
  }
  float* adv = loss->adv ? loss->adv : ws.adv;
  const AdvJob job =
      adv_job(loss->reward, batch->seq_accepted, batch->n_seq, loss->group_size,
              loss->params.adv_eps, loss->params.std_unbiased, adv);
  if (batch->n_rows == 0) return launch_group_adv(job, batch, nullptr, status_dev, st);
  const bool seq_mean = loss->params.agg != PACE_AGG_TOKEN_MEAN;
  if (seq_mean) {
    PACE_TRY_CUDA(cudaMemsetAsync(ws.seq_in, 0,
                                  static_cast<size_t>(batch->n_seq) * sizeof(*ws.seq_in), st));
    PACE_TRY_CUDA(cudaMemsetAsync(ws.n_used, 0, sizeof(int), st));
  }
  // rows in the loss (per block, per sequence) and the advantages, then the rows
  PACE_TRY(launch_count_rows(batch, ws.counts, seq_mean ? ws.seq_in : nullptr, ws.n_used, job,
                             nullptr, nullptr, status_dev, st));
  GradArgs a;
  a.seq_offsets = batch->seq_offsets;
  a.seq_accepted = batch->seq_accepted;
  a.mask = batch->mask;
  a.logprob = logprob;
  a.behav = loss->behav_lp;
  a.adv = adv;
  a.n_seq = batch->n_seq;
  a.n_rows = batch->n_rows;
  a.geom = row_geom(batch->n_rows);
  a.vec = rows_vec(logprob, loss->behav_lp, dlp, batch->mask);
  a.eps_low = loss->params.eps_low;
  a.eps_high = loss->params.eps_high;
  a.dual = loss->params.dual_clip;
  a.block_in = ws.counts.block;
  a.seq_in = ws.seq_in;
  a.n_used = ws.n_used;
  a.dlp = dlp;
  if (seq_mean)
    surrogate_grad_seq_kernel<<<static_cast<unsigned>(a.geom.blocks), kRowThreads, 0, st>>>(a);
  else
    surrogate_grad_kernel<<<static_cast<unsigned>(a.geom.blocks), kRowThreads, 0, st>>>(a);
  return last_launch_status();
}

extern "C" size_t pace_token_logprob_backward_workspace_size(int64_t n_rows, int64_t n_seq,
                                                             int32_t hidden_size,
                                                             int32_t vocab_size) {
  if (n_rows < 0 || n_seq < 0 || hidden_size <= 0 || vocab_size <= 0) return 0;
  Carver cv;
  BwWs w;
  carve_bw_ws(cv, n_rows, n_seq, hidden_size, vocab_size, &w);
  return cv.used;
}

extern "C" pace_status pace_token_logprob_backward(
    const PaceBatch* batch, const void* hidden, const void* w_vocab, const int32_t* targets,
    int32_t hidden_size, int32_t vocab_size, float temperature, const float* lse,
    const float* dlp, float* grad_hidden, float* grad_w, void* workspace,
    size_t workspace_bytes, int32_t* status_dev, void* stream) {
  const int H = hidden_size, V = vocab_size;
  PACE_TRY(check_lm_args(batch, hidden, w_vocab, targets, H, V, temperature, dlp));
  if (batch->n_rows > 0 && (!lse || !grad_hidden || !grad_w)) return PACE_ERR_INVALID_ARG;
  if (!aligned(grad_hidden, 16) || !aligned(grad_w, 16)) return PACE_ERR_UNSUPPORTED_SHAPE;
  if (!workspace || !aligned(workspace, 256)) return PACE_ERR_WORKSPACE;
  Carver cv(workspace, workspace_bytes);
  BwWs ws;
  carve_bw_ws(cv, batch->n_rows, batch->n_seq, H, V, &ws);
  if (!cv.fits()) return PACE_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  const int64_t n_rows = batch->n_rows;
  if (n_rows == 0) {
    PACE_TRY_CUDA(cudaMemsetAsync(grad_w, 0, static_cast<size_t>(V) * H * 4, st));
    return PACE_OK;
  }
  PACE_TRY_CUDA(cudaMemsetAsync(grad_hidden, 0, static_cast<size_t>(n_rows) * H * 4, st));
  // the rows in the loss, gathered densely (always compacted here)
  PACE_TRY(run_compaction(batch, ws.lm.cw, AdvJob{}, nullptr, nullptr, nullptr, nullptr, status_dev, st));
  PACE_TRY(run_gather(hidden, H, n_rows, ws.lm.cw, ws.lm.hidden_c, st));
  const int64_t rows_cap = n_rows > 128 ? n_rows : 128;
  const int64_t row_vecs = static_cast<int64_t>(H) * 2 / 16;
  zero_tail_rows_kernel<<<static_cast<unsigned>(sm_count() * 4), 256, 0, st>>>(
      static_cast<uint4*>(ws.lm.hidden_c), row_vecs, ws.lm.cw.total, rows_cap);
  PACE_TRY(last_launch_status());
  const int64_t chunk = chunk_rows(n_rows);
  const int64_t g_cols = (static_cast<int64_t>(V) + 63) / 64 * 64;
  const int64_t g_blocks = g_cols / 64;
  // TMA row coordinates of the blocked G are 32-bit
  if (g_blocks * chunk > static_cast<int64_t>(INT32_MAX)) return PACE_ERR_UNSUPPORTED_SHAPE;
  for (int64_t c0 = 0; c0 < n_rows; c0 += chunk) {
    const int64_t rows_c = (n_rows - c0) < chunk ? (n_rows - c0) : chunk;
    const int64_t rows_c_pad = (rows_c + GBM - 1) / GBM * GBM;
    const void* hc = static_cast<const uint16_t*>(ws.lm.hidden_c) + c0 * H;
    // rows of the gathered buffer from c0 on (the padded tail of a chunk past the
    // buffer is read as zeros by TMA)
    const int64_t hc_rows = (rows_cap - c0) < rows_c_pad ? (rows_cap - c0) : rows_c_pad;
    // 1. G = (g / tau) (onehot - softmax) for the chunk's rows (bf16)
    {
      CUtensorMap ta, tb, tc;
      PACE_TRY(encode_bf16_2d(&ta, hc, hc_rows, H, H, 64, GBM));
      PACE_TRY(encode_bf16_2d(&tc, ws.g, g_blocks * rows_c_pad, 64, 64, 64, 32));
      PACE_TRY(encode_bf16_2d(&tb, w_vocab, V, H, H, 64, GBN / 2));
      GemmArgs a = {};
      a.M = rows_c_pad;
      a.N = V;
      a.K = H;
      a.raster_n_fast = 0;
      a.trim = TRIM_M;
      a.chunk_row0 = c0;
      a.n_valid = ws.lm.cw.total;
      a.rowidx = ws.lm.cw.rowidx;
      a.targets = targets;
      a.lse = lse;
      a.dlp = dlp;
      a.scale_log2 = 1.4426950408889634f / temperature;
      a.inv_tau = 1.0f / temperature;
      a.g_cols = g_cols;
      a.g_pitch = rows_c_pad;
      a.V = V;
      a.status = status_dev;
      PACE_TRY((launch_gemm<false, false, EPI_G>(ta, tb, tc, a, ws.round_ctr, st)));
    }
    // 2. dH rows = G W   (W read MN-major: [K = V][N = H])
    {
      CUtensorMap ta, tb;
      PACE_TRY(encode_bf16_2d(&ta, ws.g, g_blocks * rows_c_pad, 64, 64, 64, GBM));
      PACE_TRY(encode_bf16_2d(&tb, w_vocab, V, H, H, 64, 64));
      GemmArgs a = {};
      a.M = rows_c_pad;
      a.N = H;
      a.K = V;
      a.a_pitch = rows_c_pad;
      a.raster_n_fast = 1;
      a.trim = TRIM_M;
      a.chunk_row0 = c0;
      a.n_valid = ws.lm.cw.total;
      a.rowidx = ws.lm.cw.rowidx;
      a.rows_out = grad_hidden;
      a.ldo = H;
      a.part = ws.part;
      a.status = status_dev;
      PACE_TRY((launch_gemm<false, true, EPI_ROWS>(ta, tb, ta, a, ws.round_ctr, st)));
    }
    // 3. dW += G^T H_c   (G read MN-major: [K = rows][M = V]; H_c MN-major: [K = rows][N = H])
    {
      CUtensorMap ta, tb, tc;
      PACE_TRY(encode_bf16_2d(&ta, ws.g, g_blocks * rows_c_pad, 64, 64, 64, 64));
      PACE_TRY(encode_f32_2d(&tc, grad_w, V, H, H, 32, 32));
      PACE_TRY(encode_bf16_2d(&tb, hc, hc_rows, H, H, 64, 64));
      GemmArgs a = {};
      a.M = V;
      a.N = H;
      a.K = rows_c_pad;
      a.a_pitch = rows_c_pad;
      a.raster_n_fast = 1;
      a.trim = TRIM_K;
      a.chunk_row0 = c0;
      a.n_valid = ws.lm.cw.total;
      a.acc_out = grad_w;
      a.acc_first = c0 == 0 ? 1 : 0;
      a.ldo = H;
      a.status = status_dev;
      PACE_TRY((launch_gemm<true, true, EPI_ACC>(ta, tb, tc, a, ws.round_ctr, st)));
    }
  }
  return PACE_OK;
}
