// GRPO advantages, the asymmetric dual-clipped token-mean surrogate, and the
// row compaction that feeds the fused LM head (shared training settings of
// the paper's appendix: GRPO with within-group standardisation, clip widths
// 0.20 / 0.28, dual-clip coefficient 10, token-mean aggregation; tool output
// kept in context but masked from the loss).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "pace_block.cuh"
#include "pace_internal.cuh"
#include "pace_loss.cuh"
#include "pace_rows.cuh"

namespace pace {

// ------------------------------------------------------------ advantages

// L = 2^m >= G lanes per group (32 / L groups a warp),
// lane k holding member k.  Mean and standard deviation of the accepted members'
// rewards in fp64, summed from the lowest index up (the same order as one thread
// would take), then A_i = (R_i - mean) / (std + eps), each lane its own division:
// with a thread per group, its chain of 2 G loads and G divisions took 8-11 us.
__device__ void group_adv_lanes(const float* __restrict__ reward,
                                const uint8_t* __restrict__ accepted, int64_t n_groups, int G,
                                int L, double eps, int unbiased, float* __restrict__ adv,
                                int64_t warp) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int k = lane & (L - 1);
  const int64_t g = warp * (32 / L) + lane / L;
  const bool mine = g < n_groups && k < G;
  const int64_t i = g * G + k;
  const bool in = mine && (accepted ? accepted[i] != 0 : true);
  const float rf = mine ? reward[i] : 0.0f;
  const double r = static_cast<double>(rf);
  const unsigned bal = __ballot_sync(full, in);
  const int first = lane & ~(L - 1);
  const unsigned members = bal >> first & (L == 32 ? full : (1u << L) - 1u);
  const int n = __popc(members);
  double sum = 0.0;
  for (int m = 0; m < G; ++m) {
    const double x = __shfl_sync(full, r, first + m);
    if (members >> m & 1u) sum = __dadd_rn(sum, x);
  }
  const double mean = n > 0 ? __ddiv_rn(sum, static_cast<double>(n)) : 0.0;
  const double d = __dsub_rn(r, mean);
  const double dd = __dmul_rn(d, d);
  double ss = 0.0;
  for (int m = 0; m < G; ++m) {
    const double x = __shfl_sync(full, dd, first + m);
    if (members >> m & 1u) ss = __dadd_rn(ss, x);
  }
  const int div = unbiased ? n - 1 : n;
  const double sd = div > 0 ? __dsqrt_rn(__ddiv_rn(ss, static_cast<double>(div))) : 0.0;
  const double den = __dadd_rn(sd, eps);
  if (mine) adv[i] = static_cast<float>(in && d != 0.0 ? __ddiv_rn(d, den) : 0.0);
}

// A thread per group, in the same order.
__device__ void group_adv_thread(const float* __restrict__ reward,
                                 const uint8_t* __restrict__ accepted, int64_t g, int G, double eps,
                                 int unbiased, float* __restrict__ adv) {
  const int64_t i0 = g * G;
  int64_t n = 0;
  double sum = 0.0;
  for (int k = 0; k < G; ++k) {
    if (accepted && !accepted[i0 + k]) continue;
    sum = __dadd_rn(sum, static_cast<double>(reward[i0 + k]));
    ++n;
  }
  const double mean = n > 0 ? __ddiv_rn(sum, static_cast<double>(n)) : 0.0;
  double ss = 0.0;
  for (int k = 0; k < G; ++k) {
    if (accepted && !accepted[i0 + k]) continue;
    const double d = __dsub_rn(static_cast<double>(reward[i0 + k]), mean);
    ss = __dadd_rn(ss, __dmul_rn(d, d));
  }
  const int64_t div = unbiased ? n - 1 : n;
  const double sd = div > 0 ? __dsqrt_rn(__ddiv_rn(ss, static_cast<double>(div))) : 0.0;
  const double den = __dadd_rn(sd, eps);
  for (int k = 0; k < G; ++k) {
    double a = 0.0;
    if (!accepted || accepted[i0 + k]) {
      const double d = __dsub_rn(static_cast<double>(reward[i0 + k]), mean);
      a = d == 0.0 ? 0.0 : __ddiv_rn(d, den);
    }
    adv[i0 + k] = static_cast<float>(a);
  }
}

// Lanes or threads: the lanes of a group share its chain of loads and divisions, but each
// repeats its sums and root, about G times the fp64 work, so they win while the groups are
// few enough for latency to count.  pace_group_advantages, a thread and lanes per group:
// G 2, 16,000 sequences 4.5 and 3.7 us, 32,000 4.5 and 4.8; G 8, 32,000 8.2 and 5.7,
// 64,000 8.3 and 9.1, 1M 44 and 105; G 16, 64,000 14.1 and 11.4, 128,000 14.0 and 20.3;
// G 32, 1M 47 and 198.  (One member has no work to repeat: lanes at any size.)
constexpr int64_t kLaneGroups = 6144, kLanes = 65536;

constexpr int kAdvThreads = 32;  // a warp: the groups' fp64 divisions spread over the SMs

AdvJob adv_job(const float* reward, const uint8_t* accepted, int64_t n_seq, int G, float eps,
               int unbiased, float* adv) {
  AdvJob j{};
  j.reward = reward;
  j.accepted = accepted;
  j.n_groups = n_seq / G;
  j.G = G;
  j.L = 1;
  while (j.L < G && j.L < 32) j.L *= 2;
  if (G > 32 || (G > 1 && (j.n_groups > kLaneGroups || j.n_groups * j.L > kLanes))) j.L = 0;
  j.eps = static_cast<double>(eps);
  j.unbiased = unbiased;
  j.adv = adv;
  return j;
}

// Blocks of `threads` threads that compute the advantages: with lanes, one warp each
// (their other threads have no part in it); with a thread per group, up to 128 threads.
__host__ __device__ inline int adv_threads(const AdvJob& j, int threads) {
  return j.L > 0 ? kAdvThreads : (threads < 128 ? threads : 128);
}

int adv_blocks(const AdvJob& j, int threads) {
  const int64_t per_block = adv_threads(j, threads) / (j.L > 0 ? j.L : 1);
  return static_cast<int>((j.n_groups + per_block - 1) / per_block);
}

// Block b of the job's blocks.
__device__ void adv_block(const AdvJob& j, int64_t b) {
  const int threads = adv_threads(j, blockDim.x);
  if (static_cast<int>(threadIdx.x) >= threads) return;
  if (j.L > 0) {
    group_adv_lanes(j.reward, j.accepted, j.n_groups, j.G, j.L, j.eps, j.unbiased, j.adv, b);
  } else {
    const int64_t g = b * threads + threadIdx.x;
    if (g < j.n_groups) group_adv_thread(j.reward, j.accepted, g, j.G, j.eps, j.unbiased, j.adv);
  }
}

// For list_few_rows_kernel: inlined, the 50 KB of unrolled fp64 loops in the middle of its code
// cost a list of 200 rows 4 us after other kernels (9.3 and 5.1 us).
__device__ __noinline__ void adv_block_call(const AdvJob& j, int64_t b) { adv_block(j, b); }

// Also checks the sequence offsets and clears a counter, for the launch that follows
// (offsets / counter may be null).
__global__ void __launch_bounds__(kAdvThreads)
    group_adv_kernel(AdvJob j, const int64_t* __restrict__ seq_offsets, int64_t n_seq,
                     int64_t n_rows, unsigned* counter, int32_t* status) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (counter && t == 0) *counter = 0u;
  if (seq_offsets)
    for (int64_t i = t; i < n_seq; i += static_cast<int64_t>(gridDim.x) * blockDim.x)
      check_seq(seq_offsets, i, n_rows, status);
  adv_block(j, blockIdx.x);  // past the job's blocks: none of the groups
}

// ------------------------------------------------------------ surrogate

__device__ __forceinline__ float clamped_ratio(float lp, float behav) {
  const float d = lp - behav;
  return expf(fminf(fmaxf(d, -20.0f), 20.0f));
}

__device__ __forceinline__ float clipped_term(float rho, float a, float eps_low, float eps_high,
                                              float dual) {
  const float rc = fminf(fmaxf(rho, 1.0f - eps_low), 1.0f + eps_high);
  const float p1 = -a * rho;
  const float p2 = -a * rc;
  float l = fmaxf(p1, p2);
  if (a < 0.0f) l = fminf(l, -dual * a);
  return l;
}

// The batch's numerator and denominator.  Per-token terms in fp32, every sum in
// fp64 and in a fixed order.  TOKEN_MEAN needs the whole sums only: a lane adds its
// rows, a warp its lanes, a block its warps, and the block that finishes last (the
// counter, cleared by the launch before) adds the blocks' sums and divides.
// SEQ_MEAN needs each sequence's: a warp writes the part of a sequence that begins
// in its tile to the sequence's slot and the part of one that began earlier to the
// tile's head slot; seq_mean_kernel adds a sequence's slot and head slots, a warp
// per sequence, and its last block adds the means.
struct SurrogateArgs {
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
  float* ratio;
  SurrogateWs ws;
  double* loss;
  double* partial;
};

// A lane's running sum of a tile's terms, exact to well past fp64's 53 bits, in three
// floats: each addition's rounding error is itself added, and that addition's error
// kept (Knuth's two-sum, twice).  Eight terms cost one conversion to fp64 instead of
// eight conversions and additions, which held the kernel to GB300's narrow fp64 pipe
// (61 % busy).  Terms are below 2^60 in magnitude (|A| <= sqrt(G), rho <= e^20), so
// no sum overflows; NaN stays NaN.
struct Sum3 {
  float s, e, f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x);
    const float z = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
    s = t;
    const float t2 = __fadd_rn(e, err);
    const float z2 = __fsub_rn(t2, e);
    f = __fadd_rn(f, __fadd_rn(__fsub_rn(e, __fsub_rn(t2, z2)), __fsub_rn(err, z2)));
    e = t2;
  }
  __device__ __forceinline__ double value() const {
    return __dadd_rn(static_cast<double>(s),
                     __dadd_rn(static_cast<double>(e), static_cast<double>(f)));
  }
};

__device__ __forceinline__ double warp_sum_fixed(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// By the block of a launch that finishes last (uniform over each block): the sums of
// s[0, n) and c[0, n) and the aggregate.  Every thread of every block calls it once.
__device__ void finish_in_last_block(unsigned* counter, const double* s, const double* c,
                                     int64_t n, double* loss, double* partial) {
  __shared__ bool s_last;
  __shared__ double sh_a[kRowWarps], sh_b[kRowWarps];
  __threadfence();  // this thread's sums before the block's arrival
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = 0.0, b = 0.0;
#pragma unroll 4
  for (int64_t i = threadIdx.x; i < n; i += kRowThreads) {
    a = __dadd_rn(a, __ldcg(s + i));
    b = __dadd_rn(b, __ldcg(c + i));
  }
  a = warp_sum_fixed(a);
  b = warp_sum_fixed(b);
  if ((threadIdx.x & 31) == 0) {
    sh_a[threadIdx.x >> 5] = a;
    sh_b[threadIdx.x >> 5] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kRowWarps; ++i) {
      a = __dadd_rn(a, sh_a[i]);
      b = __dadd_rn(b, sh_b[i]);
    }
    *loss = b > 0.0 ? __ddiv_rn(a, b) : 0.0;
    if (partial) {
      partial[0] = a;
      partial[1] = b;
    }
  }
}

// SEQ_MEAN: per sequence its mean (0 without rows in the loss) and whether it has any.
__global__ void __launch_bounds__(kRowThreads) seq_mean_kernel(SurrogateArgs p) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * kRowWarps;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kRowWarps + (threadIdx.x >> 5); i < p.n_seq;
       i += warps) {
    const int64_t r0 = p.seq_offsets[i], r1 = p.seq_offsets[i + 1];
    const bool any = r0 >= 0 && r1 <= p.n_rows && r1 > r0 &&
                     (p.seq_accepted ? p.seq_accepted[i] != 0 : true);
    double s = 0.0, c = 0.0;
    if (any) {
      const int64_t w0 = r0 / kRowTile, w1 = (r1 - 1) / kRowTile;
      for (int64_t w = w0 + lane; w <= w1; w += 32) {
        s = __dadd_rn(s, __ldcg(w == w0 ? p.ws.seq_sum + i : p.ws.head_sum + w));
        c = __dadd_rn(c, __ldcg(w == w0 ? p.ws.seq_cnt + i : p.ws.head_cnt + w));
      }
    }
    s = warp_sum_fixed(s);
    c = warp_sum_fixed(c);
    if (lane == 0) {
      p.ws.seq_sum[i] = c > 0.0 ? __ddiv_rn(s, c) : 0.0;
      p.ws.seq_cnt[i] = c > 0.0 ? 1.0 : 0.0;
    }
  }
  finish_in_last_block(p.ws.counter, p.ws.seq_sum, p.ws.seq_cnt, p.n_seq, p.loss, p.partial);
}

// TOKEN_MEAN: every row's term is computed once per tile, without a branch, so that the
// eight rows' chains of latencies overlap (loss and derivative over 5.4M rows 58.0 -> 55.6
// us).
__global__ void __launch_bounds__(kRowThreads, kRowMinBlocks) surrogate_kernel(SurrogateArgs p) {
  __shared__ double sh_sum[kRowWarps], sh_cnt[kRowWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t w0 = (static_cast<int64_t>(blockIdx.x) * kRowWarps + wid) * p.geom.per_warp;
  const int64_t w1 = w0 + p.geom.per_warp < p.geom.n_tiles ? w0 + p.geom.per_warp : p.geom.n_tiles;
  double tot = 0.0;
  int cnt = 0;
  if (w0 < w1) {
    int64_t t0 = w0 * kRowTile;
    RowLoads cur, nxt;
    cur.load(p.logprob, p.behav, p.mask, t0, tile_end(t0, p.n_rows), p.vec);
    PieceWalker<FloatOf> pw(p.seq_offsets, p.seq_accepted, FloatOf{p.adv}, p.n_seq, t0);
    for (int64_t w = w0; w < w1; ++w) {
      const int64_t t1 = tile_end(t0, p.n_rows);
      if (w + 1 < w1) nxt.load(p.logprob, p.behav, p.mask, t1, tile_end(t1, p.n_rows), p.vec);
      unsigned in = 0u;
      float adv[kRowsPerLane] = {};
      pw.walk(t0, t1, [&](int64_t, int64_t lo, int64_t hi, float a, int64_t) {
        const unsigned rows = piece_bits(t0, lo, hi) & cur.mask;
        in |= rows;
#pragma unroll
        for (int u = 0; u < kRowsPerLane; ++u) adv[u] = rows >> u & 1u ? a : adv[u];
      });
      if (__any_sync(0xffffffffu, in != 0u)) {
        Sum3 sum{0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int u = 0; u < kRowsPerLane; ++u) {
          cur.bh[u] = clamped_ratio(cur.lp[u], cur.bh[u]);  // the ratio, once the row is used
          const float x = clipped_term(cur.bh[u], adv[u], p.eps_low, p.eps_high, p.dual);
          sum.add(in >> u & 1u ? x : 0.0f);
        }
        tot = __dadd_rn(tot, sum.value());
        cnt += __popc(in);
      }
      if (p.ratio) store_rows(p.ratio, t0, t1, p.vec, in, cur.bh);
      cur = nxt;
      t0 = t1;
    }
  }
  tot = warp_sum_fixed(tot);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) {
    sh_sum[wid] = tot;
    sh_cnt[wid] = static_cast<double>(cnt);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = sh_sum[0], c = sh_cnt[0];
    for (int i = 1; i < kRowWarps; ++i) {
      s = __dadd_rn(s, sh_sum[i]);
      c = __dadd_rn(c, sh_cnt[i]);
    }
    p.ws.block_sum[blockIdx.x] = s;
    p.ws.block_cnt[blockIdx.x] = c;
  }
  finish_in_last_block(p.ws.counter, p.ws.block_sum, p.ws.block_cnt, gridDim.x, p.loss, p.partial);
}

// SEQ_MEAN: a tile's pieces go through shared memory; where there are several, so do its
// ratios, and groups of 16 to 4 lanes add up a piece each.  With the whole warp on every
// piece in turn, 5,000 rows of 1,000 sequences took 75 us a call (1.2 us a piece), now 20;
// 5.4M rows of 1,024 sequences 35 and 35.
__global__ void __launch_bounds__(kRowThreads, kRowMinBlocks)
    surrogate_seq_kernel(SurrogateArgs p) {
  __shared__ PieceList lists[kRowWarps];
  __shared__ float values[kRowWarps][kRowTile];            // per piece: the advantage
  __shared__ __align__(16) float ratios[kRowWarps][kRowTile];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  PieceList& list = lists[wid];
  const int64_t w0 = (static_cast<int64_t>(blockIdx.x) * kRowWarps + wid) * p.geom.per_warp;
  const int64_t w1 = w0 + p.geom.per_warp < p.geom.n_tiles ? w0 + p.geom.per_warp : p.geom.n_tiles;
  if (w0 >= w1) return;
  int64_t t0 = w0 * kRowTile;
  RowLoads cur, nxt;
  cur.load(p.logprob, p.behav, p.mask, t0, tile_end(t0, p.n_rows), p.vec);
  PieceWalker<FloatOf> pw(p.seq_offsets, p.seq_accepted, FloatOf{p.adv}, p.n_seq, t0);
  for (int64_t w = w0; w < w1; ++w) {
    const int64_t t1 = tile_end(t0, p.n_rows);
    if (w + 1 < w1) nxt.load(p.logprob, p.behav, p.mask, t1, tile_end(t1, p.n_rows), p.vec);
#pragma unroll
    for (int u = 0; u < kRowsPerLane; ++u) cur.bh[u] = clamped_ratio(cur.lp[u], cur.bh[u]);
    bool began_before = false;  // by the lane that holds the first piece
    int n = pw.collect(t0, t1, [&](int i, int64_t seq, int64_t lo, int64_t hi, float a,
                                   int64_t begin) {
      list.put(i, seq, t0, lo, hi);
      if (i < kRowTile) values[wid][i] = a;
      if (i == 0) began_before = begin < t0;
    });
    const bool first_began_before = __any_sync(0xffffffffu, began_before);
    n = n < kRowTile ? n : kRowTile;
    const auto put_part = [&](int q, double sum, int count) {
      const bool head = q == 0 && first_began_before;
      const int64_t i = head ? w : list.seq[q];
      (head ? p.ws.head_sum : p.ws.seq_sum)[i] = sum;
      (head ? p.ws.head_cnt : p.ws.seq_cnt)[i] = static_cast<double>(count);
    };
    unsigned in = 0u;
    if (n == 1) {  // a long sequence's tile: the lanes add up their own rows
      __syncwarp();
      const float a = values[wid][0];
      in = list.rows_in_piece(0) & cur.mask;
      Sum3 sum{0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int u = 0; u < kRowsPerLane; ++u) {
        const float x = clipped_term(cur.bh[u], a, p.eps_low, p.eps_high, p.dual);
        sum.add(in >> u & 1u ? x : 0.0f);
      }
      const double s = warp_sum_fixed(sum.value());
      const int c = __reduce_add_sync(0xffffffffu, __popc(in));
      if (lane == 0) put_part(0, s, c);
    } else if (n > 1) {
      float4* r4 = reinterpret_cast<float4*>(ratios[wid] + row_in_tile(0));
      r4[0] = make_float4(cur.bh[0], cur.bh[1], cur.bh[2], cur.bh[3]);
      r4[1] = make_float4(cur.bh[4], cur.bh[5], cur.bh[6], cur.bh[7]);
      list.put_mask(cur.mask);
      __syncwarp();
      const int g = n <= 2 ? 16 : (n <= 4 ? 8 : 4);  // lanes a piece
      const int sub = lane & (g - 1);
      for (int q0 = 0; q0 < n; q0 += 32 / g) {
        const int q = q0 + lane / g;
        Sum3 sum{0.0f, 0.0f, 0.0f};
        int c = 0;
        if (q < n) {
          const float a = values[wid][q];
          const int hi = list.range[q] >> 16;
          for (int r = (list.range[q] & 0xffffu) + sub; r < hi; r += g) {
            const bool take = list.in_mask(r);
            const float x = clipped_term(ratios[wid][r], a, p.eps_low, p.eps_high, p.dual);
            sum.add(take ? x : 0.0f);
            c += take;
          }
        }
        double s = sum.value();
        for (int o = g >> 1; o > 0; o >>= 1) {
          s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
          c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (q < n && sub == 0) put_part(q, s, c);
      }
      in = list.rows_in_pieces(n) & cur.mask;
    }
    if (lane == 0 && !first_began_before) {
      p.ws.head_sum[w] = 0.0;
      p.ws.head_cnt[w] = 0.0;
    }
    if (p.ratio) store_rows(p.ratio, t0, t1, p.vec, in, cur.bh);
    __syncwarp();  // the list is rewritten
    cur = nxt;
    t0 = t1;
  }
}

// loss = numerator / denominator of partials summed over the parts of a batch
// (0 for an empty loss), the same correctly rounded division as above.
__global__ void loss_from_partial_kernel(const double* __restrict__ partial,
                                         double* __restrict__ loss) {
  if (threadIdx.x == 0 && blockIdx.x == 0)
    *loss = partial[1] > 0.0 ? __ddiv_rn(partial[0], partial[1]) : 0.0;
}

void carve_surrogate_ws(Carver& cv, int64_t n_rows, int64_t n_seq, SurrogateWs* w) {
  const size_t blocks = row_blocks_bound(n_rows);
  const int64_t n_tiles = row_geom(n_rows).n_tiles;
  const size_t tiles = n_tiles > 0 ? static_cast<size_t>(n_tiles) : 1;
  w->seq_sum = cv.take<double>(n_seq > 0 ? n_seq : 1);
  w->seq_cnt = cv.take<double>(n_seq > 0 ? n_seq : 1);
  w->head_sum = cv.take<double>(tiles);
  w->head_cnt = cv.take<double>(tiles);
  w->block_sum = cv.take<double>(blocks);
  w->block_cnt = cv.take<double>(blocks);
  w->adv = cv.take<float>(n_seq > 0 ? n_seq : 1);
  w->counter = cv.take<unsigned>(1);
}

pace_status check_batch(const PaceBatch* b) {
  if (!b) return PACE_ERR_INVALID_ARG;
  if (b->n_seq < 0 || b->n_rows < 0) return PACE_ERR_INVALID_ARG;
  if (b->n_seq > 0 && !b->seq_offsets) return PACE_ERR_INVALID_ARG;
  if (b->n_rows >= (int64_t(1) << 31)) return PACE_ERR_UNSUPPORTED_SHAPE;
  return PACE_OK;
}

pace_status check_loss_args(const PaceBatch* b, const PaceLossArgs* l) {
  if (!l || !l->behav_lp || !l->reward || !l->loss) return PACE_ERR_INVALID_ARG;
  if (l->group_size < 1 || b->n_seq % l->group_size != 0) return PACE_ERR_INVALID_ARG;
  const PaceLossParams& p = l->params;
  if (!(p.eps_low >= 0.0f && p.eps_low < 1.0f) || !(p.eps_high >= 0.0f) ||
      !(p.dual_clip >= 1.0f) || !(p.adv_eps >= 0.0f))
    return PACE_ERR_INVALID_ARG;
  if (p.agg != PACE_AGG_TOKEN_MEAN && p.agg != PACE_AGG_SEQ_MEAN_TOKEN_MEAN)
    return PACE_ERR_INVALID_ARG;
  return PACE_OK;
}

pace_status launch_group_adv(const AdvJob& j, const PaceBatch* b, unsigned* counter,
                             int32_t* status, cudaStream_t st) {
  const int64_t n_seq = b ? b->n_seq : 0;
  // the offsets are checked whether or not there are advantages to compute
  int64_t blocks = (n_seq + kAdvThreads - 1) / kAdvThreads;
  if (blocks > 1024) blocks = 1024;
  if (blocks < adv_blocks(j, kAdvThreads)) blocks = adv_blocks(j, kAdvThreads);
  if (blocks == 0 && !counter) return PACE_OK;
  group_adv_kernel<<<static_cast<unsigned>(blocks > 0 ? blocks : 1), kAdvThreads, 0, st>>>(
      j, b ? b->seq_offsets : nullptr, n_seq, b ? b->n_rows : 0, counter, status);
  return last_launch_status();
}

// Advantages, per-token terms and the aggregate; logprob is [n_rows].  adv_done: an
// earlier launch of the call has computed the advantages, checked the offsets and
// cleared the counter.
pace_status run_surrogate(const PaceBatch* b, const float* logprob, const PaceLossArgs* l,
                          const SurrogateWs& ws, bool adv_done, int32_t* status,
                          cudaStream_t st) {
  float* adv = l->adv ? l->adv : ws.adv;
  if (!adv_done)
    PACE_TRY(launch_group_adv(adv_job(l->reward, b->seq_accepted, b->n_seq, l->group_size,
                                      l->params.adv_eps, l->params.std_unbiased, adv),
                              b, ws.counter, status, st));
  SurrogateArgs a;
  a.seq_offsets = b->seq_offsets;
  a.seq_accepted = b->seq_accepted;
  a.mask = b->mask;
  a.logprob = logprob;
  a.behav = l->behav_lp;
  a.adv = adv;
  a.n_seq = b->n_seq;
  a.n_rows = b->n_rows;
  a.geom = row_geom(b->n_rows);
  a.vec = rows_vec(logprob, l->behav_lp, l->ratio, b->mask);
  a.eps_low = l->params.eps_low;
  a.eps_high = l->params.eps_high;
  a.dual = l->params.dual_clip;
  a.ratio = l->ratio;
  a.ws = ws;
  a.loss = l->loss;
  a.partial = l->partial;
  const unsigned grid = static_cast<unsigned>(a.geom.blocks > 0 ? a.geom.blocks : 1);
  if (l->params.agg == PACE_AGG_TOKEN_MEAN) {
    surrogate_kernel<<<grid, kRowThreads, 0, st>>>(a);
    return last_launch_status();
  }
  surrogate_seq_kernel<<<grid, kRowThreads, 0, st>>>(a);
  PACE_TRY(last_launch_status());
  int64_t blocks = (b->n_seq + kRowWarps - 1) / kRowWarps;
  const int64_t most = static_cast<int64_t>(sm_count()) * 8;
  if (blocks > most) blocks = most;
  seq_mean_kernel<<<static_cast<unsigned>(blocks > 0 ? blocks : 1), kRowThreads, 0, st>>>(a);
  return last_launch_status();
}

// ------------------------------------------------------------ compaction

// Rows in the loss per warp and per block of the row walk; the same blocks check the
// offsets, and the blocks after the walk's compute the advantages of a call that
// needs them.  Clears the two counters of the launches that follow (either may be
// null).  seq_in (or null): rows in the loss per sequence, added to, and n_used the
// sequences that have any.
template <bool kPerSeq>
__global__ void __launch_bounds__(kRowThreads)
    count_rows_kernel(const int64_t* __restrict__ seq_offsets,
                      const uint8_t* __restrict__ seq_accepted, const uint8_t* __restrict__ mask,
                      int64_t n_seq, int64_t n_rows, RowGeom geom, bool vec, RowCounts counts,
                      unsigned long long* __restrict__ seq_in, int* __restrict__ n_used,
                      AdvJob adv, unsigned* counter0, unsigned* counter1, int32_t* status) {
  if (static_cast<int>(blockIdx.x) >= geom.blocks) {
    adv_block(adv, blockIdx.x - geom.blocks);
    return;
  }
  __shared__ long long sh[kRowWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t == 0) {
    if (counter0) *counter0 = 0u;
    if (counter1) *counter1 = 0u;
  }
  const int64_t threads = static_cast<int64_t>(geom.blocks) * blockDim.x;
  for (int64_t i = t; i < n_seq; i += threads) check_seq(seq_offsets, i, n_rows, status);
  const int64_t warp = static_cast<int64_t>(blockIdx.x) * kRowWarps + wid;
  const int64_t w0 = warp * geom.per_warp;
  const int64_t w1 = w0 + geom.per_warp < geom.n_tiles ? w0 + geom.per_warp : geom.n_tiles;
  int c = 0;
  if constexpr (kPerSeq) {
    // a lane counts a piece (the warp on one piece after the other waited for each atomic's
    // result, about 1 us)
    __shared__ PieceList lists[kRowWarps];
    PieceList& list = lists[wid];
    if (w0 < w1) {
      PieceWalker<NoValue> pw(seq_offsets, seq_accepted, NoValue{}, n_seq, w0 * kRowTile);
      for (int64_t w = w0; w < w1; ++w) {
        const int64_t t0 = w * kRowTile, t1 = tile_end(t0, n_rows);
        list.put_mask(load_mask_bits(mask, t0, t1, vec));
        int n = pw.collect(t0, t1, [&](int i, int64_t seq, int64_t lo, int64_t hi, NoValue, int64_t) {
          list.put(i, seq, t0, lo, hi);
        });
        n = n < kRowTile ? n : kRowTile;
        __syncwarp();
        int first = 0;
        for (int q = lane; q < n; q += 32) {
          const int k = list.rows_in_mask(q);
          if (k > 0 && atomicAdd(seq_in + list.seq[q], static_cast<unsigned long long>(k)) == 0)
            ++first;
          c += k;
        }
        first = __reduce_add_sync(0xffffffffu, first);
        if (lane == 0 && first > 0) atomicAdd(n_used, first);
        __syncwarp();  // the list is rewritten
      }
    }
  } else {
    walk_rows_in_loss(seq_offsets, seq_accepted, mask, n_seq, n_rows, w0, w1, vec,
                      [&](int64_t, int64_t, unsigned in) { c += __popc(in); });
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) {
    sh[wid] = c;
    counts.warp[warp] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long s = 0;
    for (int i = 0; i < kRowWarps; ++i) s += sh[i];
    counts.block[blockIdx.x] = s;
  }
}

// A tile's rows in the loss (the lanes' bits) into the list from entry `before` on; lp
// and lse (or null) of its other rows are set to 0.
__device__ __forceinline__ void list_tile(int64_t t0, int64_t t1, unsigned in, long long& before,
                                          int32_t* __restrict__ rowidx, float* __restrict__ lp,
                                          float* __restrict__ lse) {
  const int lane = threadIdx.x & 31;
  // 32 rows at a time, lane l row l of them (held by lane l / 8 of four), so that the
  // warp's stores are consecutive
#pragma unroll
  for (int u = 0; u < kRowTile / 32; ++u) {
    const int64_t r = t0 + 32 * u + lane;
    const bool k = __shfl_sync(0xffffffffu, in, 4 * u + (lane >> 3)) >> (lane & 7) & 1u;
    const unsigned bal = __ballot_sync(0xffffffffu, k);
    if (k) {
      rowidx[before + __popc(bal & ((1u << lane) - 1u))] = static_cast<int32_t>(r);
    } else if (r < t1) {
      if (lp) lp[r] = 0.0f;
      if (lse) lse[r] = 0.0f;
    }
    before += __popc(bal);
  }
}

// The row indices of the rows in the loss, in row order; their number in *total.
// Every block adds up the counts of the blocks before it itself (at most
// kMaxRowBlocks of them), so there is no launch for a scan.  lp and lse (or null) of
// rows outside the loss are set to 0 here.
__global__ void __launch_bounds__(kRowThreads)
    write_rows_kernel(const int64_t* __restrict__ seq_offsets,
                      const uint8_t* __restrict__ seq_accepted, const uint8_t* __restrict__ mask,
                      int64_t n_seq, int64_t n_rows, RowGeom geom, bool vec, RowCounts counts,
                      int32_t* __restrict__ rowidx, long long* __restrict__ total,
                      float* __restrict__ lp, float* __restrict__ lse) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t warp = static_cast<int64_t>(blockIdx.x) * kRowWarps + wid;
  const int64_t w0 = warp * geom.per_warp;
  const int64_t w1 = w0 + geom.per_warp < geom.n_tiles ? w0 + geom.per_warp : geom.n_tiles;
  long long mine = 0;
  for (int i = threadIdx.x; i < static_cast<int>(blockIdx.x); i += kRowThreads)
    mine += counts.block[i];
  const int wc = lane < wid ? counts.warp[warp - wid + lane] : 0;
  long long before = 0;
  block_exclusive_scan<long long>(mine, &before);
  if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1)
    *total = before + counts.block[blockIdx.x];
  before += __reduce_add_sync(0xffffffffu, wc);
  walk_rows_in_loss(seq_offsets, seq_accepted, mask, n_seq, n_rows, w0, w1, vec,
                    [&](int64_t t0, int64_t t1, unsigned in) {
                      list_tile(t0, t1, in, before, rowidx, lp, lse);
                    });
}

// Up to kFewRows rows: the count and the list in one launch, whose blocks (32 tiles each,
// one a warp) count the tiles before theirs again.  Bound by latency and the launch: a
// log-prob call (H 64, V 64, one graph replay of ten) took 30 us in two launches and 25
// in one at 200 rows, 38 and 34 at 4,096, 39 and 37 at 10,000, 39.6 and 39.6 at 16,384,
// 39.7 and 41.7 at 24,576, where the line could lie no higher.
constexpr int kFewThreads = 1024;
constexpr int kFewWarps = kFewThreads / 32;
constexpr int64_t kFewRows = 2 * kFewWarps * kRowTile;

__global__ void __launch_bounds__(kFewThreads)
    list_few_rows_kernel(const int64_t* __restrict__ seq_offsets,
                         const uint8_t* __restrict__ seq_accepted,
                         const uint8_t* __restrict__ mask, int64_t n_seq, int64_t n_rows,
                         int blocks, bool vec, int32_t* __restrict__ rowidx,
                         long long* __restrict__ total, float* __restrict__ lp,
                         float* __restrict__ lse, AdvJob adv, unsigned* counter0,
                         unsigned* counter1, int32_t* status) {
  if (static_cast<int>(blockIdx.x) >= blocks) {
    adv_block_call(adv, blockIdx.x - blocks);
    return;
  }
  __shared__ int sh_before[kFewWarps], sh_own[kFewWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t t = static_cast<int64_t>(blockIdx.x) * kFewThreads + threadIdx.x;
  if (t == 0) {
    if (counter0) *counter0 = 0u;
    if (counter1) *counter1 = 0u;
  }
  for (int64_t i = t; i < n_seq; i += static_cast<int64_t>(blocks) * kFewThreads)
    check_seq(seq_offsets, i, n_rows, status);
  // block b's 32 warps share the 32 b tiles before its own, b each
  const int64_t b = blockIdx.x, n_tiles = (n_rows + kRowTile - 1) / kRowTile;
  int c = 0;
  walk_rows_in_loss(seq_offsets, seq_accepted, mask, n_seq, n_rows, wid * b, (wid + 1) * b, vec,
                    [&](int64_t, int64_t, unsigned in) { c += __popc(in); });
  const int64_t w = b * kFewWarps + wid;
  unsigned own = 0u;
  walk_rows_in_loss(seq_offsets, seq_accepted, mask, n_seq, n_rows, w, w < n_tiles ? w + 1 : w,
                    vec, [&](int64_t, int64_t, unsigned in) { own = in; });
  c = __reduce_add_sync(0xffffffffu, c);
  const int n_own = __reduce_add_sync(0xffffffffu, __popc(own));
  if (lane == 0) {
    sh_before[wid] = c;
    sh_own[wid] = n_own;
  }
  __syncthreads();
  long long before = __reduce_add_sync(0xffffffffu, sh_before[lane] + (lane < wid ? sh_own[lane] : 0));
  if (b == blocks - 1 && wid == kFewWarps - 1 && lane == 0) *total = before + n_own;
  if (w < n_tiles) {
    const int64_t t0 = w * kRowTile;
    list_tile(t0, tile_end(t0, n_rows), own, before, rowidx, lp, lse);
  }
}

// Copy the hidden rows listed in rowidx into a dense buffer, one warp per row,
// 16 bytes per lane per step.
__global__ void gather_rows_kernel(const uint4* __restrict__ hidden, int64_t row_vecs,
                                   const int32_t* __restrict__ rowidx,
                                   const long long* __restrict__ n_in, uint4* __restrict__ out) {
  const long long m = *n_in;
  const int lane = threadIdx.x & 31;
  const int64_t warps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; r < m;
       r += warps) {
    const uint4* src = hidden + static_cast<int64_t>(rowidx[r]) * row_vecs;
    uint4* dst = out + r * row_vecs;
    for (int64_t v = lane; v < row_vecs; v += 32) dst[v] = __ldg(src + v);
  }
}

RowCounts carve_row_counts(Carver& cv, int64_t n_rows) {
  const size_t blocks = row_blocks_bound(n_rows);
  RowCounts c;
  c.block = cv.take<long long>(blocks);
  c.warp = cv.take<int>(blocks * kRowWarps);
  return c;
}

void carve_compact_ws(Carver& cv, int64_t n_rows, CompactWs* w) {
  w->counts = carve_row_counts(cv, n_rows);
  w->total = cv.take<long long>(1);
  w->rowidx = cv.take<int32_t>(n_rows > 0 ? n_rows : 1);
}

pace_status launch_count_rows(const PaceBatch* b, RowCounts counts, unsigned long long* seq_in,
                              int* n_used, const AdvJob& adv, unsigned* counter0,
                              unsigned* counter1, int32_t* status, cudaStream_t st) {
  const RowGeom g = row_geom(b->n_rows);
  const auto kernel = seq_in ? count_rows_kernel<true> : count_rows_kernel<false>;
  kernel<<<static_cast<unsigned>(g.blocks + adv_blocks(adv, kRowThreads)), kRowThreads, 0, st>>>(
      b->seq_offsets, b->seq_accepted, b->mask, b->n_seq, b->n_rows, g, aligned(b->mask, 8), counts,
      seq_in, n_used, adv, counter0, counter1, status);
  return last_launch_status();
}

pace_status run_compaction(const PaceBatch* b, const CompactWs& ws, const AdvJob& adv,
                           unsigned* counter0, unsigned* counter1, float* lp, float* lse,
                           int32_t* status, cudaStream_t st) {
  if (b->n_seq == 0 || b->n_rows == 0) {
    PACE_TRY_CUDA(cudaMemsetAsync(ws.total, 0, sizeof(long long), st));
    const size_t bytes = static_cast<size_t>(b->n_rows) * sizeof(float);
    if (lp && bytes) PACE_TRY_CUDA(cudaMemsetAsync(lp, 0, bytes, st));
    if (lse && bytes) PACE_TRY_CUDA(cudaMemsetAsync(lse, 0, bytes, st));
    if (counter1) PACE_TRY_CUDA(cudaMemsetAsync(counter1, 0, sizeof(unsigned), st));
    return launch_group_adv(adv, b, counter0, status, st);
  }
  if (b->n_rows <= kFewRows) {
    const int blocks = static_cast<int>((b->n_rows + kFewWarps * kRowTile - 1) /
                                        (kFewWarps * kRowTile));
    list_few_rows_kernel<<<static_cast<unsigned>(blocks + adv_blocks(adv, kFewThreads)), kFewThreads, 0, st>>>(
        b->seq_offsets, b->seq_accepted, b->mask, b->n_seq, b->n_rows, blocks,
        aligned(b->mask, 8), ws.rowidx, ws.total, lp, lse, adv, counter0, counter1, status);
    return last_launch_status();
  }
  PACE_TRY(launch_count_rows(b, ws.counts, nullptr, nullptr, adv, counter0, counter1, status, st));
  const RowGeom g = row_geom(b->n_rows);
  write_rows_kernel<<<static_cast<unsigned>(g.blocks), kRowThreads, 0, st>>>(
      b->seq_offsets, b->seq_accepted, b->mask, b->n_seq, b->n_rows, g, aligned(b->mask, 8),
      ws.counts, ws.rowidx,
      ws.total, lp, lse);
  return last_launch_status();
}

pace_status run_gather(const void* hidden, int H, int64_t n_rows, const CompactWs& ws,
                       void* out, cudaStream_t st) {
  if (n_rows == 0) return PACE_OK;
  const int64_t row_vecs = static_cast<int64_t>(H) * 2 / 16;
  int64_t blocks = (n_rows + 7) / 8;
  const int64_t cap = static_cast<int64_t>(sm_count()) * 16;
  if (blocks > cap) blocks = cap;
  gather_rows_kernel<<<static_cast<unsigned>(blocks), 256, 0, st>>>(
      static_cast<const uint4*>(hidden), row_vecs, ws.rowidx, ws.total,
      static_cast<uint4*>(out));
  return last_launch_status();
}

}  // namespace pace

using namespace pace;

extern "C" void pace_loss_params_default(PaceLossParams* p) {
  if (!p) return;
  p->eps_low = 0.2f;
  p->eps_high = 0.28f;
  p->dual_clip = 10.0f;
  p->adv_eps = 1e-6f;
  p->agg = PACE_AGG_TOKEN_MEAN;
  p->std_unbiased = 1;
}

extern "C" pace_status pace_group_advantages(const float* reward, const uint8_t* seq_accepted,
                                             int64_t n_seq, int32_t group_size, float adv_eps,
                                             int32_t std_unbiased, float* adv, void* stream) {
  if (n_seq < 0 || group_size < 1 || n_seq % group_size != 0) return PACE_ERR_INVALID_ARG;
  if (n_seq > 0 && (!reward || !adv)) return PACE_ERR_INVALID_ARG;
  if (!(adv_eps >= 0.0f)) return PACE_ERR_INVALID_ARG;
  return launch_group_adv(
      adv_job(reward, seq_accepted, n_seq, group_size, adv_eps, std_unbiased, adv), nullptr,
      nullptr, nullptr, as_stream(stream));
}

extern "C" size_t pace_surrogate_loss_workspace_size(int64_t n_rows, int64_t n_seq) {
  if (n_rows < 0 || n_seq < 0) return 0;
  Carver cv;
  SurrogateWs w;
  carve_surrogate_ws(cv, n_rows, n_seq, &w);
  return cv.used;
}

extern "C" pace_status pace_surrogate_loss(const PaceBatch* batch, const float* logprob,
                                           const PaceLossArgs* loss, void* workspace,
                                           size_t workspace_bytes, int32_t* status_dev,
                                           void* stream) {
  PACE_TRY(check_batch(batch));
  PACE_TRY(check_loss_args(batch, loss));
  if (batch->n_rows > 0 && !logprob) return PACE_ERR_INVALID_ARG;
  if (!workspace || !aligned(workspace, 256)) return PACE_ERR_WORKSPACE;
  Carver cv(workspace, workspace_bytes);
  SurrogateWs ws;
  carve_surrogate_ws(cv, batch->n_rows, batch->n_seq, &ws);
  if (!cv.fits()) return PACE_ERR_WORKSPACE;
  return run_surrogate(batch, logprob, loss, ws, false, status_dev, as_stream(stream));
}

extern "C" pace_status pace_loss_from_partial(const double* partial, double* loss,
                                              void* stream) {
  if (!partial || !loss) return PACE_ERR_INVALID_ARG;
  pace::loss_from_partial_kernel<<<1, 32, 0, pace::as_stream(stream)>>>(partial, loss);
  return pace::last_launch_status();
}
