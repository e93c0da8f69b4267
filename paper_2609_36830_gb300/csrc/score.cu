// Pool scoring: Lemma 1 / Eq. 2 staleness decomposition, Eqs. 7-10 scores and
// the per-group mean, on sm_103a.
//
//   tag_reduce_kernel   one streaming pass over the int32 version tags (HBM
//                       bound): per trajectory the count T of policy tokens,
//                       the exact integer sum of their tags and the largest
//                       tag (+1, for the Lemma 1 premise check).
//                       The same launch also prepares the
//                       prefix-score window (extra blocks
//                       after the streaming ones, run in its tail): each puts a
//                       part of W in its sorted places and tabulates a part
//                       of F = phi(count / |W|) (Eqs. 9-10) for every
//                       possible count 0..|W| (F depends on s only through
//                       the count).
//   score_finalize_kernel  one thread per trajectory: K_gen, K_wait, the ECDF
//                       count of s against the window (binary search in the
//                       sorted window), F from the table, the mode's score
//                       (Eqs. 7-8), and the mean of each group of G in fixed
//                       left-to-right order.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "pace_internal.cuh"

namespace pace {
namespace {

constexpr int kReduceThreads = 256;  // 8 warps
constexpr int kTileTokens = 128;     // one int4 per lane
// Tiles of a warp's batch (128 tokens each), two register sets of them in flight in
// turn, and resident blocks per SM: 24 warps with 80 registers keep 48-96 KB of loads
// in flight per SM, which is what the memory needs.  No L2 prefetch runs beside them (only
// a range's first two batches are asked for early, before the search for its first
// trajectory): one of four batches ahead held every pool back (the prefetched lines compete
// with the loads).  Whole scoring + selection calls, graph replay: 20k pool 72.0 -> 66.7 us, 128k
// 316 -> 282, 1M 2203 -> 2129; pace_stale_k on 128k 293 -> 257.  Measured without the
// prefetch (tiles x blocks per SM, 128k / 1M pool): 8 x 2 337 us / 2.51 ms, 6 x 3 288 /
// 2.13, 4 x 4 296 / 2.16 (spills), 3 x 4 289 / 2.13, 2 x 6 367 / 3.0, one register set
// 4 x 6 595 / 4.6.  A plain read of the same bytes takes 239 us / 1.95 ms.
constexpr int kTiles = 4, kBlocksPerSm = 3;
constexpr int64_t kBatchTokens = kTileTokens * kTiles;
// Short streams get fewer warps rather than fewer batches a warp: below this
// many batches a warp, trajectories spread over several warps' ranges and their
// totals need more head slots.  On the 1k sweep pool (3.6 M tags, ~3,500 a
// trajectory) whole calls took 30.3 / 29.0 / 27.2 / 28.6 / 31.3 us with at
// least 1 / 2 / 4 / 8 / 16 batches a warp (the stream itself 12.3 -> 18.3 us);
// pools from ~15 M tags keep one full wave and are not affected.
constexpr int64_t kMinBatchesPerWarp = 4;
constexpr int kMaxWindow = 4096;
// Pools of at least this many trajectories finalise inside the tag reduction's
// launch (pace_set_score_fused_min_traj); smaller ones use a launch of their own.
constexpr int64_t kFusedMinTrajDefault = int64_t(1) << 18;

std::atomic<int64_t>& fused_min_traj() {
  static std::atomic<int64_t> v{kFusedMinTrajDefault};
  return v;
}

// Whether the current device takes cooperative launches (cached per device);
// where it does not, every pool finalises in a launch of its own.
bool cooperative_launch_ok() {
  constexpr int kMaxDevices = 64;
  static std::atomic<int> cache[kMaxDevices];  // 0 unknown, 1 yes, 2 no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
  int c = cache[dev].load();
  if (c == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) {
      (void)cudaGetLastError();
      v = 0;
    }
    c = v ? 1 : 2;
    cache[dev].store(c);
  }
  return c == 1;
}

__device__ __forceinline__ int4 ld_stream_v4(const int32_t* p) {
  int4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Batches of a range asked into L2 before the search for its first trajectory.
constexpr int kFirstBatches = 2;

// Bulk prefetch of a 16-byte-aligned range into L2 (no data returned).
__device__ __forceinline__ void l2_prefetch_bulk(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)),
               "r"(bytes)
               : "memory");
}

// Preparation blocks (32 window values each) from which, and batches a resident warp up to
// which, the stream leaves them room in its wave.
constexpr unsigned kRoomPrepBlocks = 64;
constexpr int64_t kRoomBatches = 12;

// ---- exact integer quotients without the fp64 pipe
//
// GB300's fp64 pipe is narrow.  The function below builds the same double from integer
// arithmetic: the result of __ddiv_rn(__ll2double_rn(S), T) for 64-bit S and 32-bit T > 0,
// bit for bit.  pace_stale_k's quotients are built this way (as fast as in fp64 there); the
// scores' finalisation divides in fp64.

// RN(RN53(S) / T): exactly __ddiv_rn(__ll2double_rn(S), (double)T), T >= 1.
// |S| is first rounded to 53 significant bits (a * 2^e, a < 2^53) as the
// conversion does; then q = a / T, r = a % T and the fraction r / T is
// developed in 32-bit digits by integer division, giving a 64-bit quotient
// with its leading bit set plus a sticky bit, which is rounded to 53 bits
// (nearest, ties to even).  The quotient lies in [2^-32, 2^63], always normal.
__device__ __forceinline__ double i64_div_u32_rn(long long S, unsigned T) {
  if (S == 0) return 0.0;
  const unsigned long long sign = S < 0 ? (1ull << 63) : 0ull;
  unsigned long long a = S < 0 ? 0ull - static_cast<unsigned long long>(S)
                               : static_cast<unsigned long long>(S);
  int e = 0;  // the dividend is a * 2^e
  {
    const int top = 63 - __clzll(static_cast<long long>(a));
    if (top > 52) {
      const int sh = top - 52;
      unsigned long long m = a >> sh;
      const unsigned long long rem = a & ((1ull << sh) - 1);
      const unsigned long long half = 1ull << (sh - 1);
      if (rem > half || (rem == half && (m & 1ull))) ++m;
      e = sh;
      if (m >> 53) {  // 2^53 = 2^52 * 2: keep a below 2^53
        m >>= 1;
        ++e;
      }
      a = m;
    }
  }
  const unsigned long long t = T;
  const unsigned long long q = a / t;
  const unsigned long long r = a - q * t;
  // fraction digits of r / T (r < T < 2^32, so each digit fits 32 bits)
  const unsigned long long n1 = r << 32;
  const unsigned long long d1 = n1 / t;
  const unsigned long long r1 = n1 - d1 * t;
  const unsigned long long n2 = r1 << 32;
  const unsigned long long d2 = n2 / t;
  const unsigned long long r2 = n2 - d2 * t;
  const unsigned long long frac = (d1 << 32) | d2;  // r / T = frac * 2^-64 + ...
  unsigned long long x;  // 64 significant bits, leading bit at 63
  bool sticky;
  int exp2;              // exponent of the leading bit
  if (q != 0) {
    const int lq = 64 - __clzll(static_cast<long long>(q));  // bits of q, 1..53
    const int f = 64 - lq;                                   // fraction bits kept, 11..63
    x = (q << f) | (frac >> lq);
    sticky = r2 != 0 || (frac & ((1ull << lq) - 1)) != 0;
    exp2 = lq - 1 + e;
  } else {
    // r / T >= 2^-32: frac has at most 31 leading zeros; a third digit refills them
    const unsigned long long n3 = r2 << 32;
    const unsigned long long d3 = n3 / t;
    const unsigned long long r3 = n3 - d3 * t;
    const int lz = __clzll(static_cast<long long>(frac));  // 0..31
    x = lz ? (frac << lz) | (d3 >> (32 - lz)) : frac;
    sticky = r3 != 0 || (lz ? ((d3 << (32 + lz)) != 0) : (d3 != 0));
    exp2 = -1 - lz + e;
  }
  unsigned long long mant = x >> 11;  // 53 bits
  const bool round_bit = (x >> 10) & 1ull;
  const bool rest = sticky || (x & 0x3FFull) != 0;
  if (round_bit && (rest || (mant & 1ull))) ++mant;
  if (mant >> 53) {
    mant >>= 1;
    ++exp2;
  }
  const unsigned long long bits = sign | (static_cast<unsigned long long>(exp2 + 1023) << 52) |
                                  (mant & ((1ull << 52) - 1));
  return __longlong_as_double(static_cast<long long>(bits));
}

struct LaneAcc {
  long long sum;   // sum of policy tags seen by this lane for the current trajectory
  unsigned cnt;    // number of policy tokens
  unsigned maxp1;  // max over policy tokens of (unsigned)v + 1 (0 if none)
};

__device__ __forceinline__ void acc_elem(LaneAcc& a, int32_t v, bool in_range) {
  const bool in = in_range && (v != -1);
  a.sum += in ? static_cast<long long>(v) : 0ll;
  a.cnt += in ? 1u : 0u;
  const unsigned vp1 = static_cast<unsigned>(v) + 1u;
  a.maxp1 = (in && vp1 > a.maxp1) ? vp1 : a.maxp1;
}

// The stream's per-trajectory totals, written without atomics (so nothing has
// to be zeroed before a call).  The warp holding a trajectory's first token
// writes its slot with one 16-byte store: x = the sum of its part's policy tags
// with bit 63 set when the trajectory continues past that warp's range (the sum
// of valid tags is below 2^63), y = count | (max tag + 1) << 32.  Every warp
// writes one head slot: its part of the trajectory that began before its range
// (traj = -1 if none).  A continuing trajectory's totals are its slot plus the
// head slots of the following warps up to the one holding its last token.
constexpr unsigned long long kContinues = 1ull << 63;

struct HeadSlot {
  long long traj;
  unsigned long long sum;
  unsigned cnt, maxp1;
  long long pad;
};

struct TagTotals {
  ulonglong2* slot;  // [n_traj]
  HeadSlot* head;    // [stream warps]
};

// Geometry of one tag-reduction launch: warp w streams batches
// [n_batches w / n_warps, n_batches (w + 1) / n_warps).
struct StreamGeom {
  int64_t n_batches;
  int64_t n_warps;
};

// The last warp whose range starts at or before batch b (the one that streams it).
__host__ __device__ __forceinline__ int64_t warp_of_batch(const StreamGeom& g, int64_t b) {
  return ((b + 1) * g.n_warps - 1) / g.n_batches;
}

// Warp-reduce the lane partials and write them: the head slot of this warp, or
// trajectory traj's slot.  Integer adds and max are order-independent, so the
// totals are exact and deterministic however trajectories are split.
__device__ __forceinline__ void emit(LaneAcc& a, int64_t traj, bool continues, bool head,
                                     int64_t warp, const TagTotals& tt) {
  const unsigned full = 0xffffffffu;
  // the lanes' 64-bit sums in three digits of 26, 26 and 12 bits, each a 32-bit warp
  // reduction that cannot overflow (the top one wraps like the 64-bit sum would)
  const unsigned long long u = static_cast<unsigned long long>(a.sum);
  const unsigned d0 = __reduce_add_sync(full, static_cast<unsigned>(u) & 0x3ffffffu);
  const unsigned d1 = __reduce_add_sync(full, static_cast<unsigned>(u >> 26) & 0x3ffffffu);
  const unsigned d2 = __reduce_add_sync(full, static_cast<unsigned>(u >> 52));
  const unsigned long long s = d0 + (static_cast<unsigned long long>(d1) << 26) +
                               (static_cast<unsigned long long>(d2) << 52);
  const unsigned c = __reduce_add_sync(full, a.cnt);
  const unsigned m = __reduce_max_sync(full, a.maxp1);
  if ((threadIdx.x & 31) == 0) {
    if (head) {
      HeadSlot h;
      h.traj = traj;
      h.sum = s;
      h.cnt = c;
      h.maxp1 = m;
      h.pad = 0;
      tt.head[warp] = h;
    } else {
      ulonglong2 v;
      v.x = s | (continues ? kContinues : 0ull);
      v.y = static_cast<unsigned long long>(c) | (static_cast<unsigned long long>(m) << 32);
      tt.slot[traj] = v;
    }
  }
  a.sum = 0;
  a.cnt = 0;
  a.maxp1 = 0;
}

// Trajectory i's totals (T, the exact sum of its policy tags, the largest tag
// + 1) from its slot v and the head slots, given its offsets o0, o1.  Empty (or
// inconsistent) ranges have zero totals (their slot, loaded regardless so that
// the load need not wait for the offsets, is not used).  The head slots of a continuing
// trajectory are loaded two at a time before either is used.  L2 loads: other
// blocks of the same launch may have written the slots.
__device__ __forceinline__ void traj_totals(const TagTotals& tt, const StreamGeom& g,
                                            int64_t n_tokens, int64_t i, int64_t o0, int64_t o1,
                                            const ulonglong2& v, long long& sum, unsigned& cnt,
                                            unsigned& maxp1) {
  sum = 0;
  cnt = 0u;
  maxp1 = 0u;
  if (o0 < 0 || o1 <= o0 || o0 >= n_tokens) return;
  sum = static_cast<long long>(v.x & ~kContinues);
  cnt = static_cast<unsigned>(v.y);
  maxp1 = static_cast<unsigned>(v.y >> 32);
  if (v.x & kContinues) {
    const int64_t last = (o1 < n_tokens ? o1 : n_tokens) - 1;
    const int64_t w0 = warp_of_batch(g, o0 / kBatchTokens);
    const int64_t w1 = warp_of_batch(g, last / kBatchTokens);
    for (int64_t w = w0 + 1; w <= w1; w += 2) {
      longlong2 h0[2], h1[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (w + u <= w1) {
          const longlong2* hp = reinterpret_cast<const longlong2*>(tt.head + w + u);
          h0[u] = __ldcg(hp);
          h1[u] = __ldcg(hp + 1);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (w + u <= w1 && h0[u].x == i) {
          sum += h0[u].y;
          cnt += static_cast<unsigned>(h1[u].x);
          const unsigned m = static_cast<unsigned>(static_cast<unsigned long long>(h1[u].x) >> 32);
          maxp1 = m > maxp1 ? m : maxp1;
        }
      }
    }
  }
}

// The stream is integer-ALU heavy (a few operations per 4-byte tag), so the
// common cases avoid per-element work: a tag is a policy tag below 2^26 exactly
// when none of its bits 26..31 is set, so one OR over a group of tags decides
// whether the whole group is (no tool tag -1, nothing negative or huge), and
// then up to 32 of them fit a 32-bit sum; 3-input max (DPX) halves the max tree.
__device__ __forceinline__ bool small_policy(int bits_or) {
  return (static_cast<unsigned>(bits_or) >> 26) == 0u;
}

// Sum, count and max of a batch that lies inside one trajectory and holds only
// policy tags below 2^26.  Returns false (and leaves acc untouched) when the
// batch needs the per-group path.
__device__ __forceinline__ bool acc_batch_fast(LaneAcc& a, const int4 (&v)[kTiles]) {
  int o = 0, mx = 0, s = 0;
#pragma unroll
  for (int u = 0; u < kTiles; ++u) {
    o |= (v[u].x | v[u].y) | (v[u].z | v[u].w);
    mx = __vimax3_s32(__vimax3_s32(mx, v[u].x, v[u].y), v[u].z, v[u].w);
    s += (v[u].x + v[u].y) + (v[u].z + v[u].w);
  }
  if (!small_policy(o)) return false;
  a.sum += s;
  a.cnt += 4 * kTiles;
  const unsigned mp1 = static_cast<unsigned>(mx) + 1u;
  a.maxp1 = mp1 > a.maxp1 ? mp1 : a.maxp1;
  return true;
}

// The four tags of one lane's int4, all inside the current trajectory.
__device__ __forceinline__ void acc_group(LaneAcc& a, const int4& q) {
  if (small_policy((q.x | q.y) | (q.z | q.w))) {
    a.sum += (q.x + q.y) + (q.z + q.w);
    a.cnt += 4u;
    const unsigned mp1 = static_cast<unsigned>(__vimax3_s32(q.x, q.y, max(q.z, q.w))) + 1u;
    a.maxp1 = mp1 > a.maxp1 ? mp1 : a.maxp1;
  } else {
    acc_elem(a, q.x, true);
    acc_elem(a, q.y, true);
    acc_elem(a, q.z, true);
    acc_elem(a, q.w, true);
  }
}

// phi_gamma(q) of Eq. 10 with integer gamma, powers by repeated
// multiplication, every operation rounded once (no FMA).
__device__ __forceinline__ double sharpen(double q, int gamma) {
  const double omq = __dsub_rn(1.0, q);
  double a = q, b = omq;
  for (int g = 1; g < gamma; ++g) {
    a = __dmul_rn(a, q);
    b = __dmul_rn(b, omq);
  }
  return __ddiv_rn(a, __dadd_rn(a, b));
}

// The prefix-score window's preparation, done by extra blocks of the tag
// reduction's launch (the blocks after its streaming blocks): they are
// scheduled as the streaming blocks retire, so the preparation runs in the
// reduction's ragged tail instead of as a launch of its own.  Every prep block
// tabulates F[c] = phi_gamma(c / n) for kPrepPerBlock of c = 0..n and puts as many
// window values in their places of the ascending order, each by counting the values
// before it (ties by index), so that neither the table's fp64 divisions nor the order
// wait for one SM.  A bitonic sort by one block (45 to 78 steps behind barriers) held
// short streams' launches open: whole calls (graph replay) 20k trajectories with a window
// of 777 65.0 and now 62.2 us, 32k with 4,096 91.5 and 65.7 (128 values a block 79.1, 64
// 69.9), 128k with 4,096 303 and 284, 300k 378 and 364, 16k with 512 52.9 both.  NaN in the window is a data error.
constexpr int kPrepPerBlock = 32;
constexpr int kPrepParts = kReduceThreads / kPrepPerBlock;  // threads a value, each for a
                                                            // part of the window

struct WindowPrep {
  const float* window;  // null: no preparation blocks
  int n;
  int gamma;
  float* sorted;        // [n]
  double* f_table;      // [n + 1]
  int32_t* status;
};

inline unsigned window_prep_blocks(int64_t n) {
  return static_cast<unsigned>((n + 1 + kPrepPerBlock - 1) / kPrepPerBlock);
}

inline size_t window_prep_smem(int64_t n) {
  return static_cast<size_t>((n + 3) / 4 * 4) * sizeof(float);
}

// The values of sw[a, b) (both multiples of 4) that lie before v.
template <bool kOrEqual>
__device__ __forceinline__ int count_before(const float* sw, int a, int b, float v) {
  int c = 0;
#pragma unroll 4
  for (int k = a; k < b; k += 4) {
    const float4 y = *reinterpret_cast<const float4*>(sw + k);
    c += kOrEqual ? (y.x <= v) + (y.y <= v) + (y.z <= v) + (y.w <= v)
                  : (y.x < v) + (y.y < v) + (y.z < v) + (y.w < v);
  }
  return c;
}

__device__ void window_prep_block(int b, const WindowPrep& w) {
  extern __shared__ __align__(16) float sw[];  // the window, padded with +inf to a multiple of 4
  __shared__ int s_rank[kPrepParts][kPrepPerBlock];
  const int n = w.n, n4 = (n + 3) & ~3;
  for (int k = threadIdx.x; k < n4; k += blockDim.x) {
    float v = k < n ? w.window[k] : __int_as_float(0x7f800000);
    if (isnan(v)) {
      report(w.status, PACE_ERR_NAN_INPUT);
      v = __int_as_float(0x7f800000);
    }
    sw[k] = v;
  }
  __syncthreads();
  const int e = static_cast<int>(threadIdx.x) % kPrepPerBlock;
  const int part = static_cast<int>(threadIdx.x) / kPrepPerBlock;
  const int c0 = b * kPrepPerBlock, i = c0 + e;  // value i, table entry i
  const int per = (n4 / 4 + kPrepParts - 1) / kPrepParts * 4;
  const int from = min(part * per, n4), to = min(from + per, n4);
  int rank = 0;
  if (i < n) {
    const float v = sw[i];
    rank = count_before<true>(sw, from, min(to, c0), v);  // equal ones of lower index: before
    for (int k = max(from, c0); k < min(to, c0 + kPrepPerBlock); ++k)
      rank += sw[k] < v || (sw[k] == v && k < i);
    rank += count_before<false>(sw, max(from, c0 + kPrepPerBlock), to, v);
  }
  s_rank[part][e] = rank;
  __syncthreads();
  if (part == 0 && i < n) {
#pragma unroll
    for (int q = 1; q < kPrepParts; ++q) rank += s_rank[q][e];
    w.sorted[rank] = sw[i];
  } else if (part == 1 && i <= n) {
    w.f_table[i] = sharpen(__ddiv_rn(static_cast<double>(i), static_cast<double>(n)), w.gamma);
  }
}

// Each warp owns a contiguous range of batches (kTiles x 128 tokens) of
// the flattened tag stream and walks the CSR offsets forward through it, so trajectories of
// any length mix are balanced across warps.  The walk never leaves
// [0, n_traj) and loads only tags[0, n_tokens), whatever the offsets hold;
// inconsistent offsets are reported by the finalize kernel.
//
// One warp's share of the stream (every warp of the first n_stream_blocks
// blocks calls it; it returns early when the range is empty or the offsets end
// before the tokens do).
__device__ __forceinline__ void stream_warp_range(const int32_t* __restrict__ tags,
                                                  const int64_t* __restrict__ offsets,
                                                  int64_t n_traj, int64_t n_tokens,
                                                  const TagTotals& tt, int n_stream_blocks) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = (static_cast<int64_t>(n_stream_blocks) * blockDim.x) >> 5;
  const int64_t n_batches = (n_tokens + kBatchTokens - 1) / kBatchTokens;
  const int64_t b_begin = n_batches * warp / n_warps;
  const int64_t b_end = n_batches * (warp + 1) / n_warps;
  if (b_begin >= b_end) {  // no tokens: no head part either
    if (lane == 0) tt.head[warp].traj = -1;
    return;
  }
  const int64_t t_begin = b_begin * kBatchTokens;
  const int64_t t_end = b_end * kBatchTokens < n_tokens ? b_end * kBatchTokens : n_tokens;

  // Start the stream before the search below: the warp's first batches are
  // requested into L2 while the offsets are searched (lanes 0.., one batch each).
  if (lane < kFirstBatches) {
    const int64_t pf = b_begin + lane;
    if (pf < b_end && (pf + 1) * kBatchTokens <= n_tokens)
      l2_prefetch_bulk(tags + pf * kBatchTokens, static_cast<uint32_t>(kBatchTokens * 4));
  }

  // trajectory holding token t_begin: the largest i in [1, n_traj) with
  // offsets[i] <= t_begin, else 0.  A 32-way search: the lanes probe 32 points of
  // [lo, hi) at once and a ballot keeps the sub-range after the last probe that
  // is <= t_begin (4 rounds for a million trajectories instead of 20 dependent
  // loads).  Whatever the offsets hold, lo stays in [0, n_traj).
  int64_t lo = 0, hi = n_traj;
  while (hi - lo > 1) {
    const int64_t span = hi - lo;
    const int64_t q = lo + 1 + ((span - 1) * lane) / 32;  // in [lo + 1, hi - 1], nondecreasing
    const unsigned bal = __ballot_sync(0xffffffffu, offsets[q] <= t_begin);
    if (bal == 0u) {
      hi = lo + 1;
    } else {
      const int j = 31 - __clz(bal);
      const int64_t qj = lo + 1 + ((span - 1) * j) / 32;
      hi = j < 31 ? lo + 1 + ((span - 1) * (j + 1)) / 32 : hi;
      lo = qj;
    }
  }
  // Positions from here on are relative to the range (32 bits: a warp's share of the
  // tags that fit a GPU's memory is far below 2^31), ends past it clamped.
  const int len = static_cast<int>(t_end - t_begin);
  const int32_t* base = tags + t_begin;
  auto rel = [&](int64_t o) -> int {
    const int64_t d = o - t_begin;
    return d > len + 1 ? len + 1 : (d < 0 ? 0 : static_cast<int>(d));
  };
  int64_t cur = lo;
  // the first trajectory began before this range: this warp's part of it is its
  // head slot; otherwise the head slot says there is none
  const bool head_open = offsets[cur] < t_begin;
  bool cur_here = offsets[cur] < t_end;  // the current trajectory begins before t_end
  int cur_end = rel(offsets[cur + 1]);
  if (!head_open && lane == 0) tt.head[warp].traj = -1;
  LaneAcc acc{0, 0u, 0u};
  constexpr int kBatch = static_cast<int>(kBatchTokens);

  auto load_batch = [&](int4 (&v)[kTiles], int at) {
    if (at + kBatch <= len) {
#pragma unroll
      for (int u = 0; u < kTiles; ++u)
        v[u] = ld_stream_v4(base + at + u * kTileTokens + lane * 4);
    } else {
#pragma unroll
      for (int u = 0; u < kTiles; ++u) {
        const int t = at + u * kTileTokens + lane * 4;
        v[u].x = (t + 0 < len) ? base[t + 0] : -1;
        v[u].y = (t + 1 < len) ? base[t + 1] : -1;
        v[u].z = (t + 2 < len) ? base[t + 2] : -1;
        v[u].w = (t + 3 < len) ? base[t + 3] : -1;
      }
    }
  };

  // Adds the batch at `at` to the running trajectory sums; false when the offsets end
  // before the tokens do (inconsistent offsets: stop).
  auto process = [&](const int4 (&v)[kTiles], int at) -> bool {
    const int end = at + kBatch < len ? at + kBatch : len;
    int pos = at;
    while (true) {
      const int seg_hi = cur_end < end ? cur_end : end;
      if (pos == at && seg_hi == at + kBatch) {
        // whole batch inside one trajectory: no position tests
        if (!acc_batch_fast(acc, v)) {
#pragma unroll
          for (int u = 0; u < kTiles; ++u) acc_group(acc, v[u]);
        }
      } else if (seg_hi > pos) {
        // the bounds are the same in every lane, so whole 128-token tiles outside
        // [lo_r, hi_r) are skipped and tiles inside it need no position tests
        const int lo_r = pos - at, hi_r = seg_hi - at;
#pragma unroll
        for (int u = 0; u < kTiles; ++u) {
          const int t0 = u * kTileTokens;
          if (t0 + kTileTokens <= lo_r || t0 >= hi_r) continue;
          if (t0 >= lo_r && t0 + kTileTokens <= hi_r) {
            acc_group(acc, v[u]);
          } else {
            const int t = t0 + lane * 4;
            acc_elem(acc, v[u].x, t + 0 >= lo_r && t + 0 < hi_r);
            acc_elem(acc, v[u].y, t + 1 >= lo_r && t + 1 < hi_r);
            acc_elem(acc, v[u].z, t + 2 >= lo_r && t + 2 < hi_r);
            acc_elem(acc, v[u].w, t + 3 >= lo_r && t + 3 < hi_r);
          }
        }
      }
      if (cur_end > end) return true;  // trajectory continues into the next batch
      emit(acc, cur, false, head_open && cur == lo, warp, tt);
      if (seg_hi > pos) pos = seg_hi;
      ++cur;
      if (cur >= n_traj) return false;  // tokens past the last trajectory: offsets are bad
      cur_here = cur_end < len;
      cur_end = rel(offsets[cur + 1]);
      // the next trajectory starts at the batch edge: continue in the next batch;
      // otherwise loop (more of this batch, or empty trajectories to step over)
      if (pos >= end && cur_end > end) return true;
    }
  };

  // two register sets: the next batch's loads are in flight while one is added up
  int4 va[kTiles], vb[kTiles];
  int at = 0;
  load_batch(va, at);
  while (true) {
    if (at + kBatch < len) load_batch(vb, at + kBatch);
    if (!process(va, at)) return;
    at += kBatch;
    if (at >= len) break;
    if (at + kBatch < len) load_batch(va, at + kBatch);
    if (!process(vb, at)) return;
    at += kBatch;
    if (at >= len) break;
  }
  // the trajectory still open continues past this range (one that begins at
  // t_end belongs to the next warp)
  if (cur < n_traj && cur_here) emit(acc, cur, true, head_open && cur == lo, warp, tt);
}

struct FinalizeArgs {
  const int64_t* offsets;
  const int32_t* c_version;
  const float* s_pre;
  const float* window_sorted;   // ascending, window_len values (with window_ready)
  const double* f_table;        // F for counts 0..window_len (with window_ready)
  TagTotals tt;
  StreamGeom geom;
  int64_t n_traj;
  int64_t n_tokens;
  int32_t j;
  int32_t window_len;
  int32_t window_ready;
  int32_t mode;
  int32_t group_size;
  double inv_group;             // 1 / G for G a power of two (exact), else 0
  double f_missing;
  double* kgen;
  double* kwait;
  double* weight;
  double* score;
  double* unit_score;
  int32_t* status;
};

// Shared memory of one finalisation pass: the sorted window (padded to a multiple of
// 4 floats), the F table and the scores of the pass's trajectories.
struct FinalizeSmem {
  float* swin;
  double* ftab;    // [window_len + 1]
  double* sscore;  // [tpb]
};

__host__ __device__ inline size_t finalize_smem_bytes(int64_t window_len, int tpb) {
  return align_up(static_cast<size_t>((window_len + 3) & ~3) * sizeof(float), 16) +
         static_cast<size_t>(window_len + 1) * sizeof(double) +
         static_cast<size_t>(tpb) * sizeof(double);
}

__device__ __forceinline__ FinalizeSmem finalize_smem(unsigned char* raw, int window_len) {
  FinalizeSmem m;
  const int wpad = (window_len + 3) & ~3;
  m.swin = reinterpret_cast<float*>(raw);
  m.ftab = reinterpret_cast<double*>(raw + align_up(wpad * sizeof(float), 16));
  m.sscore = m.ftab + window_len + 1;
  return m;
}

// The sorted window and the F table into shared memory, four loads of each per thread in
// flight at a time.  L2 loads: another block of the same launch may have written them.
// Every thread of the block calls it.
__device__ void finalize_load_window(const FinalizeArgs& p, const FinalizeSmem& m) {
  if (p.window_ready) {
    const int tlen = p.window_len + 1;
    const int nb = static_cast<int>(blockDim.x);
    for (int k0 = threadIdx.x; k0 < tlen; k0 += 4 * nb) {
      float w[4];
      double f[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = k0 + j * nb;
        w[j] = k < p.window_len ? __ldcg(p.window_sorted + k) : 0.0f;
        f[j] = k < tlen ? __ldcg(p.f_table + k) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = k0 + j * nb;
        if (k < p.window_len) m.swin[k] = w[j];
        if (k < tlen) m.ftab[k] = f[j];
      }
    }
  }
  __syncthreads();
}

// What one thread of a pass reads for its trajectory: the inputs (loadable any
// time) and the stream's totals from the slots (only once the stream blocks that
// hold its tokens are done).
struct TrajIn {
  float s;
  int32_t c;
  int64_t o0, o1;
  ulonglong2 slot;
  unsigned long long sum;
  unsigned cnt, maxp1;
};

__device__ __forceinline__ void load_traj_inputs(const FinalizeArgs& p, int64_t i0, int64_t i_end,
                                                 int tpb, TrajIn& in) {
  const int tid = static_cast<int>(threadIdx.x);
  const int64_t i = i0 + tid;
  if (tid < tpb && i < i_end) {
    in.s = p.s_pre ? p.s_pre[i] : __int_as_float(0x7fc00000);
    in.c = p.c_version[i];
    in.o0 = p.offsets[i];
    in.o1 = p.offsets[i + 1];
  }
}

// The stream's slot of this thread's trajectory (issue it early: its load need
// not wait for anything), then the totals (which may load head slots).
__device__ __forceinline__ void load_traj_slot(const FinalizeArgs& p, int64_t i0, int64_t i_end,
                                               int tpb, TrajIn& in) {
  const int tid = static_cast<int>(threadIdx.x);
  const int64_t i = i0 + tid;
  if (tid < tpb && i < i_end) in.slot = __ldcg(p.tt.slot + i);
}

__device__ __forceinline__ void load_traj_acc(const FinalizeArgs& p, int64_t i0, int64_t i_end,
                                              int tpb, TrajIn& in) {
  const int tid = static_cast<int>(threadIdx.x);
  const int64_t i = i0 + tid;
  if (tid < tpb && i < i_end) {
    long long sum;
    traj_totals(p.tt, p.geom, p.n_tokens, i, in.o0, in.o1, in.slot, sum, in.cnt, in.maxp1);
    in.sum = static_cast<unsigned long long>(sum);
  }
}

// One pass over trajectories [i0, i0 + tpb) clipped to i_end (i0 and tpb whole
// groups), from what load_traj_inputs and load_traj_acc read: threads t < tpb do
// trajectory i0 + t, then consecutive threads the groups' means in fixed left-to-right
// order.  Every thread of the block calls it.
__device__ void finalize_pass(const FinalizeArgs& p, int64_t i0, int64_t i_end, int tpb,
                              const FinalizeSmem& m, const TrajIn& in) {
  const int tid = static_cast<int>(threadIdx.x);
  const int64_t i = i0 + tid;
  if (tid < tpb && i < i_end) {
    const float s = in.s;
    const int64_t o0 = in.o0, o1 = in.o1;
    if (o1 < o0 || (i == 0 && o0 != 0) || (i == p.n_traj - 1 && o1 != p.n_tokens))
      report(p.status, PACE_ERR_INVALID_ARG);
    const int64_t c = in.c;
    const unsigned t_count = in.cnt;
    const unsigned mp1 = in.maxp1;
    const long long tag_sum = static_cast<long long>(in.sum);
    if (c < 0 || mp1 >= 0x80000000u) report(p.status, PACE_ERR_INVALID_ARG);
    if (c > p.j || (mp1 != 0u && static_cast<int64_t>(mp1) - 1 > c))
      report(p.status, PACE_ERR_VERSION_ORDER);
    // Lemma 1: K_gen = (1/T) sum (c - v_t) = (c T - sum v_t) / T, exact integers
    const long long gen_sum = static_cast<long long>(c) * static_cast<long long>(t_count) - tag_sum;
    // the correctly rounded K_gen and K_wait
    const double kgen = t_count > 0u ? __ddiv_rn(__ll2double_rn(gen_sum), __uint2double_rn(t_count))
                                     : 0.0;
    const double kwait = __ll2double_rn(static_cast<long long>(p.j) - c);
    double f;
    if (!p.window_ready) {
      f = 1.0;
    } else if (isnan(s)) {
      f = p.f_missing;
    } else {
      // count of window values <= s: the first index of the sorted window
      // holding a value > s
      int lo = 0, hi = p.window_len;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (m.swin[mid] <= s) lo = mid + 1;
        else hi = mid;
      }
      f = m.ftab[lo];
    }
    double sc;
    if (p.mode == PACE_SCORE_EFF) sc = __dadd_rn(kwait, __dmul_rn(f, kgen));
    else if (p.mode == PACE_SCORE_RAW) sc = __dadd_rn(kwait, kgen);
    else sc = __dmul_rn(f, kgen);
    if (p.kgen) p.kgen[i] = kgen;
    if (p.kwait) p.kwait[i] = kwait;
    if (p.weight) p.weight[i] = f;
    p.score[i] = sc;
    m.sscore[tid] = sc;
  }
  __syncthreads();
  // The groups' means, a thread per group, the groups in consecutive threads: a chain of
  // G additions holds the narrow fp64 pipe for as many warps as have a group, which with
  // the first thread of each group working was every warp (half of the kernel's time).
  // With the pipe free of them, K_gen's quotient is faster in fp64 than from integer
  // divisions: whole calls (graph replay) 1k pool 24.6 -> 23.7 us, 16k 62.8 -> 61.9, 20k in
  // groups of 12 73.3 -> 72.6, 128k 319.9 -> 317.9, 1M 2229 -> 2214.
  const int G = p.group_size;
  if (p.unit_score) {
    const int64_t n = i_end - i0 < tpb ? i_end - i0 : tpb;  // whole groups
    const int units = static_cast<int>(n) / G;
    for (int u = tid; u < units; u += static_cast<int>(blockDim.x)) {
      const double* s = m.sscore + u * G;
      double acc = 0.0;
      for (int g = 0; g < G; ++g) acc = __dadd_rn(acc, s[g]);
      // for G = 2^m, acc * 2^-m is the same correctly rounded value as acc / G
      // (2^-m is exact), one multiplication instead of a division
      p.unit_score[i0 / G + u] = p.inv_group != 0.0 ? __dmul_rn(acc, p.inv_group)
                                                    : __ddiv_rn(acc, static_cast<double>(G));
    }
  }
}

// The finalisation as a launch of its own: blockDim.x trajectories (whole groups) per
// block.
__global__ void score_finalize_kernel(FinalizeArgs p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tpb = static_cast<int>(blockDim.x);
  const FinalizeSmem m = finalize_smem(smem_raw, p.window_len);
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * tpb;
  // the inputs, the slot and the window are in flight together; the head slots
  // of continuing trajectories are loaded once the window is in place
  TrajIn in;
  load_traj_inputs(p, i0, p.n_traj, tpb, in);
  load_traj_slot(p, i0, p.n_traj, tpb, in);
  finalize_load_window(p, m);
  load_traj_acc(p, i0, p.n_traj, tpb, in);
  finalize_pass(p, i0, p.n_traj, tpb, m, in);
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The finalisation inside the tag reduction's launch (groups of at most 256).
// The launch is cooperative, so all its blocks are resident at once and every
// wait below ends as soon as the blocks it waits for have streamed their share.
struct FusedFinalize {
  unsigned* done;       // [stream blocks] set once a block's warps have all streamed; null: off
  unsigned* ticket;     // counts the blocks that have finished streaming
  unsigned* prep_done;  // counts the finished preparation tasks
  int prep_tasks;       // parts of the sorted window and the F table (0: no window)
  int tpb;              // trajectories per finalisation pass
  WindowPrep prep;
  FinalizeArgs fin;
};

// Run by every block once its own warps have streamed: publish that, take a
// finishing ticket (the first finishers, idle in the reduction's ragged tail,
// run the window's preparation tasks: each sorts in 32 values of W and tabulates
// F for 32 counts), then finalise this block's slice of the groups,
// [U b / S, U (b + 1) / S), once the stream blocks covering those groups'
// tokens and the preparation are done.  Each block thus finalises in the tail
// as soon as its neighbourhood of the stream is complete, and no launch of its
// own is needed.
__device__ __forceinline__ void fused_finalize(const int64_t* __restrict__ offsets,
                                               int64_t n_tokens, int n_stream_blocks,
                                               const FusedFinalize& fz) {
  __shared__ unsigned s_ticket;
  const int tid = static_cast<int>(threadIdx.x);
  const int S = n_stream_blocks;
  const int64_t blk = blockIdx.x;
  __threadfence();  // this thread's slot stores before the block's flag
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    atomicAdd(fz.done + blk, 1u);
    s_ticket = atomicAdd(fz.ticket, 1u);
  }
  __syncthreads();
  for (unsigned task = s_ticket; task < static_cast<unsigned>(fz.prep_tasks);
       task += static_cast<unsigned>(S)) {
    window_prep_block(static_cast<int>(task), fz.prep);
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(fz.prep_done, 1u);
  }

  const FinalizeArgs& p = fz.fin;
  const int G = p.group_size;
  const int64_t U = p.n_traj / G;
  const int64_t u_lo = U * blk / S, u_hi = U * (blk + 1) / S;
  if (u_lo >= u_hi) return;
  const int64_t i_lo = u_lo * G, i_hi = u_hi * G;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const FinalizeSmem m = finalize_smem(smem_raw, p.window_len);
  // the first pass's inputs are in flight while the waits below run
  TrajIn cur;
  load_traj_inputs(p, i_lo, i_hi, fz.tpb, cur);
  if (tid < 32) {
    const int lane = tid;
    // stream blocks holding the tokens of trajectories [i_lo, i_hi): the warp of
    // batch b is the last w with n_batches * w / n_warps <= b
    int64_t b_lo = 0, b_hi = -1;
    int64_t t0 = offsets[i_lo], t1 = offsets[i_hi];
    t0 = t0 < 0 ? 0 : (t0 > n_tokens ? n_tokens : t0);
    t1 = t1 < 0 ? 0 : (t1 > n_tokens ? n_tokens : t1);
    if (t1 < t0) {  // inconsistent offsets (reported by the pass): wait for every block
      b_hi = S - 1;
    } else if (t1 > t0) {
      const StreamGeom& g = p.geom;
      b_lo = warp_of_batch(g, t0 / kBatchTokens) / (kReduceThreads / 32);
      b_hi = warp_of_batch(g, (t1 - 1) / kBatchTokens) / (kReduceThreads / 32);
    }
    bool ok = true;
    const uint64_t start = global_timer_ns();
    for (int64_t b = b_lo + lane; ok && b <= b_hi; b += 32) {
      while (ld_acquire_u32(fz.done + b) == 0u) {
        if (global_timer_ns() - start > kWaitLimitNs) {
          ok = false;
          break;
        }
        __nanosleep(64);
      }
    }
    if (lane == 0 && fz.prep_tasks > 0) {
      while (ok && ld_acquire_u32(fz.prep_done) < static_cast<unsigned>(fz.prep_tasks)) {
        if (global_timer_ns() - start > kWaitLimitNs) ok = false;
        else __nanosleep(64);
      }
    }
    if (!__all_sync(0xffffffffu, ok) && lane == 0) report(p.status, PACE_ERR_TIMEOUT);
  }
  __syncthreads();
  load_traj_slot(p, i_lo, i_hi, fz.tpb, cur);
  finalize_load_window(p, m);
  load_traj_acc(p, i_lo, i_hi, fz.tpb, cur);
  for (int64_t i0 = i_lo; i0 < i_hi; i0 += fz.tpb) {
    // the next pass's reads are in flight while this pass computes
    TrajIn nxt;
    const int64_t i1 = i0 + fz.tpb;
    if (i1 < i_hi) {
      load_traj_inputs(p, i1, i_hi, fz.tpb, nxt);
      load_traj_slot(p, i1, i_hi, fz.tpb, nxt);
      load_traj_acc(p, i1, i_hi, fz.tpb, nxt);
    }
    finalize_pass(p, i0, i_hi, fz.tpb, m, cur);
    __syncthreads();  // the pass's shared scores and counts are reused
    cur = nxt;
  }
}

template <bool kFused>
__global__ void __launch_bounds__(kReduceThreads, kBlocksPerSm)
    tag_reduce_kernel(const int32_t* __restrict__ tags, const int64_t* __restrict__ offsets,
                      int64_t n_traj, int64_t n_tokens, TagTotals tt, int n_stream_blocks,
                      WindowPrep prep, FusedFinalize fz) {
  if (static_cast<int>(blockIdx.x) >= n_stream_blocks) {  // the window's preparation
    window_prep_block(static_cast<int>(blockIdx.x) - n_stream_blocks, prep);
    return;
  }
  stream_warp_range(tags, offsets, n_traj, n_tokens, tt, n_stream_blocks);
  if (kFused) fused_finalize(offsets, n_tokens, n_stream_blocks, fz);
}

// Stale-k admission (Sec. 2): kbar = sum (j - v_t) / T = (j T - sum v_t) / T in
// exact integers, one rounding; admitted when kbar <= k_max.
__global__ void stale_k_kernel(const int64_t* __restrict__ offsets, TagTotals tt, StreamGeom geom,
                               int64_t n_traj, int64_t n_tokens, int32_t j, double k_max,
                               double* __restrict__ kbar, uint8_t* __restrict__ admitted,
                               int32_t* status) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n_traj) return;
  const int64_t o0 = offsets[i], o1 = offsets[i + 1];
  if (o1 < o0 || (i == 0 && o0 != 0) || (i == n_traj - 1 && o1 != n_tokens))
    report(status, PACE_ERR_INVALID_ARG);
  long long tag_sum;
  unsigned t_count, mp1;
  traj_totals(tt, geom, n_tokens, i, o0, o1, __ldcg(tt.slot + i), tag_sum, t_count, mp1);
  if (mp1 >= 0x80000000u) report(status, PACE_ERR_INVALID_ARG);
  if (mp1 != 0u && static_cast<int64_t>(mp1) - 1 > j) report(status, PACE_ERR_VERSION_ORDER);
  const long long lag_sum = static_cast<long long>(j) * static_cast<long long>(t_count) - tag_sum;
  const double kb = t_count > 0u ? i64_div_u32_rn(lag_sum, t_count) : 0.0;
  if (kbar) kbar[i] = kb;
  admitted[i] = kb <= k_max ? 1 : 0;
}

// Stream blocks of one launch at most (one wave: SMs x resident blocks per SM).
constexpr int kMaxStreamBlocks = 2048;

struct ScoreWs {
  TagTotals tt;     // slots [n_traj], head slots [kMaxStreamBlocks x 8 warps]
  unsigned* flags;  // [2 + kMaxStreamBlocks]: ticket, preparation count, stream blocks done
};

struct WindowWs {
  float* sorted;    // [window_len]
  double* f_table;  // [window_len + 1]
};

WindowWs carve_window_ws(Carver& cv, int64_t window_len) {
  WindowWs w;
  w.sorted = cv.take<float>(static_cast<size_t>(window_len > 0 ? window_len : 1));
  w.f_table = cv.take<double>(static_cast<size_t>(window_len + 1));
  return w;
}

ScoreWs carve_score_ws(Carver& cv, int64_t n_traj) {
  ScoreWs w;
  w.tt.slot = cv.take<ulonglong2>(static_cast<size_t>(n_traj));
  w.tt.head = cv.take<HeadSlot>(static_cast<size_t>(kMaxStreamBlocks) * (kReduceThreads / 32));
  w.flags = cv.take<unsigned>(2 + kMaxStreamBlocks);
  return w;
}

// The two kernels that hold the sorted window and the F table are allowed the shared
// memory of the largest window once per device, whatever window a call has: a limit set
// per call could be lowered by another thread between its setting and the launch.
// (Below kPlainSmem no permission is needed, the kernels' static shared memory included.)
constexpr size_t kPlainSmem = 40 * 1024;

pace_status allow_window_smem() {
  constexpr int kMaxDevices = 64;
  static bool done[kMaxDevices] = {};
  static std::mutex mu;
  int dev = 0;
  PACE_TRY_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return PACE_ERR_CUDA;
  std::lock_guard<std::mutex> g(mu);
  if (done[dev]) return PACE_OK;
  PACE_TRY_CUDA(cudaFuncSetAttribute(score_finalize_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(finalize_smem_bytes(kMaxWindow, 1024))));
  PACE_TRY_CUDA(cudaFuncSetAttribute(
      tag_reduce_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      static_cast<int>(finalize_smem_bytes(kMaxWindow, kReduceThreads))));
  done[dev] = true;
  return PACE_OK;
}

// Resident blocks per SM of the fused tag reduction with the given dynamic shared
// memory (cached per device and size).
pace_status reduce_blocks_per_sm(size_t smem, int* out) {
  constexpr int kMaxDevices = 64;
  static int cache[kMaxDevices] = {};
  static size_t cache_smem[kMaxDevices] = {};
  static std::mutex mu;
  int dev = 0;
  PACE_TRY_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> g(mu);
  if (dev >= 0 && dev < kMaxDevices && cache[dev] > 0 && cache_smem[dev] == smem) {
    *out = cache[dev];
    return PACE_OK;
  }
  int nb = 0;
  PACE_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, tag_reduce_kernel<true>,
                                                              kReduceThreads, smem));
  if (dev >= 0 && dev < kMaxDevices) {
    cache[dev] = nb;
    cache_smem[dev] = smem;
  }
  *out = nb;
  return PACE_OK;
}

pace_status launch_tag_reduce(unsigned grid, size_t smem, bool fused, cudaStream_t st,
                              const int32_t* tags, const int64_t* offsets, int64_t n_traj,
                              int64_t n_tokens, const ScoreWs& ws, int stream_blocks,
                              const WindowPrep& prep, const FusedFinalize& fz) {
  if (!fused) {
    tag_reduce_kernel<false><<<grid, kReduceThreads, smem, st>>>(
        tags, offsets, n_traj, n_tokens, ws.tt, stream_blocks, prep, fz);
    return last_launch_status();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kReduceThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  PACE_TRY_CUDA(cudaLaunchKernelEx(&cfg, tag_reduce_kernel<true>, tags, offsets, n_traj, n_tokens,
                                   ws.tt, stream_blocks, prep, fz));
  return last_launch_status();
}

// Stream the tags once into the slots (nothing to zero first).  With
// prep.window set, the same launch also sorts the window and tabulates F
// (extra blocks, run in the stream's tail).  With `fused` (fz.done is filled in
// here, its flags zeroed), the launch is cooperative and also finalises every
// trajectory and group (fused_finalize): one wave of stream blocks, at least
// one block even for an empty stream.  *geom receives the launch's geometry.
pace_status run_tag_reduce(const int32_t* tags, const int64_t* offsets, int64_t n_traj,
                           int64_t n_tokens, const ScoreWs& ws, const WindowPrep& prep,
                           FusedFinalize fz, bool fused, size_t fused_smem, StreamGeom* geom,
                           cudaStream_t st) {
  const unsigned prep_blocks = (prep.window && !fused) ? window_prep_blocks(prep.n) : 0u;
  size_t smem = prep_blocks ? window_prep_smem(prep.n) : 0;
  if (fused) smem = fused_smem;
  int per_sm = kBlocksPerSm;
  if (fused) {
    if (smem > kPlainSmem) PACE_TRY(allow_window_smem());
    int nb = 0;
    PACE_TRY(reduce_blocks_per_sm(smem, &nb));
    if (nb < 1) return PACE_ERR_UNSUPPORTED_SHAPE;
    per_sm = nb < per_sm ? nb : per_sm;
  }
  const int64_t n_batches = (n_tokens + kBatchTokens - 1) / kBatchTokens;
  const int warps_per_block = kReduceThreads / 32;
  const int64_t per_block = warps_per_block * kMinBatchesPerWarp;
  int64_t blocks = (n_batches + per_block - 1) / per_block;
  int64_t cap = static_cast<int64_t>(sm_count()) * per_sm;  // one wave
  if (cap > kMaxStreamBlocks) cap = kMaxStreamBlocks;
  // A large window's preparation blocks would wait for a short stream's blocks to retire and
  // then be waited for, so they get room in the wave.  Calls (graph replay) without and with
  // room, window 4,096: 4,096 trajectories 23.9 and 18.9 us, 8,184 26.8 and 22.4; window
  // 2,048: 18.3 and 15.4, 20.4 and 20.2.  Not for windows of 1,024 (8,184 18.3 / 19.1), nor
  // for longer streams (20,000 with 24 batches a warp and window 2,048 33.0 / 35.1) or
  // trajectories shorter than a batch (65,536 of 136 tags, window 4,096 35.0 / 39.3).
  if (prep_blocks >= kRoomPrepBlocks && 2 * static_cast<int64_t>(prep_blocks) < cap &&
      n_batches <= cap * warps_per_block * kRoomBatches && n_traj <= n_batches)
    cap -= prep_blocks;
  if (blocks > cap) blocks = cap;
  if (fused && blocks < 1) blocks = 1;
  geom->n_batches = n_batches;
  geom->n_warps = blocks * warps_per_block;
  if (blocks == 0 && prep_blocks == 0) return PACE_OK;
  if (fused) {
    PACE_TRY_CUDA(cudaMemsetAsync(ws.flags, 0, static_cast<size_t>(2 + blocks) * sizeof(unsigned),
                                  st));
    fz.ticket = ws.flags;
    fz.prep_done = ws.flags + 1;
    fz.done = ws.flags + 2;
    fz.fin.geom = *geom;
  } else {
    fz = FusedFinalize{};
  }
  const unsigned grid = static_cast<unsigned>(blocks) + prep_blocks;
  const int stream_blocks = static_cast<int>(blocks);
  const ProfileEvents& pe = profile_events(PACE_PROFILE_TAG_REDUCE);
  if (pe.begin) PACE_TRY_CUDA(cudaEventRecord(pe.begin, st));
  PACE_TRY(launch_tag_reduce(grid, smem, fused, st, tags, offsets, n_traj, n_tokens, ws,
                             stream_blocks, prep, fz));
  if (pe.end) PACE_TRY_CUDA(cudaEventRecord(pe.end, st));
  return PACE_OK;
}

}  // namespace
}  // namespace pace

using namespace pace;

extern "C" size_t pace_stale_k_workspace_size(int64_t n_traj) {
  return pace_score_pool_workspace_size(n_traj, 0);
}

extern "C" pace_status pace_stale_k(const int32_t* tags, const int64_t* offsets, int64_t n_traj,
                                    int64_t n_tokens, int32_t trainer_version, double k_max,
                                    double* kbar, uint8_t* admitted, void* workspace,
                                    size_t workspace_bytes, int32_t* status_dev, void* stream) {
  if (n_traj < 0 || n_tokens < 0 || n_traj > (int64_t(1) << 31)) return PACE_ERR_INVALID_ARG;
  if (n_traj > 0 && (!offsets || !admitted)) return PACE_ERR_INVALID_ARG;
  if (n_tokens > 0 && !tags) return PACE_ERR_INVALID_ARG;
  if (isnan(k_max)) return PACE_ERR_INVALID_ARG;
  if (tags && !aligned(tags, 16)) return PACE_ERR_UNSUPPORTED_SHAPE;
  if (n_traj == 0) return n_tokens == 0 ? PACE_OK : PACE_ERR_INVALID_ARG;
  if (!workspace || !aligned(workspace, 256)) return PACE_ERR_WORKSPACE;
  Carver cv(workspace, workspace_bytes);
  ScoreWs ws = carve_score_ws(cv, n_traj);
  if (!cv.fits()) return PACE_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  StreamGeom geom{};
  PACE_TRY(run_tag_reduce(tags, offsets, n_traj, n_tokens, ws, WindowPrep{}, FusedFinalize{},
                          false, 0, &geom, st));
  const int threads = 256;
  stale_k_kernel<<<static_cast<unsigned>((n_traj + threads - 1) / threads), threads, 0, st>>>(
      offsets, ws.tt, geom, n_traj, n_tokens, trainer_version, k_max, kbar,
      admitted, status_dev);
  return last_launch_status();
}

extern "C" pace_status pace_set_score_fused_min_traj(int64_t min_traj) {
  if (min_traj < 0) return PACE_ERR_INVALID_ARG;
  fused_min_traj().store(min_traj == 0 ? 0 : min_traj);
  return PACE_OK;
}

extern "C" int64_t pace_score_fused_min_traj_default(void) { return kFusedMinTrajDefault; }

extern "C" void pace_score_params_default(PaceScoreParams* p) {
  if (!p) return;
  p->mode = PACE_SCORE_EFF;
  p->gamma = 4;
  p->min_obs = 32;
  p->group_size = 8;
  p->f_missing = 1.0;
}

extern "C" size_t pace_score_pool_workspace_size(int64_t n_traj, int64_t window_len) {
  if (n_traj < 0 || window_len < 0) return 0;
  Carver cv;
  carve_score_ws(cv, n_traj);
  carve_window_ws(cv, window_len);
  return cv.used;
}

extern "C" pace_status pace_score_pool(const int32_t* tags, const int64_t* offsets,
                                       const int32_t* c_version, const float* s_pre,
                                       int64_t n_traj, int64_t n_tokens, int32_t trainer_version,
                                       const float* window, int64_t window_len,
                                       const PaceScoreParams* params, double* kgen,
                                       double* kwait, double* weight, double* score,
                                       double* unit_score, void* workspace,
                                       size_t workspace_bytes, int32_t* status_dev,
                                       void* stream) {
  if (!params) return PACE_ERR_INVALID_ARG;
  if (n_traj < 0 || n_tokens < 0 || n_traj > (int64_t(1) << 31)) return PACE_ERR_INVALID_ARG;
  if (n_traj > 0 && (!offsets || !c_version || !score)) return PACE_ERR_INVALID_ARG;
  if (n_tokens > 0 && !tags) return PACE_ERR_INVALID_ARG;
  const int G = params->group_size;
  if (G < 1 || G > 1024 || n_traj % G != 0) return PACE_ERR_INVALID_ARG;
  if (params->gamma < 1 || params->gamma > 64) return PACE_ERR_INVALID_ARG;
  if (params->mode != PACE_SCORE_EFF && params->mode != PACE_SCORE_RAW &&
      params->mode != PACE_SCORE_GEN)
    return PACE_ERR_INVALID_ARG;
  if (window_len < 0 || window_len > kMaxWindow) return PACE_ERR_UNSUPPORTED_SHAPE;
  if (window_len > 0 && !window) return PACE_ERR_INVALID_ARG;
  if (tags && !aligned(tags, 16)) return PACE_ERR_UNSUPPORTED_SHAPE;
  if (n_traj == 0) return n_tokens == 0 ? PACE_OK : PACE_ERR_INVALID_ARG;
  if (!workspace || !aligned(workspace, 256)) return PACE_ERR_WORKSPACE;
  Carver cv(workspace, workspace_bytes);
  ScoreWs ws = carve_score_ws(cv, n_traj);
  WindowWs wws = carve_window_ws(cv, window_len);
  if (!cv.fits()) return PACE_ERR_WORKSPACE;

  cudaStream_t st = as_stream(stream);
  const bool window_ready = window_len > 0 && window_len >= params->min_obs;
  // With the sorted window and the F table the finalisation takes one binary
  // search and one table read per trajectory; their preparation runs inside the
  // tag reduction's launch.  (Small pools counted against the raw window instead, eight
  // threads a trajectory, while one block sorted it; whole calls by graph replay that way
  // and now: 64 trajectories 17.8 and 16.4 us, 1,024 22.6 and 21.2, 4,096 28.8 and 27.8,
  // 2,048 with a window of 4,096 34.9 and 31.5, 6,000 with 1,024 32.8 and 31.3.)
  WindowPrep prep{};
  if (window_ready) {
    prep.window = window;
    prep.n = static_cast<int>(window_len);
    prep.gamma = params->gamma;
    prep.sorted = wws.sorted;
    prep.f_table = wws.f_table;
    prep.status = status_dev;
  }
  FinalizeArgs a;
  a.offsets = offsets;
  a.c_version = c_version;
  a.s_pre = s_pre;
  a.window_sorted = wws.sorted;
  a.f_table = wws.f_table;
  a.tt = ws.tt;
  a.geom = StreamGeom{};
  a.n_traj = n_traj;
  a.n_tokens = n_tokens;
  a.j = trainer_version;
  a.window_len = window_ready ? static_cast<int32_t>(window_len) : 0;
  a.window_ready = window_ready ? 1 : 0;
  a.mode = params->mode;
  a.group_size = G;
  a.inv_group = (G & (G - 1)) == 0 ? 1.0 / static_cast<double>(G) : 0.0;
  a.f_missing = params->f_missing;
  a.kgen = kgen;
  a.kwait = kwait;
  a.weight = weight;
  a.score = score;
  a.unit_score = unit_score;
  a.status = status_dev;

  if (G <= kReduceThreads && n_traj >= fused_min_traj().load() && cooperative_launch_ok()) {
    // Large pools whose groups fit one block: the finalisation runs inside the
    // tag reduction's launch, each stream block finalising its slice of the
    // groups in the stream's ragged tail.  The chain after the last stream block
    // (flags, waits, one pass) costs more than a launch of its own (16k 55.2 against
    // 51.8 us per call, 128k 282.8 / 278.7), on large pools hardly more (1M 2142 /
    // 2138), where it saves the launch.  Passes
    // of whole groups over the block's 256 threads.
    FusedFinalize fz{};
    fz.tpb = (kReduceThreads / G) * G;
    fz.fin = a;
    if (window_ready) {
      fz.prep = prep;
      fz.prep_tasks = static_cast<int>(window_prep_blocks(prep.n));
    }
    const size_t smem = finalize_smem_bytes(a.window_len, fz.tpb);  // at least the preparation's
    StreamGeom geom{};
    return run_tag_reduce(tags, offsets, n_traj, n_tokens, ws, WindowPrep{}, fz, true, smem, &geom,
                          st);
  }

  PACE_TRY(run_tag_reduce(tags, offsets, n_traj, n_tokens, ws, prep, FusedFinalize{}, false, 0,
                          &a.geom, st));
  // A launch of its own: whole groups per block, one thread per trajectory.  With the
  // window, 256 threads per block, so that one round of loads brings it and the F table
  // into shared memory; without, about 64, so that the little fp64 work left is spread
  // over more SMs.
  const int max_units = G >= 256 ? 1 : 256 / G;
  const int64_t n_units = n_traj / G;
  const int64_t spread = 2 * static_cast<int64_t>(sm_count());
  const int min_units = window_ready ? max_units : (G >= 64 ? 1 : (64 + G - 1) / G);
  int64_t want = (n_units + spread - 1) / spread;
  want = want < min_units ? min_units : want;
  const int tpb = (want > max_units ? max_units : static_cast<int>(want)) * G;
  const int64_t blocks = (n_traj + tpb - 1) / tpb;
  const size_t smem = finalize_smem_bytes(a.window_len, tpb);
  if (smem > kPlainSmem) PACE_TRY(allow_window_smem());
  score_finalize_kernel<<<static_cast<unsigned>(blocks), tpb, smem, st>>>(a);
  return last_launch_status();
}

namespace pace {
namespace {

// Both constructions of the same doubles, side by side (the self-test below).
__global__ void div_selftest_kernel(const long long* __restrict__ S,
                                    const unsigned* __restrict__ T, int64_t n,
                                    double* __restrict__ q_int, double* __restrict__ q_fp64,
                                    double* __restrict__ c_int, double* __restrict__ c_fp64) {
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    q_int[i] = i64_div_u32_rn(S[i], T[i]);
    q_fp64[i] = __ddiv_rn(__ll2double_rn(S[i]), __ull2double_rn(T[i]));
    c_int[i] = i64_div_u32_rn(S[i], 1u);
    c_fp64[i] = __ll2double_rn(S[i]);
  }
}

}  // namespace
}  // namespace pace

extern "C" pace_status pace_div_selftest(const int64_t* S, const uint32_t* T, int64_t n,
                                         double* q_int, double* q_fp64, double* c_int,
                                         double* c_fp64, void* stream) {
  if (n < 0 || (n > 0 && (!S || !T || !q_int || !q_fp64 || !c_int || !c_fp64)))
    return PACE_ERR_INVALID_ARG;
  if (n == 0) return PACE_OK;
  pace::div_selftest_kernel<<<static_cast<unsigned>(n < 4096 ? (n + 255) / 256 : 16 * pace::sm_count()),
                              256, 0, pace::as_stream(stream)>>>(
      reinterpret_cast<const long long*>(S), reinterpret_cast<const unsigned*>(T), n, q_int,
      q_fp64, c_int, c_fp64);
  return pace::last_launch_status();
}
