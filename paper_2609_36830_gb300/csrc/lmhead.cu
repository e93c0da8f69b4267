// Fused LM head: per-token log-probabilities under the current policy
// (Sec. 2: the policy factorises over tokens, log pi_theta(y_t | x, y_<t);
// training temperature from the shared settings), without writing logits.
//
// lmhead_lse_kernel (sm_103a, persistent CTA pairs, one CTA per SM, 192
// threads, warp-specialised, tcgen05 on the pair):
//   warp 0            TMA producer, in both CTAs: per K step the CTA's own
//                     128x64 hidden tile and its own half (128x64) of the pair's
//                     256x64 vocabulary tile, into its own 4-stage shared-memory
//                     ring (128-byte swizzle), as one TMA instruction of lanes
//                     0..n (lane 0 the vocabulary half-tile, lanes 1..n the n
//                     boxes of the hidden tile); each CTA arrives on the even
//                     CTA's full barrier with its own bytes.  Contiguous rows:
//                     one 128-row box.  Rows in the loss a subset (mask,
//                     rejected groups, fewer than 128 rows): the hidden tile is
//                     read straight from the caller's hidden-state tensor
//                     through the compact-row index.  Per work item the warp
//                     splits the block's 128 rows into runs of consecutive
//                     source rows (plan_block_loads) and the runs into boxes
//                     (Boxes; one for a block inside a response; the first and
//                     last of several runs, rounded up to one box, spill into
//                     16 KB regions around the tile).  A block of more than 31 boxes is
//                     fetched by four-row TMA gathers (tile::gather4), one per
//                     lane.  No copy of the rows is made.
//   warp 1 / lane 0   MMA issuer, even CTA only: tcgen05.mma.cta_group::2
//                     kind::f16 (bf16 x bf16 -> fp32), M=256 (128 rows from each
//                     CTA), N=256 (128 vocabulary rows from each CTA), K=16 per
//                     instruction; each CTA's tensor memory receives its own
//                     128x256 logit tile; two accumulators (512 TMEM columns)
//                     so the epilogue of tile n overlaps the MMAs of tile n+1.
//   warps 2..5        epilogue, in both CTAs: each thread owns one row (one
//                     TMEM lane), reads its 256 logits 32 columns at a time
//                     with tcgen05.ld, keeps a running base-2 max and sum of
//                     exponentials (online log-sum-exp) and picks out the
//                     target's logit.
// No operand is multicast: every CTA reads only its own tiles; the pair shares
// the vocabulary tile through the 2-CTA MMA itself.
// Work is cut in two (lm_plan, evaluated on the device from the rows actually
// present).  Rounds: an item is a pair of 128-row blocks (one per CTA of the
// cluster) and one of S contiguous vocabulary splits, and every round gives each
// cluster one item; consecutive items share a row pair, so the hidden tiles re-read
// for every vocabulary tile stay in L2 while the vocabulary streams.  Tail: the
// row pairs that would not fill a last round (all of them in a small batch) are
// dealt to the clusters tile by tile (TailSpan), so that every cluster gets the
// same number of tiles, give or take one, and all of them walk the vocabulary
// together.  Each CTA writes one (max, sum) pair per row and split (rounds) or per
// row and cluster that shares the row (tail).  A soft
// barrier at item boundaries (wait_round) keeps the clusters of a split
// together, so each vocabulary tile is fetched from DRAM about once per round:
// left alone, the clusters' small speed differences add up over the hundreds
// of rounds of a long launch, the leaders fetch tiles from DRAM that the
// laggards fetch again later, and the extra DRAM traffic costs the
// power-capped SMs their clock (a 1.01M-row launch of the 7B head read the
// vocabulary 8.7 times per round; paced, 1.02 times).
//
// lse_merge_kernel: per row, merges its partial pairs into the log-sum-exp
//   and writes lp = z_y / tau - lse.
//
// Every mbarrier wait is bounded (2 s); on timeout the CTA reports
// PACE_ERR_TIMEOUT, tells its peer to stop, waits (bounded) for its in-flight
// copies and MMAs, frees its tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "pace_internal.cuh"
#include "pace_loss.cuh"
#include "pace_tma.cuh"

namespace pace {
namespace {

constexpr int BM = 128;                         // rows per CTA; the pair's MMA covers 256
constexpr int BN = 256;                         // vocabulary rows per MMA tile (both CTAs)
constexpr int BK = 64;
constexpr int STAGES = 4;
constexpr int CLUSTER = 2;                      // the CTA pair of one 2-CTA MMA
constexpr int kThreads = 192;
constexpr uint32_t kStageA = BM * BK * 2;       // 16 KB: this CTA's 128 hidden rows
constexpr uint32_t kStageB = BN / CLUSTER * BK * 2;  // 16 KB: this CTA's half of the vocabulary tile
constexpr uint32_t kTmemCols = 2 * BN;          // two fp32 accumulators of 256 columns
constexpr uint32_t kIdesc = idesc_bf16_f32(CLUSTER * BM, BN);
// Shared memory: the hidden tiles, each with a 16 KB spill region before and
// after it (shared by neighbours: spill | A0 | spill | A1 | ... | A3 | spill),
// so a 128-row box may start up to 127 rows before or after its tile's first
// row; then the vocabulary tiles; then barriers and flags (256 bytes) and, for
// rows read by index, the block's source rows (int32 [128]) and its planned
// loads (int2 [128]).
constexpr uint32_t kSpill = kStageA;
constexpr uint32_t kARegion = kSpill + STAGES * (kStageA + kSpill);
constexpr uint32_t kMiscBytes = 256 + BM * 4 + BM * 8;
constexpr size_t kSmemBytes =
    1024 /* alignment slack */ + kARegion + STAGES * kStageB + kMiscBytes;
__host__ __device__ constexpr uint32_t a_tile_off(uint32_t s) {
  return kSpill + s * (kStageA + kSpill);
}
__host__ __device__ constexpr uint32_t b_tile_off(uint32_t s) { return kARegion + s * kStageB; }
// Tensor maps of the hidden states with boxes of several heights (64 columns, 128-byte
// swizzle).  An SM takes in operand tiles at close to the rate the tensor cores use
// them, so the rows a block's boxes load beyond its 128 cost their share of time, and
// so do its boxes: with every block cut alike (19,456 rows, H 2048, V 151,936) one and
// two boxes run at 1934 TFLOP/s, three at 1896, four at 1770, eight at 1344.
//   Fine: 1, 2, ..., 128 rows, so every run is one box.  128 maps take 3.6 us of host
//     time to encode and 16 KB of kernel parameters, so for large launches only
//     (kFineFlops).
//   Coarse: 1, 2, 4, 8, 16, 24, ..., 128 rows: the first and last run of a block are one
//     box each, of at most 7 rows more than they have; a run in between takes up to four.
// One launch, coarse and fine: 2,582 rows of eight sequences (H 2048 head) 1050 and 963
// us where a block has three runs, 37k rows of multi-turn sequences (H 3584) 24.0 and
// 23.5 ms; powers of two only were 7-12 % slower still on micro-batches.
template <bool kFine>
struct Boxes {
  static constexpr int kLevels = kFine ? 128 : 19;
  __host__ __device__ static constexpr int rows(int level) {
    return kFine ? level + 1 : (level < 3 ? 1 << level : 8 * (level - 2));
  }
  // the lowest box of at least n rows, the tallest of at most n (n in 1..128)
  __host__ __device__ static constexpr int covering(int n) {
    return kFine || n <= 2 ? n - 1 : (n <= 4 ? 2 : 2 + (n + 7) / 8);
  }
  __host__ __device__ static constexpr int within(int n) {
    return kFine ? n - 1 : (n >= 8 ? 2 + n / 8 : (n >= 4 ? 2 : (n >= 2 ? 1 : 0)));
  }
};
static_assert(Boxes<false>::rows(18) == BM && Boxes<true>::rows(127) == BM,
              "the tallest box is a block");
constexpr int kMaxBoxes = 31;  // more boxes in a block: four-row gathers instead
constexpr double kFineFlops = 4e11;  // about 200 us
template <bool kFine>
struct AMaps {
  CUtensorMap box[Boxes<kFine>::kLevels];  // box[j]: Boxes::rows(j) rows
};
constexpr int kMaxSplits = 8;
constexpr int kMaxClusters = 76;  // clusters launched at most (bounds the tail's partials)

// How row_pairs row pairs over n_vtiles vocabulary tiles are dealt to n_clusters
// persistent clusters.
//
// Rounds: the first `rounds_rp` row pairs in items of (row pair, one of S
// contiguous splits of tiles_per_split tiles), as many as make whole rounds of one
// item per cluster.  With S = 4 the 19 clusters sweeping one split stay close
// enough for L2 to serve each vocabulary tile to all of them; S = 2 is 2-10 %
// faster on some GPUs and as much slower on others (the power-capped clock), S = 1
// far slower, so a preferred count (pace_set_lmhead_splits, from a measurement on
// this GPU) replaces 4 when it still gives every cluster at least four items.  A
// vocabulary of so few tiles that 4 splits are over 5 % uneven takes 2 or 1.
//
// Tail: the other row pairs, fewer than n_clusters, whose tiles are dealt one by
// one (TailSpan).  Split into equal items instead (the best of 2, 3, 4, 6 and 8
// splits), they left part of the chip idle in the last round; with the tail, one
// launch on the H 2048 / V 151,936 head went from 866 to 276 us on 290 rows, 1016 to
// 967 on 2,582 (rows of one run a block) and 4060 to 3650-3760 on 10,589, and from
// 1260 to 1178 us on 20,506 rows of H 1024 / V 50,001.  Dealing every batch of fewer
// than n_clusters pairs this way (no rounds at all) is as fast up to about 40 pairs
// but 17 % slower on 57 pairs of the H 3584 head, where the 76 clusters drift apart
// over the vocabulary (9.1 against 10.6 ms), so whole rounds come first.
//
// Evaluated identically by the LM head and the merge, from the device-side count.
struct LmPlan {
  int64_t rounds_rp;
  int splits, tiles_per_split;
  int tail_rp;     // row pairs of the tail, 0 .. n_clusters - 1
  int tail_slots;  // partials per row of the tail: clusters that may share its tiles
};

__host__ __device__ inline LmPlan lm_plan(int64_t row_pairs, int n_clusters, int n_vtiles,
                                          int pref) {
  LmPlan p;
  int sp = 4;
  if (pref > 0 && row_pairs * (pref < n_vtiles ? pref : n_vtiles) >= 4 * int64_t{n_clusters}) {
    sp = pref < n_vtiles ? pref : n_vtiles;
  } else {
    while (sp > 1 && (n_vtiles + sp - 1) / sp * sp * 20 > n_vtiles * 21) sp /= 2;
  }
  int g = n_clusters, r = sp;  // gcd
  while (r) {
    const int q = g % r;
    g = r;
    r = q;
  }
  const int64_t unit = n_clusters / g;  // row pairs of the smallest whole number of rounds
  p.splits = sp;
  p.tiles_per_split = (n_vtiles + sp - 1) / sp;
  p.rounds_rp = row_pairs / unit * unit;
  p.tail_rp = static_cast<int>(row_pairs - p.rounds_rp);
  p.tail_slots = p.tail_rp ? n_clusters / p.tail_rp + 2 : 0;
  return p;
}

// The tail's tiles of one cluster.  Row pair i of R covers [i C, (i + 1) C) of a
// line and cluster c of C the stretch [c R, (c + 1) R) of it, so a cluster shares
// at most two row pairs (R < C) and a row pair at most C / R + 2 clusters.  Tile t
// of row pair i sits at i C + (t R mod C): successive tiles step from cluster to
// cluster, every cluster gets floor or ceil of the mean number of tiles, its k-th
// tile is tile k C / R to within one, whatever its row pairs (so all clusters walk
// the vocabulary together and each tile is fetched from DRAM once), and no tile
// number comes to it twice.
struct TailSpan {
  int R, C;
  int rp;    // first of its row pairs (of the tail's)
  int a0;    // its stretch starts at rp * C + a0
  bool two;  // the stretch reaches into row pair rp + 1
  __device__ TailSpan(int tail_rp, int n_clusters, int c) : R(tail_rp), C(n_clusters) {
    const int64_t x = static_cast<int64_t>(c) * R;
    rp = static_cast<int>(x / C);
    a0 = static_cast<int>(x - static_cast<int64_t>(rp) * C);
    two = a0 + R > C;
  }
  // y = t R mod C, advanced by step() from tile to tile; 0 or 1: tile t of row
  // pair rp or rp + 1 is this cluster's; -1: no tile t is
  __device__ int which(int y) const {
    return y >= a0 && y < a0 + R ? 0 : (y < a0 + R - C ? 1 : -1);
  }
  __device__ int step(int y) const {
    y += R;
    return y >= C ? y - C : y;
  }
};

// First cluster that shares row pair i of the tail (its slot is 0).
__device__ __forceinline__ int tail_first_cluster(int i, int tail_rp, int n_clusters) {
  return static_cast<int>(static_cast<int64_t>(i) * n_clusters / tail_rp);
}

struct LmArgs {
  int64_t rows_cap;             // rows of the A tensor map
  const long long* n_valid_dev; // rows actually present (device), or null = rows_cap
  int32_t H, V;
  int32_t n_vtiles;
  int32_t split_pref;           // preferred vocabulary splits, 0 = automatic
  float scale_log2;             // log2(e) / temperature
  const int32_t* targets;
  const int32_t* rowidx;        // compact row -> original row, or null (identity)
  int32_t gather;               // 1: rows read by index (rowidx), in planned boxes
  int32_t max_level;            // largest box level no taller than the hidden-state tensor
  float* part_m;                // the rounds' rows: row r's splits at r * S; then the
  float* part_s;                // tail's rows, tail_slots each
  float* tgt_logit;             // [rows_cap]
  unsigned* round_ctr;          // pacing counter, zero at launch (or null: no pacing)
  int32_t* status;
};

__device__ __forceinline__ uint64_t make_policy_evict_normal() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// One cluster's work in order: its items of the rounds (taken round-robin by the
// persistent clusters, so all of them sweep their splits in step), then its share
// of the tail.  The two CTAs of a cluster take the two 128-row blocks of a row pair
// and sweep the same vocabulary tiles, each loading its half of every 256-row tile.
// A segment's tiles are those of [tile0, tile1) for which tile() says 0 or 1 (of
// which of its row pairs); tile() is called once for each of them, in order.
struct Segments {
  const LmPlan& w;
  const TailSpan& span;
  int n_vtiles;
  int64_t item, n_items;
  int n_clusters;
  bool is_tail;  // the current segment is the tail's
  int64_t rp;    // its first row pair
  int split, tile0, tile1;
  int y;
  __device__ Segments(const LmPlan& w_, const TailSpan& s_, int nt, int cid, int nc)
      : w(w_), span(s_), n_vtiles(nt), item(cid), n_items(w_.rounds_rp * w_.splits),
        n_clusters(nc), is_tail(false), rp(0), split(0), tile0(0), tile1(0), y(0) {}
  // loads the current segment; false when there is none left
  __device__ bool load() {
    if (is_tail) return false;
    if (item < n_items) {
      rp = item / w.splits;
      split = static_cast<int>(item % w.splits);
      tile0 = split * w.tiles_per_split;
      tile1 = min(tile0 + w.tiles_per_split, n_vtiles);
      item += n_clusters;
      return true;
    }
    if (w.tail_rp == 0) return false;
    is_tail = true;
    rp = w.rounds_rp + span.rp;
    tile0 = 0;
    tile1 = n_vtiles;
    return true;
  }
  __device__ bool two() const { return is_tail && span.two; }
  __device__ int tile() {
    if (!is_tail) return 0;
    const int r = span.which(y);
    y = span.step(y);
    return r;
  }
};

// One lane's part of a 128-row block's loads: lane 0 the vocabulary half-tile,
// lanes 1..n the n boxes of the hidden tile.
struct BlockLoads {
  int n;             // boxes
  uint32_t a_bytes;  // the block's hidden-tile bytes per K step
  int32_t psrc;      // this lane's box: first source row
  int pdst, plev;    // first block row (-127..127), box level
  int32_t g4[4];     // scattered blocks: this lane's four source rows
  bool scattered;
};

// The loads of one 128-row block whose rows are read by index.  Block row r is
// compact row row0 + r; its source row is rowidx[row0 + r] while that is below
// n_valid.  A run is a maximal stretch of block rows with consecutive source
// rows; the rows past n_valid (loaded, never written back) belong to the last
// run.  A block of one run is loaded exactly, tallest boxes first (one 128-row box
// when the tensor has 128 rows or more).  Of several runs, the first is the lowest
// box that covers it, ending at the run's end (its earlier rows land in the spill
// region before the tile), the last one such box starting at the run's start (its
// later rows land in the spill region after the tile), and a run in between is
// loaded exactly.  Boxes never overlap inside the tile, and no box is taller than
// Boxes::rows(max_level) (the tallest map the hidden-state tensor allows).  Writes the source rows to row_src[BM], the boxes to piece[] as
// (first source row, (first block row + 128) | level << 9), their number to
// plan[0] and their bytes per K step to plan[1].  All 32 lanes call it.
template <bool kFine>
__device__ void plan_block_loads(const int32_t* __restrict__ rowidx, int64_t row0,
                                 int64_t n_valid, int max_level, int lane, int32_t* row_src,
                                 int2* piece, volatile int* plan) {
  const int64_t left = n_valid - row0;
  const int r_inv = left <= 0 ? 0 : (left >= BM ? BM : static_cast<int>(left));
  int32_t v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = 32 * j + lane;
    v[j] = r < r_inv ? rowidx[row0 + r] : 0;
  }
  uint32_t starts[4];
  uint32_t carry = 0;  // source row of the previous word's last row
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = 32 * j + lane;
    uint32_t prev = __shfl_up_sync(0xffffffffu, static_cast<uint32_t>(v[j]), 1);
    if (lane == 0) prev = carry;
    const bool st = r == 0 || (r < r_inv && static_cast<uint32_t>(v[j]) != prev + 1u);
    starts[j] = __ballot_sync(0xffffffffu, st);
    carry = __shfl_sync(0xffffffffu, static_cast<uint32_t>(v[j]), 31);
    row_src[r] = v[j];
  }
  __syncwarp();
  if (lane == 0) {
    const uint64_t lo = starts[0] | (static_cast<uint64_t>(starts[1]) << 32);
    const uint64_t hi = starts[2] | (static_cast<uint64_t>(starts[3]) << 32);
    const int m = __popcll(lo) + __popcll(hi);  // runs in the block
    int n = 0, k = 0, r = 0;
    uint32_t rows = 0;
    while (r < BM) {
      const int q = r + 1;  // the run ends at the next start at or after q (BM: none)
      const uint64_t mlo = q < 64 ? (lo & (~0ull << q)) : 0ull;
      int e;
      if (mlo) {
        e = __ffsll(static_cast<long long>(mlo)) - 1;
      } else {
        const uint64_t mhi = q < 64 ? hi : (q < BM ? (hi & (~0ull << (q - 64))) : 0ull);
        e = mhi ? 64 + __ffsll(static_cast<long long>(mhi)) - 1 : BM;
      }
      const int32_t s0 = row_src[r];
      const int len = e - r;
      const int cl = Boxes<kFine>::covering(len);
      if (m > 1 && (k == 0 || k == m - 1) && cl <= max_level) {
        // first or last of several runs: one box that covers it, ending at the
        // first run's end (spilling before the tile) or starting at the last
        // run's start (spilling after it)
        const int at = k == 0 ? len - Boxes<kFine>::rows(cl) : r;
        piece[n++] = make_int2(s0 + (at - r), (at + BM) | (cl << 9));
        rows += Boxes<kFine>::rows(cl);
      } else {  // the only run, or one in between: exactly
        int at = r, left_rows = len;
        int32_t src = s0;
        while (left_rows > 0) {
          int lev = Boxes<kFine>::within(left_rows);
          if (lev > max_level) lev = max_level;
          const int h = Boxes<kFine>::rows(lev);
          piece[n++] = make_int2(src, (at + BM) | (lev << 9));
          rows += h;
          at += h;
          src += h;
          left_rows -= h;
        }
      }
      r = e;
      ++k;
    }
    plan[0] = n;
    plan[1] = static_cast<int>(rows * (BK * 2));
  }
  __syncwarp();
}

template <bool kFine>
__global__ void __cluster_dims__(CLUSTER, 1, 1) __launch_bounds__(kThreads, 1)
    lmhead_lse_kernel(const __grid_constant__ AMaps<kFine> am, const __grid_constant__ CUtensorMap tm_b,
                      LmArgs p) {
  extern __shared__ unsigned char smem_raw[];
  // the same offsets in both CTAs: the pair's MMA reads each CTA's operand
  // tiles at the addresses the even CTA's descriptors name
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kARegion + STAGES * kStageB);
  uint64_t* full = bars;                     // [STAGES] even CTA: both CTAs' tiles landed
  uint64_t* empty = bars + STAGES;           // [STAGES] the pair's MMAs are done with the stage
  uint64_t* tmem_full = bars + 2 * STAGES;   // [2] this CTA's accumulator is ready
  uint64_t* tmem_empty = tmem_full + 2;      // [2] even CTA: both CTAs' epilogues drained it
  uint64_t* mma_done = tmem_empty + 2;       // [1]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* plan = reinterpret_cast<volatile int*>(tmem_slot + 2);  // [2] boxes, A bytes
  int32_t* row_src = reinterpret_cast<int32_t*>(reinterpret_cast<unsigned char*>(bars) + 256);
  int2* piece = reinterpret_cast<int2*>(row_src + BM);                            // [BM]

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t crank = cluster_ctarank();
  const bool leader = crank == 0;
  const int n_clusters = static_cast<int>(gridDim.x) / CLUSTER;
  const int cid = static_cast<int>(blockIdx.x) / CLUSTER;
  const int64_t n_valid = p.n_valid_dev ? static_cast<int64_t>(*p.n_valid_dev) : p.rows_cap;
  const int64_t row_pairs = (n_valid + 2 * BM - 1) / (2 * BM);
  const LmPlan plan_w = lm_plan(row_pairs, n_clusters, p.n_vtiles, p.split_pref);
  // every CTA reads the same n_valid: the exit is uniform, and comes before the
  // pair's collective tensor-memory allocation
  if (row_pairs == 0) return;
  const TailSpan span(plan_w.tail_rp > 0 ? plan_w.tail_rp : 1, n_clusters, cid);
  Segments seg(plan_w, span, p.n_vtiles, cid, n_clusters);  // each role walks its own copy
  const int nkb = p.H / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], CLUSTER);  // each CTA's producer arrives with its bytes
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tmem_full[b], 1);
      mbar_init(&tmem_empty[b], CLUSTER * 4);  // one arrival per epilogue warp of the pair
    }
    mbar_init(mma_done, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  cluster_sync();  // both CTAs run and their barriers exist
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();  // both CTAs' tensor memory is allocated before any MMA writes it
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t peer_abort = cluster_addr(const_cast<int*>(abort_flag), crank ^ 1u);
  // first timeout: report it, and make both CTAs of the pair stop issuing
  auto give_up = [&]() {
    if (!*abort_flag) report(p.status, PACE_ERR_TIMEOUT);
    *abort_flag = 1;
    st_cluster_u32(peer_abort, 1u);
  };

  if (warp == 0) {
    // ------------------------------------------------ TMA producer (both CTAs)
    // The whole warp produces.  Per K step one TMA instruction, issued by
    // lanes 0..n: lane 0 loads the CTA's half of the vocabulary tile, lanes
    // 1..n the n boxes of its hidden tile (one 128-row box for contiguous rows;
    // for rows read by index, the boxes plan_block_loads gives).  A block of
    // more than kMaxBoxes boxes is gathered four rows a lane instead.
    const bool gather = p.gather != 0;
    if (lane == 0) tma_prefetch_desc(&tm_b);
    if (lane == 1) tma_prefetch_desc(&am.box[Boxes<kFine>::kLevels - 1]);
    const uint64_t pol = make_policy_evict_normal();
    uint32_t it = 0;
    bool ok = true;
    unsigned round = 0;  // this cluster's items so far (the round of the current one)
    // the loads of row pair rp's block of this CTA
    auto plan_block = [&](int64_t rp, BlockLoads& bl) {
      const int64_t row0 = (rp * CLUSTER + crank) * BM;
      bl.n = 1;
      bl.a_bytes = kStageA;
      bl.psrc = static_cast<int32_t>(row0);
      bl.pdst = 0;
      bl.plev = Boxes<kFine>::kLevels - 1;
#pragma unroll
      for (int j = 0; j < 4; ++j) bl.g4[j] = 0;
      bl.scattered = false;
      if (!gather) return;
      plan_block_loads<kFine>(p.rowidx, row0, n_valid, p.max_level, lane, row_src, piece, plan);
      bl.n = plan[0];
      bl.scattered = bl.n > kMaxBoxes;
      if (!bl.scattered) {
        bl.a_bytes = static_cast<uint32_t>(plan[1]);
        if (lane >= 1 && lane <= bl.n) {
          const int2 pc = piece[lane - 1];
          bl.psrc = pc.x;
          bl.pdst = (pc.y & 0x1ff) - BM;
          bl.plev = pc.y >> 9;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) bl.g4[j] = row_src[4 * lane + j];  // row 0 past the end
      }
      __syncwarp();  // row_src and piece are rewritten by the next plan
    };
    for (; ok && seg.load(); ++round) {
      BlockLoads b0, b1;
      plan_block(seg.rp, b0);
      b1 = b0;
      if (seg.two()) plan_block(seg.rp + 1, b1);
      // every round is full, so round k (or the tail) starts once all clusters
      // issued their round k-1 loads (the even CTA paces the pair)
      if (leader && lane == 0 && round > 0 && p.round_ctr)
        wait_round(p.round_ctr, round * static_cast<unsigned>(n_clusters));
      __syncwarp();
      for (int t = seg.tile0; t < seg.tile1 && ok; ++t) {
        const int which = seg.tile();
        if (which < 0) continue;
        const BlockLoads bl = which ? b1 : b0;
        const int issuers = bl.scattered ? 1 : bl.n + 1;
        const int32_t nb = t * BN + static_cast<int32_t>(crank) * (BN / CLUSTER);
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const uint32_t s = it % STAGES;
          const uint32_t ph = (it / STAGES) & 1u;
          // one outcome for the warp
          if (!__all_sync(0xffffffffu, mbar_wait_bounded(&empty[s], ph ^ 1u, abort_flag))) {
            ok = false;
            break;
          }
          unsigned char* sa = smem + a_tile_off(s);
          unsigned char* sb = smem + b_tile_off(s);
          const uint32_t bar = cluster_addr(&full[s], 0);
          if (lane == 0) {
            // this CTA's bytes of the stage, announced with its arrival on the
            // even CTA's barrier (which completes once both CTAs' bytes land)
            if (leader)
              mbar_arrive_expect_tx(&full[s], bl.a_bytes + kStageB);
            else
              mbar_arrive_expect_tx_cluster(bar, bl.a_bytes + kStageB);
          }
          // Reconverge, so that the lanes' loads below are one TMA instruction:
          // when lane 0 comes out of the arrival alone and issues its load by
          // itself, every launch is 20-25 % slower.
          __syncwarp();
          if (lane < issuers) {
            const void* desc = lane == 0 ? static_cast<const void*>(&tm_b)
                                         : static_cast<const void*>(&am.box[bl.plev]);
            unsigned char* dst = lane == 0 ? sb : sa + bl.pdst * (BK * 2);
            tma_load_2d_pair(dst, desc, bar, kb * BK, lane == 0 ? nb : bl.psrc, pol);
          }
          if (bl.scattered)
            tma_gather4_pair(sa + lane * 4 * (BK * 2), &am.box[0], bar, kb * BK, bl.g4[0],
                             bl.g4[1], bl.g4[2], bl.g4[3], pol);
        }
      }
      if (leader && lane == 0 && ok && p.round_ctr) atomicAdd(p.round_ctr, 1u);
    }
    if (lane == 0) {
      if (!ok) give_up();
      // Drain: every copy issued must have landed before the CTA exits.  The
      // even CTA sees both CTAs' bytes (every lane's loads included) on its
      // full barriers; the odd CTA sees its stages consumed on its empty
      // barriers.  After a timeout anywhere the waits are short: copies land
      // in microseconds.
      const uint64_t lim = *abort_flag ? 1000000ull : kWaitLimitNs;
      for (uint32_t s = 0; s < STAGES && s < it; ++s) {
        const uint32_t last = it - 1 - ((it - 1 - s) % STAGES);  // last index with stage s
        if (leader)
          mbar_wait_bounded(&full[s], (last / STAGES) & 1u, nullptr, lim);
        else
          mbar_wait_bounded(&empty[s], (last / STAGES) & 1u, nullptr, lim);
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      // ------------------------------------------------ MMA issuer (even CTA)
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      while (ok && seg.load()) {
        for (int t = seg.tile0; t < seg.tile1 && ok; ++t) {
          if (seg.tile() < 0) continue;
          const uint32_t acc = tcount & 1u;
          const uint32_t acc_ph = (tcount >> 1) & 1u;
          ++tcount;
          if (!mbar_wait_bounded_cluster(&tmem_empty[acc], acc_ph ^ 1u, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + acc * BN;
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const uint32_t s = it % STAGES;
            const uint32_t ph = (it / STAGES) & 1u;
            if (!mbar_wait_bounded(&full[s], ph, abort_flag)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + a_tile_off(s));
            const uint32_t sb = smem_u32(smem + b_tile_off(s));
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              tc_mma_f16_pair(d_tmem, smem_desc_k128(sa + k * 32), smem_desc_k128(sb + k * 32),
                              kIdesc, (kb > 0 || k > 0) ? 1u : 0u);
            }
            // the stage is free in both CTAs once these MMAs have read it
            tc_commit_pair(cluster_addr(&empty[s], 0));
            tc_commit_pair(cluster_addr(&empty[s], 1));
          }
          if (!ok) break;
          tc_commit_pair(cluster_addr(&tmem_full[acc], 0));
          tc_commit_pair(cluster_addr(&tmem_full[acc], 1));
        }
      }
      if (!ok) give_up();
      // all MMAs issued by this thread complete before tensor memory is freed
      tc_commit_pair(cluster_addr(mma_done, 0));
      mbar_wait_bounded(mma_done, 0, nullptr);
    }
  } else {
    // ------------------------------------------------ epilogue (4 warps, both CTAs)
    const int quad = warp & 3;  // TMEM lanes this warp may access
    const int r_local = quad * 32 + lane;
    const float scale = p.scale_log2;
    const uint32_t empty0 = cluster_addr(&tmem_empty[0], 0);
    const uint32_t empty1 = cluster_addr(&tmem_empty[1], 0);
    uint32_t tcount = 0;
    bool ok = true;
    // a row's running state over its vocabulary tiles
    struct RowState {
      int64_t row;
      bool row_ok, have_tgt;
      int32_t y;
      float m, s, tgt;
    };
    auto start_row = [&](int64_t rp, RowState& rs) {
      rs.row = (rp * CLUSTER + crank) * BM + r_local;
      rs.row_ok = rs.row < n_valid;
      rs.y = -1;
      if (rs.row_ok) {
        const int64_t orig = p.rowidx ? static_cast<int64_t>(p.rowidx[rs.row]) : rs.row;
        rs.y = p.targets[orig];
      }
      rs.m = -INFINITY;
      rs.s = 0.0f;
      rs.tgt = 0.0f;
      rs.have_tgt = false;
    };
    auto finish_row = [&](const RowState& rs, int64_t o) {
      if (!rs.row_ok) return;
      p.part_m[o] = rs.m;
      p.part_s[o] = rs.s;
      if (rs.have_tgt) p.tgt_logit[rs.row] = rs.tgt;
    };
    while (ok && seg.load()) {
      RowState r0, r1;
      start_row(seg.rp, r0);
      r1 = r0;
      if (seg.two()) start_row(seg.rp + 1, r1);
      for (int t = seg.tile0; t < seg.tile1; ++t) {
        const int which = seg.tile();
        if (which < 0) continue;
        const uint32_t acc = tcount & 1u;
        const uint32_t acc_ph = (tcount >> 1) & 1u;
        ++tcount;
        // one outcome for the whole warp: tcgen05.ld below is warp-collective,
        // and a lane that saw the peer's abort must not leave its warp behind
        const bool got = __all_sync(0xffffffffu,
                                    mbar_wait_bounded(&tmem_full[acc], acc_ph, abort_flag));
        if (!got) {
          give_up();
          ok = false;
          break;
        }
        tc_fence_after();
        const int32_t n0 = t * BN;
        const uint32_t tbase = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + acc * BN;
        const int32_t y = which ? r1.y : r0.y;
        float m = which ? r1.m : r0.m, s = which ? r1.s : r0.s, tgt = which ? r1.tgt : r0.tgt;
        bool have_tgt = which ? r1.have_tgt : r0.have_tgt;
#pragma unroll 1
        for (int cc = 0; cc < BN; cc += 32) {
          float v[32];
          tmem_ld_32x32b_x32(tbase + cc, v);
          tmem_wait_ld();
          const int32_t col0 = n0 + cc;
          if (col0 + 32 > p.V) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (col0 + i >= p.V) v[i] = -INFINITY;
          }
          float cm = v[0];
#pragma unroll
          for (int i = 1; i < 32; ++i) cm = fmaxf(cm, v[i]);
          const float m_new = fmaxf(m, cm * scale);
          float acc_s = 0.0f;
#pragma unroll
          for (int i = 0; i < 32; ++i) acc_s += ex2_approx(fmaf(v[i], scale, -m_new));
          s = s * ex2_approx(m - m_new) + acc_s;
          m = m_new;
          const uint32_t off = static_cast<uint32_t>(y - col0);
          if (off < 32u) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (off == static_cast<uint32_t>(i)) tgt = v[i];
            have_tgt = true;
          }
        }
        // this warp is done reading the accumulator: one arrival per warp on the
        // even CTA's barrier, after every lane's loads have completed
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc ? empty1 : empty0);
        if (which) {
          r1.m = m;
          r1.s = s;
          r1.tgt = tgt;
          r1.have_tgt = have_tgt;
        } else {
          r0.m = m;
          r0.s = s;
          r0.tgt = tgt;
          r0.have_tgt = have_tgt;
        }
      }
      if (!ok) break;
      if (!seg.is_tail) {
        finish_row(r0, r0.row * plan_w.splits + seg.split);
      } else {  // a cluster that got none of a row pair's tiles writes an empty partial
        const int64_t row_base = plan_w.rounds_rp * (CLUSTER * BM);
        const int64_t base = row_base * plan_w.splits;
        const int R = plan_w.tail_rp;
        finish_row(r0, base + (r0.row - row_base) * plan_w.tail_slots + cid -
                           tail_first_cluster(span.rp, R, n_clusters));
        if (span.two)
          finish_row(r1, base + (r1.row - row_base) * plan_w.tail_slots + cid -
                             tail_first_cluster(span.rp + 1, R, n_clusters));
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA frees its tensor memory or leaves while the pair's MMAs, copies
  // or arrivals may still reach it
  cluster_sync();
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
  cluster_sync();  // the collective release is complete in both CTAs
}

// Per row in the loss: log-sum-exp from the split partials, then
// lp = z_y / tau - lse, scattered back to the original row.  Up to 78 partials a row are
// merged, so the sum keeps its additions' errors: a plain sum drops each partial below half
// a last place of the sum so far, 75 of them 4e-6 in all, where sums of 8 partials kept most.
// Where the tail's rows have more than kMergeLanes partials, as many lanes take each row:
// one thread's chain of 78 was 4 us of a call of 200 rows (H 1,024 / V 50,001 62.4 us with a
// plain sum, 65.6 with its errors, 57.9 so).  Otherwise a thread a row (9,000 rows of V 64
// 16.8 us, 17.9 with eight lanes).
constexpr int kMergeLanes = 8;
constexpr int kMergeThreads = 256;

// sum += x; the addition's error goes to err (Knuth's two-sum).
__device__ __forceinline__ void add_with_error(float& sum, float& err, float x) {
  const float t = __fadd_rn(sum, x);
  const float z = __fsub_rn(t, sum);
  err = __fadd_rn(err, __fadd_rn(__fsub_rn(sum, __fsub_rn(t, z)), __fsub_rn(x, z)));
  sum = t;
}

__global__ void __launch_bounds__(kMergeThreads)
    lse_merge_kernel(int64_t rows_cap, const long long* __restrict__ n_valid_dev, int lm_clusters,
                     int n_vtiles, int split_pref, int32_t V, float inv_temp,
                     const float* __restrict__ part_m, const float* __restrict__ part_s,
                     const float* __restrict__ tgt_logit, const int32_t* __restrict__ targets,
                     const int32_t* __restrict__ rowidx, float* __restrict__ logprob,
                     float* __restrict__ lse_out, int32_t* status) {
  const unsigned full = 0xffffffffu;
  const int64_t n_valid = n_valid_dev ? static_cast<int64_t>(*n_valid_dev) : rows_cap;
  // how the LM head dealt these rows
  const LmPlan plan = lm_plan((n_valid + 2 * BM - 1) / (2 * BM), lm_clusters, n_vtiles, split_pref);
  const int64_t tail_row0 = plan.rounds_rp * (2 * BM);
  const int64_t threads = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + (threadIdx.x & ~31u);
  const int lanes = plan.tail_slots > kMergeLanes ? kMergeLanes : 1;
  const int lane = threadIdx.x & 31, sub = lane & (lanes - 1);
  for (int64_t t = t0; t < n_valid * lanes; t += threads) {  // lanes * the warp's first row
    const int64_t r = (t + lane) / lanes;
    const bool valid = r < n_valid;
    int64_t o = r * plan.splits;
    int splits = plan.splits;
    if (r >= tail_row0) {  // the clusters whose stretch meets the row pair's
      o = tail_row0 * plan.splits + (r - tail_row0) * plan.tail_slots;
      if (valid) {
        const int i = static_cast<int>((r - tail_row0) / (2 * BM));
        const int64_t x1 = static_cast<int64_t>(i + 1) * lm_clusters - 1;
        splits = static_cast<int>(x1 / plan.tail_rp) -
                 tail_first_cluster(i, plan.tail_rp, lm_clusters) + 1;
      }
    }
    if (!valid) splits = 0;
    float mm = -INFINITY;
    for (int s = sub; s < splits; s += lanes) mm = fmaxf(mm, part_m[o + s]);
    for (int x = lanes >> 1; x > 0; x >>= 1) mm = fmaxf(mm, __shfl_xor_sync(full, mm, x));
    float ss = 0.0f, se = 0.0f;  // the sum and its additions' errors
    for (int s = sub; s < splits; s += lanes)
      add_with_error(ss, se, part_s[o + s] * ex2_approx(part_m[o + s] - mm));
    for (int x = lanes >> 1; x > 0; x >>= 1) {
      const float s2 = __shfl_xor_sync(full, ss, x);
      se = __fadd_rn(se, __shfl_xor_sync(full, se, x));
      add_with_error(ss, se, s2);
    }
    if (!valid || sub != 0) continue;
    const float lse = (mm + lg2_approx(__fadd_rn(ss, se))) * 0.69314718055994531f;
    const int64_t orig = rowidx ? static_cast<int64_t>(rowidx[r]) : r;
    const int32_t y = targets[orig];
    float lp;
    if (y < 0 || y >= V) {
      report(status, PACE_ERR_INVALID_ARG);
      lp = __int_as_float(0x7fc00000);
    } else {
      lp = tgt_logit[r] * inv_temp - lse;
    }
    logprob[orig] = lp;
    if (lse_out) lse_out[orig] = lse;
  }
}

// ---------------------------------------------------------------- host side

struct LmLaunchInfo {
  int max_clusters = 0;
};

// Tensor maps, launch of one instance.
struct LmLaunch {
  const void* hidden;
  int64_t n_rows;
  int H;
  bool compact;
  CUtensorMap tm_b;
  unsigned grid;
};
template <bool kFine>
pace_status launch_lmhead(const LmLaunch& l, LmArgs a, cudaStream_t st) {
  using B = Boxes<kFine>;
  AMaps<kFine> am;
  // boxes up to the tensor's height (at most 128 rows); taller levels repeat the
  // tallest valid map and are never used, nor are the others without a row index
  int max_level = 0;
  while (max_level + 1 < B::kLevels && B::rows(max_level + 1) <= l.n_rows) ++max_level;
  if (!l.compact && max_level != B::kLevels - 1) return PACE_ERR_INVALID_ARG;  // n_rows >= 128
  PACE_TRY(encode_bf16_2d(&am.box[max_level], l.hidden, l.n_rows, l.H, l.H, BK, B::rows(max_level)));
  for (int j = 0; j < B::kLevels; ++j) {
    if (l.compact && j < max_level)
      PACE_TRY(encode_bf16_2d(&am.box[j], l.hidden, l.n_rows, l.H, l.H, BK, B::rows(j)));
    else
      am.box[j] = am.box[max_level];
  }
  a.max_level = max_level;
  lmhead_lse_kernel<kFine><<<l.grid, kThreads, kSmemBytes, st>>>(am, l.tm_b, a);
  return last_launch_status();
}

// Dynamic shared memory opt-in and the number of 2-CTA clusters that can be
// resident at once on the current device (cached per device).
pace_status lm_launch_info(LmLaunchInfo* out) {
  constexpr int kMaxDevices = 64;
  static LmLaunchInfo info[kMaxDevices];
  static std::mutex mu;
  int dev = 0;
  PACE_TRY_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return PACE_ERR_CUDA;
  std::lock_guard<std::mutex> g(mu);
  if (info[dev].max_clusters == 0) {
    PACE_TRY_CUDA(cudaFuncSetAttribute(lmhead_lse_kernel<false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kSmemBytes)));
    PACE_TRY_CUDA(cudaFuncSetAttribute(lmhead_lse_kernel<true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(kSmemBytes)));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(sm_count()), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = CLUSTER;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, lmhead_lse_kernel<false>, &cfg) != cudaSuccess || n < 1)
      n = sm_count() / CLUSTER;
    info[dev].max_clusters = n < kMaxClusters ? n : kMaxClusters;
  }
  *out = info[dev];
  return PACE_OK;
}

}  // namespace

void carve_lm_ws(Carver& cv, int64_t n_rows, int64_t n_seq, int H, bool dense_rows,
                 LmWs* w) {
  const int64_t rows_cap = n_rows > BM ? n_rows : BM;
  carve_compact_ws(cv, n_rows, &w->cw);
  carve_surrogate_ws(cv, n_rows, n_seq, &w->sw);
  w->hidden_c =
      dense_rows ? static_cast<void*>(cv.take<uint16_t>(static_cast<size_t>(rows_cap) * H))
                 : nullptr;
  // partials: of rp row pairs, kMaxSplits a row in the rounds, and C / R + 2 a row
  // for the R row pairs of the tail
  const int64_t rp = (rows_cap + 2 * BM - 1) / (2 * BM);
  const size_t parts = 2 * BM * (kMaxClusters + static_cast<size_t>(rp) * kMaxSplits);
  w->part_m = cv.take<float>(parts);
  w->part_s = cv.take<float>(parts);
  w->tgt = cv.take<float>(static_cast<size_t>(rows_cap));
  w->round_ctr = cv.take<unsigned>(1);
}

bool lm_needs_compaction(const PaceBatch* b) {
  return b->mask || b->seq_accepted || b->n_rows < BM;
}

pace_status check_lm_args(const PaceBatch* batch, const void* hidden, const void* w_vocab,
                          const int32_t* targets, int H, int V, float temperature,
                          const float* logprob) {
  PACE_TRY(check_batch(batch));
  if (H < 64 || H > 16384 || H % 64 != 0) return PACE_ERR_UNSUPPORTED_SHAPE;
  if (V < 1 || V > (1 << 24)) return PACE_ERR_UNSUPPORTED_SHAPE;
  if (!(temperature > 0.0f) || !isfinite(temperature)) return PACE_ERR_INVALID_ARG;
  if (batch->n_rows > 0 && (!hidden || !w_vocab || !targets || !logprob))
    return PACE_ERR_INVALID_ARG;
  if (!aligned(hidden, 16) || !aligned(w_vocab, 16)) return PACE_ERR_UNSUPPORTED_SHAPE;
  return PACE_OK;
}

// Compaction, fused LM head and merge: lp (and lse) for every row in
// the batch's loss, 0 elsewhere.  When the rows are compacted, the same launches also
// compute the advantages of `adv` and clear `counter` (the caller does otherwise).
pace_status run_logprob(const PaceBatch* batch, const void* hidden, const void* w_vocab,
                        const int32_t* targets, int H, int V, float temperature, float* logprob,
                        float* lse, const LmWs& ws, const AdvJob& adv, unsigned* counter,
                        int32_t* status_dev, cudaStream_t st) {
  const int64_t n_rows = batch->n_rows;
  const bool compact = lm_needs_compaction(batch);
  const long long* n_valid_dev = nullptr;
  const int32_t* rowidx = nullptr;
  int64_t rows_cap = n_rows;
  if (compact) {
    // the LM head reads the rows in the loss through rowidx (no dense copy)
    PACE_TRY(run_compaction(batch, ws.cw, adv, counter, ws.round_ctr, logprob, lse, status_dev, st));
    n_valid_dev = ws.cw.total;
    rowidx = ws.cw.rowidx;
    rows_cap = n_rows > BM ? n_rows : BM;
  }
  if (n_rows == 0) return PACE_OK;
  const int n_vtiles = (V + BN - 1) / BN;
  LmLaunch l;
  l.hidden = hidden;
  l.n_rows = n_rows;
  l.H = H;
  l.compact = compact;
  PACE_TRY(encode_bf16_2d(&l.tm_b, w_vocab, V, H, H, BK, BN / CLUSTER));  // one CTA's half tile
  LmLaunchInfo li;
  PACE_TRY(lm_launch_info(&li));
  LmArgs a;
  a.rows_cap = rows_cap;
  a.n_valid_dev = n_valid_dev;
  a.H = H;
  a.V = V;
  a.n_vtiles = n_vtiles;
  a.split_pref = lmhead_split_pref().load();
  a.scale_log2 = 1.4426950408889634f / temperature;
  a.targets = targets;
  a.rowidx = rowidx;
  a.gather = compact ? 1 : 0;
  a.part_m = ws.part_m;
  a.part_s = ws.part_s;
  a.tgt_logit = ws.tgt;
  a.round_ctr = ws.round_ctr;
  a.status = status_dev;
  // persistent: at most one wave of 2-CTA clusters, never more clusters than the
  // rows could make tiles
  const int64_t tiles = (rows_cap + 2 * BM - 1) / (2 * BM) * n_vtiles;
  const int64_t clusters = tiles < li.max_clusters ? tiles : li.max_clusters;
  l.grid = static_cast<unsigned>(clusters * CLUSTER);
  if (!compact) PACE_TRY_CUDA(cudaMemsetAsync(ws.round_ctr, 0, sizeof(unsigned), st));
  const ProfileEvents& pe = profile_events(PACE_PROFILE_LMHEAD);
  if (pe.begin) PACE_TRY_CUDA(cudaEventRecord(pe.begin, st));
  const bool fine =
      compact && n_rows >= BM && 2.0 * H * V * static_cast<double>(n_rows) >= kFineFlops;
  PACE_TRY(fine ? launch_lmhead<true>(l, a, st) : launch_lmhead<false>(l, a, st));
  if (pe.end) PACE_TRY_CUDA(cudaEventRecord(pe.end, st));
  const int64_t per_block = kMergeThreads / kMergeLanes;
  int64_t mblocks = (rows_cap + per_block - 1) / per_block;
  const int64_t cap = static_cast<int64_t>(sm_count()) * 8;
  if (mblocks > cap) mblocks = cap;
  lse_merge_kernel<<<static_cast<unsigned>(mblocks), kMergeThreads, 0, st>>>(
      rows_cap, n_valid_dev, static_cast<int>(clusters), n_vtiles, a.split_pref, V,
      1.0f / temperature, ws.part_m, ws.part_s, ws.tgt, targets, rowidx, logprob, lse, status_dev);
  return last_launch_status();
}

}  // namespace pace

using namespace pace;

extern "C" size_t pace_token_logprob_workspace_size(int64_t n_rows, int64_t n_seq,
                                                    int32_t hidden_size, int32_t vocab_size) {
  if (n_rows < 0 || n_seq < 0 || hidden_size <= 0 || vocab_size <= 0) return 0;
  Carver cv;
  LmWs w;
  carve_lm_ws(cv, n_rows, n_seq, hidden_size, false, &w);
  return cv.used;
}

extern "C" pace_status pace_token_logprob(const PaceBatch* batch, const void* hidden,
                                          const void* w_vocab, const int32_t* targets,
                                          int32_t hidden_size, int32_t vocab_size,
                                          float temperature, float* logprob, float* lse,
                                          const PaceLossArgs* loss, void* workspace,
                                          size_t workspace_bytes, int32_t* status_dev,
                                          void* stream) {
  PACE_TRY(check_lm_args(batch, hidden, w_vocab, targets, hidden_size, vocab_size, temperature,
                         logprob));
  if (loss) PACE_TRY(check_loss_args(batch, loss));
  if (!workspace || !aligned(workspace, 256)) return PACE_ERR_WORKSPACE;
  Carver cv(workspace, workspace_bytes);
  LmWs ws;
  carve_lm_ws(cv, batch->n_rows, batch->n_seq, hidden_size, false, &ws);
  if (!cv.fits()) return PACE_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  AdvJob adv{};
  if (loss)
    adv = adv_job(loss->reward, batch->seq_accepted, batch->n_seq, loss->group_size,
                  loss->params.adv_eps, loss->params.std_unbiased,
                  loss->adv ? loss->adv : ws.sw.adv);
  PACE_TRY(run_logprob(batch, hidden, w_vocab, targets, hidden_size, vocab_size, temperature,
                       logprob, lse, ws, adv, loss ? ws.sw.counter : nullptr, status_dev, st));
  if (loss)
    PACE_TRY(run_surrogate(batch, logprob, loss, ws.sw, lm_needs_compaction(batch), status_dev,
                           st));
  return PACE_OK;
}
