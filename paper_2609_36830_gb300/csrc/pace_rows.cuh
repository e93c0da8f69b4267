// The rows of a batch walked in flat tiles: a warp takes a contiguous range of
// 256-row tiles, whatever sequences they belong to, so long and short sequences load
// the chip alike, and loads the next tile's rows while it works on one.  (With a
// block per sequence, the longest sequence's chain of dependent loads set the time:
// 80 us over 5.4M rows of 1,024 sequences, a tenth of the memory's rate.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pace_internal.cuh"

namespace pace {

constexpr int kRowTile = 256;
constexpr int kRowsPerLane = kRowTile / 32;
constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;
// Three blocks an SM (80 registers), one wave: the loss and its derivative over 5.4M
// rows took 83 us (graph replay) with a tile a warp in four waves of blocks and 66 with
// a range a warp, 58 with 32-byte accesses and each tile's terms computed once whatever
// its sequences, 55.6 without a branch per row; four blocks an SM spill (109).  Staging
// two tiles a warp in shared memory needs fewer registers and took 64 to 67.
constexpr int kRowMinBlocks = 3;
constexpr int kMaxRowBlocks = 152 * kRowMinBlocks;

// One launch over n_rows rows: block b's warp w walks `per_warp` tiles from tile
// (b * kRowWarps + w) * per_warp on.
struct RowGeom {
  int64_t n_tiles;
  int64_t per_warp;
  int blocks;
};

inline RowGeom row_geom(int64_t n_rows) {
  RowGeom g;
  g.n_tiles = (n_rows + kRowTile - 1) / kRowTile;
  const int64_t most = static_cast<int64_t>(kMaxRowBlocks) * kRowWarps;
  g.per_warp = (g.n_tiles + most - 1) / most;
  if (g.per_warp < 1) g.per_warp = 1;
  const int64_t per_block = g.per_warp * kRowWarps;
  g.blocks = static_cast<int>((g.n_tiles + per_block - 1) / per_block);
  return g;
}

// Blocks that a workspace for n_rows rows holds.  A launch's own count falls where
// per_warp steps up; this one never does, so a workspace made for the largest batch
// serves every smaller one.
inline size_t row_blocks_bound(int64_t n_rows) {
  const int64_t n_tiles = (n_rows + kRowTile - 1) / kRowTile;
  const int64_t b = (n_tiles + kRowWarps - 1) / kRowWarps;
  return static_cast<size_t>(b < 1 ? 1 : (b < kMaxRowBlocks ? b : kMaxRowBlocks));
}

// Reports offsets that do not partition the rows (any thread of a grid: sequence i).
__device__ __forceinline__ void check_seq(const int64_t* __restrict__ offsets, int64_t i,
                                          int64_t n_rows, int32_t* status) {
  const int64_t r0 = offsets[i], r1 = offsets[i + 1];
  if (r1 < r0 || r0 < 0 || r1 > n_rows || (i == 0 && r0 != 0)) report(status, PACE_ERR_INVALID_ARG);
}

// What a walk wants to know of a sequence: nothing, or a float of an array.
struct NoValue {
  using Value = NoValue;
  __device__ Value operator()(int64_t) const { return {}; }
};
struct FloatOf {
  using Value = float;
  const float* a;
  __device__ Value operator()(int64_t i) const { return a[i]; }
};
__device__ __forceinline__ NoValue shfl_value(NoValue v, int) { return v; }
__device__ __forceinline__ float shfl_value(float v, int j) {
  return __shfl_sync(0xffffffffu, v, j);
}

// Walks the sequences along a warp's tiles.  31 sequences' offsets, flags and values
// (Of's, computed by as many lanes at once) are held at a time, one per lane.  All lanes
// call everything together.
template <class Of>
struct PieceWalker {
  const int64_t* offsets;
  const uint8_t* accepted;  // null: all accepted
  Of of;
  int64_t n_seq;
  int64_t base;             // sequence of lane 0
  int j;                    // current sequence: base + j
  int64_t o;                // lane's offset, value; the lanes' accepted flags
  typename Of::Value v;
  unsigned acc_bits;

  __device__ void load() {
    const int lane = threadIdx.x & 31;
    const int64_t i = base + lane;
    const int64_t is = i < n_seq ? i : n_seq - 1;
    o = offsets[i < n_seq ? i : n_seq];
    v = of(is);
    acc_bits = __ballot_sync(0xffffffffu, accepted ? accepted[is] != 0 : true);
    j = 0;
  }

  // to the last sequence from lo on that begins at or before t, else to lo
  // (a 32-way search: two rounds at 1,024 sequences)
  __device__ void seek(int64_t lo, int64_t t) {
    const int lane = threadIdx.x & 31;
    int64_t hi = n_seq;
    while (hi - lo > 1) {
      const int64_t span = hi - lo;
      const int64_t q = lo + 1 + ((span - 1) * lane) / 32;  // in [lo + 1, hi - 1], nondecreasing
      const unsigned bal = __ballot_sync(0xffffffffu, offsets[q] <= t);
      if (bal == 0u) {
        hi = lo + 1;
      } else {
        const int k = 31 - __clz(bal);
        const int64_t qk = lo + 1 + ((span - 1) * k) / 32;
        hi = k < 31 ? lo + 1 + ((span - 1) * (k + 1)) / 32 : hi;
        lo = qk;
      }
    }
    base = lo;
    load();
  }

  __device__ PieceWalker(const int64_t* offsets_, const uint8_t* accepted_, Of of_, int64_t n_seq_,
                         int64_t t0)
      : offsets(offsets_), accepted(accepted_), of(of_), n_seq(n_seq_), base(0), j(0), o(0), v{},
        acc_bits(0u) {
    if (n_seq > 0) seek(0, t0);
  }

  // Calls f(seq, lo, hi, value, begin) for every piece [lo, hi) of an accepted sequence
  // (which begins at row `begin`) inside the tile [t0, t1), in order; tiles are walked
  // in ascending order.  Whatever the offsets hold, it ends and pieces lie in the tile.
  template <class F>
  __device__ __forceinline__ void walk(int64_t t0, int64_t t1, F f) {
    const unsigned full = 0xffffffffu;
    while (base + j < n_seq) {
      const int64_t o0 = __shfl_sync(full, o, j);
      const int64_t o1 = __shfl_sync(full, o, j + 1);
      const typename Of::Value val = shfl_value(v, j);
      const int64_t p0 = o0 < t0 ? t0 : o0;
      const int64_t p1 = o1 < t1 ? o1 : t1;
      if (p0 < p1 && (acc_bits >> j & 1u)) f(base + j, p0, p1, val, o0);
      if (o1 >= t1) return;  // (o1 == t1: the next tile steps over it)
      if (++j == 31) {
        base += 31;
        if (base < n_seq) {
          load();
          // a run of empty sequences is searched over, not walked (100,000 of them between
          // two sequences of 150,000 rows: loss 11.5 ms walked, 20 us searched)
          if (__shfl_sync(full, o, 31) <= o1) seek(base, o1);
        }
      }
    }
  }

  // The same pieces (walk or collect, not both), 31 sequences at a time: the lane that holds
  // a piece's sequence calls f(index, seq, lo, hi, value, begin), index counting the tile's
  // pieces.  Returns their number.
  template <class F>
  __device__ __forceinline__ int collect(int64_t t0, int64_t t1, F f) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int n = 0;
    while (base + j < n_seq) {
      const int64_t o1 = __shfl_down_sync(full, o, 1);
      const bool held = lane >= j && lane < 31 && base + lane < n_seq;
      const unsigned stop = __ballot_sync(full, held && o1 >= t1);
      const int last = stop ? __ffs(stop) - 1 : 31;
      const int64_t p0 = o < t0 ? t0 : o;
      const int64_t p1 = o1 < t1 ? o1 : t1;
      const bool mine = held && lane <= last && p0 < p1 && (acc_bits >> lane & 1u);
      const unsigned bal = __ballot_sync(full, mine);
      if (mine) f(n + __popc(bal & ((1u << lane) - 1u)), base + lane, p0, p1, v, o);
      n += __popc(bal);
      if (stop) {
        j = last;
        return n;
      }
      const int64_t end = __shfl_sync(full, o, 31);  // of the sequences held
      base += 31;
      j = 0;
      if (base < n_seq) {
        load();
        if (__shfl_sync(full, o, 31) <= end) seek(base, end);
      }
    }
    return n;
  }
};

// A lane's rows of a tile: row t0 + 8 lane + u for u = 0 .. 7, so that aligned arrays
// are read and written as 32 bytes a lane (`vec`: every array of the launch is aligned
// for that) and a piece of the tile is a range of each lane's rows.
__device__ __forceinline__ int row_in_tile(int u) {
  return kRowsPerLane * static_cast<int>(threadIdx.x & 31) + u;
}

inline bool rows_vec(const void* a, const void* b, const void* c, const uint8_t* mask) {
  return aligned(a, 32) && aligned(b, 32) && aligned(c, 32) && aligned(mask, 8);
}

// The mask of the lane's rows as bits (rows at or past t1: 0).
__device__ __forceinline__ unsigned load_mask_bits(const uint8_t* __restrict__ mask, int64_t t0,
                                                   int64_t t1, bool vec) {
  if (vec && t1 - t0 == kRowTile) {
    if (!mask) return 0xffu;
    const uint2 q = *(reinterpret_cast<const uint2*>(mask + t0) + (threadIdx.x & 31));
    uint32_t x = __vcmpne4(q.x, 0u) & 0x08040201u;  // byte k's bit k
    x |= __vcmpne4(q.y, 0u) & 0x80402010u;          // byte k's bit 4 + k
    x |= x >> 16;
    return (x | x >> 8) & 0xffu;
  }
  uint8_t m[kRowsPerLane];
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) {
    const int64_t r = t0 + row_in_tile(u);
    m[u] = r < t1 ? (mask ? mask[r] : 1) : 0;
  }
  unsigned bits = 0u;
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) bits |= (m[u] != 0 ? 1u : 0u) << u;
  return bits;
}

__device__ __forceinline__ void load_rows(const float* __restrict__ a, int64_t t0, int64_t t1,
                                          bool vec, float (&x)[kRowsPerLane]) {
  if (vec && t1 - t0 == kRowTile) {
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]),
                   "=f"(x[6]), "=f"(x[7])
                 : "l"(a + t0 + row_in_tile(0)));
    return;
  }
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) {
    const int64_t r = t0 + row_in_tile(u);
    x[u] = r < t1 ? a[r] : 0.0f;
  }
}

// x of the rows whose bit is set, 0 of the tile's others.
__device__ __forceinline__ void store_rows(float* __restrict__ a, int64_t t0, int64_t t1, bool vec,
                                           unsigned bits, const float (&x)[kRowsPerLane]) {
  float y[kRowsPerLane];
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) y[u] = bits >> u & 1u ? x[u] : 0.0f;
  if (vec && t1 - t0 == kRowTile) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(a + t0 +
                                                                                 row_in_tile(0)),
                 "f"(y[0]), "f"(y[1]), "f"(y[2]), "f"(y[3]), "f"(y[4]), "f"(y[5]), "f"(y[6]),
                 "f"(y[7])
                 : "memory");
    return;
  }
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) {
    const int64_t r = t0 + row_in_tile(u);
    if (r < t1) a[r] = y[u];
  }
}

// The lane's rows that lie in [lo, hi) of the tile at t0, as bits.
__device__ __forceinline__ unsigned piece_bits(int64_t t0, int64_t lo, int64_t hi) {
  const int first = row_in_tile(0);
  const int a = min(max(static_cast<int>(lo - t0) - first, 0), kRowsPerLane);
  const int b = min(max(static_cast<int>(hi - t0) - first, 0), kRowsPerLane);
  return (1u << b) - (1u << a);
}

__device__ __forceinline__ int64_t tile_end(int64_t t0, int64_t n_rows) {
  return t0 + kRowTile < n_rows ? t0 + kRowTile : n_rows;
}

// Calls f(t0, t1, bits) for each of a warp's tiles, bits the lane's rows in the loss;
// the next tile's mask is loaded meanwhile.
template <class F>
__device__ __forceinline__ void walk_rows_in_loss(const int64_t* __restrict__ offsets,
                                                  const uint8_t* __restrict__ accepted,
                                                  const uint8_t* __restrict__ mask, int64_t n_seq,
                                                  int64_t n_rows, int64_t tile0, int64_t tile1,
                                                  bool vec, F f) {
  if (tile0 >= tile1) return;
  int64_t t0 = tile0 * kRowTile;
  unsigned bits = load_mask_bits(mask, t0, tile_end(t0, n_rows), vec);
  PieceWalker<NoValue> pw(offsets, accepted, NoValue{}, n_seq, t0);
  for (int64_t w = tile0; w < tile1; ++w) {
    const int64_t t1 = tile_end(t0, n_rows);
    unsigned next = 0u;
    if (w + 1 < tile1) next = load_mask_bits(mask, t1, tile_end(t1, n_rows), vec);
    unsigned in = 0u;
    pw.walk(t0, t1, [&](int64_t, int64_t lo, int64_t hi, NoValue, int64_t) {
      in |= piece_bits(t0, lo, hi);
    });
    f(t0, t1, in & bits);
    bits = next;
    t0 = t1;
  }
}

// The pieces of a warp's tile and its mask, in shared memory, so that the lanes can share
// out what there is to do per piece.
struct PieceList {
  int64_t seq[kRowTile];
  uint32_t range[kRowTile];  // first row in the tile | end << 16
  unsigned mask[kRowTile / 32];

  // piece n, by one lane (offsets that overlap may make more than a tile has rows: left out)
  __device__ __forceinline__ void put(int n, int64_t s, int64_t t0, int64_t lo, int64_t hi) {
    if (n >= kRowTile) return;
    seq[n] = s;
    range[n] = static_cast<uint32_t>(lo - t0) | static_cast<uint32_t>(hi - t0) << 16;
  }
  __device__ __forceinline__ void put_mask(unsigned bits) {
    reinterpret_cast<uint8_t*>(mask)[threadIdx.x & 31] = static_cast<uint8_t>(bits);
  }
  __device__ __forceinline__ bool in_mask(int row) const { return mask[row >> 5] >> (row & 31) & 1u; }
  // the lane's rows of the tile that lie in piece n, in the first n pieces, as bits
  __device__ __forceinline__ unsigned rows_in_piece(int n) const {
    return piece_bits(0, range[n] & 0xffffu, range[n] >> 16);
  }
  __device__ __forceinline__ unsigned rows_in_pieces(int n) const {
    const int r0 = row_in_tile(0);
    int k = 0;  // the first piece that ends past the lane's first row
    for (int above = n; k < above;) {
      const int m = (k + above) >> 1;
      if (static_cast<int>(range[m] >> 16) <= r0) k = m + 1;
      else above = m;
    }
    unsigned bits = 0u;
    for (; k < n; ++k) {
      bits |= rows_in_piece(k);
      if (static_cast<int>(range[k] >> 16) >= r0 + kRowsPerLane) break;
    }
    return bits;
  }
  __device__ __forceinline__ int rows_in_mask(int n) const {
    const int lo = range[n] & 0xffffu, hi = range[n] >> 16;
    int c = 0;
    for (int w = lo >> 5; w <= (hi - 1) >> 5; ++w) {
      unsigned m = mask[w];
      if (w == lo >> 5) m &= ~0u << (lo & 31);
      if (w == hi >> 5) m &= (1u << (hi & 31)) - 1u;
      c += __popc(m);
    }
    return c;
  }
};

// A lane's log-probs and behaviour log-probs of a tile, with the mask bits.
struct RowLoads {
  float lp[kRowsPerLane], bh[kRowsPerLane];
  unsigned mask;
  __device__ __forceinline__ void load(const float* __restrict__ logprob,
                                       const float* __restrict__ behav,
                                       const uint8_t* __restrict__ mask_, int64_t t0, int64_t t1,
                                       bool vec) {
    load_rows(logprob, t0, t1, vec, lp);
    load_rows(behav, t0, t1, vec, bh);
    mask = load_mask_bits(mask_, t0, t1, vec);
  }
};

}  // namespace pace
