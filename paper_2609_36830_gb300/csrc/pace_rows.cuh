// The rows of a batch walked in flat tiles: a warp takes 512 consecutive rows,
// whatever sequences they belong to, so long and short sequences load the chip
// alike and every lane has 16 rows' loads in flight.  (With a block per sequence, the
// longest sequence's chain of dependent loads set the time: 80 us over 5.4M rows of
// 1,024 sequences, a tenth of the memory's rate.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pace_internal.cuh"

namespace pace {

constexpr int kRowTile = 512;
constexpr int kRowsPerLane = kRowTile / 32;
constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kMaxRowBlocks = 2048;  // more rows than 8.4M: several tiles a warp

// One launch over n_rows rows: block b's warp w walks `per_warp` tiles from tile
// (b * kRowWarps + w) * per_warp on.
struct RowGeom {
  int64_t n_tiles;
  int per_warp;
  int blocks;
};

__host__ __device__ inline RowGeom row_geom(int64_t n_rows) {
  RowGeom g;
  g.n_tiles = (n_rows + kRowTile - 1) / kRowTile;
  const int64_t most = static_cast<int64_t>(kMaxRowBlocks) * kRowWarps;
  g.per_warp = static_cast<int>((g.n_tiles + most - 1) / most);
  if (g.per_warp < 1) g.per_warp = 1;
  const int64_t per_block = static_cast<int64_t>(g.per_warp) * kRowWarps;
  g.blocks = static_cast<int>((g.n_tiles + per_block - 1) / per_block);
  return g;
}

// Reports offsets that do not partition the rows (any thread of a grid: sequence i).
__device__ __forceinline__ void check_seq(const int64_t* __restrict__ offsets, int64_t i,
                                          int64_t n_rows, int32_t* status) {
  const int64_t r0 = offsets[i], r1 = offsets[i + 1];
  if (r1 < r0 || r0 < 0 || r1 > n_rows || (i == 0 && r0 != 0)) report(status, PACE_ERR_INVALID_ARG);
}

// Calls f(seq, lo, hi, value) for every piece [lo, hi) of a sequence inside the tile
// [t0, t1), in order; value is seq's entry of `per_seq` (null: 0).  Pieces of
// sequences that are not accepted are left out.  All lanes call it and take every
// call of f together.  31 sequences' offsets, flags and values are loaded at a time.
// Whatever the offsets hold, it ends, and pieces lie in the tile.
template <class F>
__device__ __forceinline__ void walk_pieces(const int64_t* __restrict__ offsets,
                                            const uint8_t* __restrict__ accepted,
                                            const float* __restrict__ per_seq, int64_t n_seq,
                                            int64_t t0, int64_t t1, F f) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // the last sequence in [0, n_seq) that begins at or before t0, else 0 (32-way search)
  int64_t lo = 0, hi = n_seq;
  while (hi - lo > 1) {
    const int64_t span = hi - lo;
    const int64_t q = lo + 1 + ((span - 1) * lane) / 32;  // in [lo + 1, hi - 1], nondecreasing
    const unsigned bal = __ballot_sync(full, offsets[q] <= t0);
    if (bal == 0u) {
      hi = lo + 1;
    } else {
      const int j = 31 - __clz(bal);
      const int64_t qj = lo + 1 + ((span - 1) * j) / 32;
      hi = j < 31 ? lo + 1 + ((span - 1) * (j + 1)) / 32 : hi;
      lo = qj;
    }
  }
  for (int64_t base = lo; base < n_seq; base += 31) {
    const int64_t i = base + lane;
    const int64_t o = offsets[i < n_seq ? i : n_seq];
    const int64_t is = i < n_seq ? i : n_seq - 1;
    const bool acc = accepted ? accepted[is] != 0 : true;
    const float v = per_seq ? per_seq[is] : 0.0f;
    const unsigned acc_bits = __ballot_sync(full, acc);
    for (int j = 0; j < 31 && base + j < n_seq; ++j) {
      int64_t p0 = __shfl_sync(full, o, j);
      const int64_t o1 = __shfl_sync(full, o, j + 1);
      const float val = __shfl_sync(full, v, j);
      p0 = p0 < t0 ? t0 : p0;
      const int64_t p1 = o1 < t1 ? o1 : t1;
      if (p0 < p1 && (acc_bits >> j & 1u)) f(base + j, p0, p1, val);
      if (o1 >= t1) return;
    }
  }
}

// The tile's rows that are in the loss, as bits (bit u: row t0 + 32 u + lane).
__device__ __forceinline__ unsigned rows_in_loss(const int64_t* __restrict__ offsets,
                                                 const uint8_t* __restrict__ accepted,
                                                 const uint8_t* __restrict__ mask, int64_t n_seq,
                                                 int64_t n_rows, int64_t t0) {
  const int lane = threadIdx.x & 31;
  const int64_t t1 = t0 + kRowTile < n_rows ? t0 + kRowTile : n_rows;
  uint8_t m[kRowsPerLane];
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) {
    const int64_t r = t0 + 32 * u + lane;
    m[u] = r < t1 ? (mask ? mask[r] : 1) : 0;
  }
  unsigned bits = 0u;
#pragma unroll
  for (int u = 0; u < kRowsPerLane; ++u) bits |= (m[u] != 0 ? 1u : 0u) << u;
  unsigned in = 0u;
  walk_pieces(offsets, accepted, nullptr, n_seq, t0, t1,
              [&](int64_t, int64_t lo, int64_t hi, float) {
                // the lane's rows in [lo, hi): u from ceil((lo - t0 - lane) / 32) on
                const int a = static_cast<int>(lo - t0), b = static_cast<int>(hi - t0);
                const int u0 = a > lane ? (a - lane + 31) >> 5 : 0;
                const int u1 = b > lane ? (b - lane + 31) >> 5 : 0;
                in |= (1u << u1) - (1u << u0);
              });
  return in & bits;
}

}  // namespace pace
