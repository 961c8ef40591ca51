// frest.cuh -- filter membership (Sec. 3.2).  Shells: a pair is filtered iff
// its stencil is one of the rest mesh's filtered pairs, kept as bit masks over
// pairs of primitive clusters (broad.cu).  Rods: through the per-edge
// arc-length windows.
#pragma once
#include <cstdint>

#include "common.cuh"

// The filtered pairs of a shell's rest mesh as 32x32 bit masks over the pairs
// of clusters that hold any: an open-addressing table (linear probing, at most
// half full) of tile keys, and at the same place the mask, word r for row
// primitive r.
struct FilterMasks {
  const unsigned long long* __restrict__ key;
  const uint32_t* __restrict__ bits;
  uint32_t mask;  // table size - 1 (0: no filtered pair)

  static constexpr unsigned long long EMPTY = ~0ull;
  __host__ __device__ static __forceinline__ unsigned long long tile_key(uint32_t row, uint32_t col) {
    return ((unsigned long long)row << 32) | col;
  }
  // multiplicative (Fibonacci) hashing of the tile key, Knuth
  __host__ __device__ static __forceinline__ uint32_t hash(unsigned long long k) {
    return (uint32_t)((k * 0x9E3779B97F4A7C15ull) >> 32);
  }
  // word `lane` of the tile's mask (0 if it has none); every lane of the warp
  // calls it with the same tile, and the lanes probe 32 places at once
  __device__ __forceinline__ uint32_t row(uint32_t r, uint32_t c, int lane) const {
    if (mask == 0u) return 0u;
    const unsigned long long k = tile_key(r, c);
    for (uint32_t h = hash(k);; h += 32u) {
      const unsigned long long e = key[(h + (uint32_t)lane) & mask];
      const unsigned hit = __ballot_sync(0xffffffffu, e == k), end = __ballot_sync(0xffffffffu, e == EMPTY);
      const int at = __ffs((int)hit) - 1, stop = __ffs((int)end) - 1;
      if (at >= 0 && (stop < 0 || at < stop)) return bits[(size_t)((h + (uint32_t)at) & mask) * 32 + lane];
      if (stop >= 0) return 0u;  // (half of the table is empty: the loop ends)
    }
  }
};

// Rods: edges ki < kj of one polyline are filtered when kj is within the
// forward window of ki (kj <= win) or, on a closed loop, within its
// backward window (kj >= wst >= 0: the gap the other way round is below
// the activation).  loops: the member has closed loops (else wst is not used).
__device__ __forceinline__ bool rod_filtered(int win, int wst, bool loops, int kj) {
  return kj <= win || (loops && wst >= 0 && kj >= wst);
}

// Rods: the index gap of edges ki < kj of one polyline (Kaldor culling);
// on a closed loop of m edges the shorter way round
__device__ __forceinline__ int rod_gap(const int32_t* __restrict__ rloop, uint32_t ki, uint32_t kj) {
  const int g = (int)(kj - ki), m = rloop[ki];
  return m > 0 ? min(g, m - g) : g;
}
