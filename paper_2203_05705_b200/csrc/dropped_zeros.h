// Zeros of what a pattern drops from a weight gradient, written by the warps of the product's own kernel.  Everything is static
// to the including translation unit.  Args: hdr, out, ldo, out_is_f32 and, for rows, N.
#pragma once

#include "ard_internal.h"

namespace {

// The j-th dropped unit of a pattern: bb of them precede the first kept one, dp - 1 follow each kept one.
__device__ __forceinline__ int dropped_unit(int j, int bb, int dp) {
  const int after = j - bb;
  return after < 0 ? j : bb + after / (dp - 1) * dp + 1 + after % (dp - 1);
}

// Weight gradient: zeros of what is dropped, dealt to the grid's `warps` warps.  They go out while the first blocks are on
// their way; a kernel of its own ahead of the product was one more dependent launch (2048 x 2048, 32-wide tiles, batch 128, a
// period of 2, sampler and three products: 50.8 us with it, 48.5 without).
// Tile patterns (Sec. 3.2): a warp takes up to ZERO_PIECES pieces of a tile at a time, so that a few large tiles find as many
// warps as many small ones, and a tile of up to 64 x 64 bf16 values stays with one warp (pieces of a quarter of that: three
// products of 4096 x 4096 with 64-wide tiles, batch 1024, a period of 4, 60 -> 65 us).
template <typename Args>
__device__ __forceinline__ void zero_dropped_tiles(const Args& g, int ts, int warp, int warps, int lane) {
  constexpr int ZERO_PIECES = 512;
  const int dp = g.hdr[HDR_DP], bb = g.hdr[HDR_B] - 1, Tc = g.hdr[HDR_TC];
  const int n_drop = g.hdr[HDR_TR] * Tc - g.hdr[HDR_NKEEP], es = g.out_is_f32 ? 4 : 2;
  const size_t pitch = (size_t)g.ldo * es;
  const bool wide = ((ts * es) & 15) == 0 && (pitch & 15) == 0 && (reinterpret_cast<uintptr_t>(g.out) & 15) == 0;
  const int per_row = wide ? ts * es >> 4 : ts * es >> 1, piece = wide ? 16 : 2;
  const int step_n = 32 / per_row, step_q = 32 - step_n * per_row;
  // 32 bits: a matrix of 180 GB has fewer than 1e9 such units
  const int chunks = (int)(((long long)ts * per_row + ZERO_PIECES - 1) / ZERO_PIECES);
  for (int u = warp; u < n_drop * chunks; u += warps) {
    const int j = u / chunks;
    const unsigned long long e = (unsigned long long)(u - j * chunks) * ZERO_PIECES + lane;
    const int lin = dropped_unit(j, bb, dp);
    const int r = lin / Tc, c = lin - r * Tc;  // tile-row along the fan-in, tile-column along the neurons
    char* tile = reinterpret_cast<char*>(g.out) + (size_t)c * ts * pitch + (size_t)r * ts * es;
    int n = (int)(e >> 32 ? e / per_row : (unsigned)e / (unsigned)per_row), q = (int)(e - (unsigned long long)n * per_row);
    for (int i = 0; i < ZERO_PIECES / 32 && n < ts; ++i) {
      char* d = tile + (size_t)n * pitch + (size_t)q * piece;
      if (wide) *reinterpret_cast<uint4*>(d) = make_uint4(0u, 0u, 0u, 0u);
      else *reinterpret_cast<uint16_t*>(d) = 0;
      n += step_n;
      q += step_q;
      if (q >= per_row) { q -= per_row; ++n; }
    }
  }
}
// Row patterns (Sec. 3.1): a warp takes up to ZERO_BYTES of a row at a time.  cols: of the product, the kept fan-in where
// the layer is fed by a pattern.
template <typename Args>
__device__ __forceinline__ void zero_dropped_rows(const Args& g, int cols, int warp, int warps, int lane) {
  constexpr int ZERO_BYTES = 2048;
  const int dp = g.hdr[HDR_DP], bb = g.hdr[HDR_B] - 1, n_drop = g.N - g.hdr[HDR_NKEEP], es = g.out_is_f32 ? 4 : 2;
  const long long bytes = (long long)cols * es, chunks = (bytes + ZERO_BYTES - 1) / ZERO_BYTES;
  for (long long u = warp; u < n_drop * chunks; u += warps) {
    const int j = (int)(u / chunks);
    const long long b0 = (u - j * chunks) * ZERO_BYTES;
    char* d = reinterpret_cast<char*>(g.out) + (size_t)dropped_unit(j, bb, dp) * g.ldo * es + b0;
    const int n = (int)min((long long)ZERO_BYTES, bytes - b0);
    const int head = min(n, (int)((0 - reinterpret_cast<uintptr_t>(d)) & 15)), body = (n - head) & ~15;
    if (2 * lane < head) *reinterpret_cast<uint16_t*>(d + 2 * lane) = 0;
    for (int e = head + 16 * lane; e < head + body; e += 512) *reinterpret_cast<uint4*>(d + e) = make_uint4(0u, 0u, 0u, 0u);
    if (head + body + 2 * lane < n) *reinterpret_cast<uint16_t*>(d + head + body + 2 * lane) = 0;
  }
}

}  // namespace
