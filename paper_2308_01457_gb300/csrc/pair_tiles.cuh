// Unordered triangle pairs in tiles, and the triangle of Z they fill.
//
// The Galerkin forms are symmetric under exchanging the two triangles (the 6-point rule is the
// same on both), so only pairs t1 < t2 are evaluated and only entries on or below the diagonal
// of Z are accumulated; one pass over Z then mirrors them (mirror_lower).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace fosb {

// Tiles of W test triangles x 32 trial triangles with t2 > t1 somewhere.  Row group rg (of
// R = ceil(nt / W)) needs the column blocks from floor(W rg / 32) on; groups rg and R - 1 - rg
// together need about the same number for every rg, so they share one grid row of
// pair_tiles_width() tiles, of which at most a few are empty.
__host__ __device__ inline int64_t pair_tiles_cols(int64_t nt) { return (nt + 31) / 32; }
__host__ __device__ inline int64_t pair_tiles_rows(int64_t nt, int W) { return ((nt + W - 1) / W + 1) / 2; }
// floor(W rg / 32) + floor(W (R - 1 - rg) / 32) >= C - 3, so a grid row holds at most C + 3 tiles
__host__ __device__ inline int64_t pair_tiles_width(int64_t nt) { return pair_tiles_cols(nt) + 3; }
// Tile x of grid row y: its row group and column block; false when it is empty.
__host__ __device__ inline bool pair_tile(int64_t nt, int W, int64_t y, int64_t x, int64_t& rg, int64_t& cb) {
  const int64_t C = pair_tiles_cols(nt), R = (nt + W - 1) / W;
  rg = y;
  int64_t c0 = W * rg / 32;
  if (x < C - c0) {
    cb = c0 + x;
    return true;
  }
  x -= C - c0;
  if (R - 1 - y == y) return false;
  rg = R - 1 - y;
  c0 = W * rg / 32;
  cb = c0 + x;
  return cb < C;
}

// Position of the entry of edges e1, e2 on or below the diagonal.
__device__ __forceinline__ int64_t lower_at(int e1, int e2, int64_t ldz) {
  return e1 > e2 ? int64_t(e1) * ldz + e2 : int64_t(e2) * ldz + e1;
}

// Tile x of grid row y of the lower triangle of C x C tiles (rows y and C - 1 - y of the triangle
// share a grid row of C + 1 tiles): its row and column; false when it is empty.
__host__ __device__ inline bool lower_tile(int64_t C, int64_t y, int64_t x, int64_t& r, int64_t& c) {
  if (x <= y) {
    r = y;
    c = x;
    return true;
  }
  if (C - 1 - y == y) return false;
  r = C - 1 - y;
  c = x - y - 1;
  return true;
}

}  // namespace fosb
