// Gas labelling on 32 x 8 tiles, shared by the relabel pipeline and the
// diagnostics: union-find inside a tile in shared memory, across tile borders
// in global memory. Links always go from the larger index to the smaller
// (min-root hooking), so a component's root is its smallest row-major index.
#pragma once
#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int kTX = kRelabelTileX, kTY = kRelabelTileY;
constexpr int kUnionIters = 1 << 20;  // bound of the union/find retry loops

__device__ __forceinline__ int find_root(const int32_t* L, int a, int* fail) {
  for (int it = 0; it < kUnionIters; ++it) {
    const int p = L[a];
    if (p == a) return a;
    a = p;
  }
  *fail = 1;
  return a;
}

__device__ __forceinline__ void unite(int32_t* L, int a, int b, int* fail) {
  for (int it = 0; it < kUnionIters; ++it) {
    a = find_root(L, a, fail);
    b = find_root(L, b, fail);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    // hook the larger root a under b; if a stopped being a root meanwhile,
    // continue with the value it points to (links only ever decrease)
    const int old = atomicMin(&L[a], b);
    if (old == a) return;
    a = old;
  }
  *fail = 1;
}

// Union-find inside one 32 x 8 tile in shared memory (local indices
// ly * kTX + lx, -1 for liquid), hooking the larger root under the smaller,
// so a root is the smallest local index of its piece. Bounded like the
// global version.
__device__ __forceinline__ int tile_find(const int* sp, int a, int* fail) {
  for (int it = 0; it < kTX * kTY; ++it) {
    const int p = sp[a];
    if (p == a) return a;
    a = p;
  }
  *fail = 1;
  return a;
}

__device__ __forceinline__ void tile_unite(int* sp, int a, int b, int* fail) {
  for (int it = 0; it < kTX * kTY; ++it) {
    a = tile_find(sp, a, fail);
    b = tile_find(sp, b, fail);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    const int old = atomicMin(&sp[a], b);
    if (old == a) return;
    a = old;
  }
  *fail = 1;
}

// Global index of the tile-local root of local cell li (a gas cell).
__device__ __forceinline__ int32_t tile_root_index(const int* sp, int li, int x0, int y0, int nx, int* fail) {
  const int r = tile_find(sp, li, fail);
  return (int32_t)((y0 + r / kTX) * nx + x0 + r % kTX);
}

// Labels of four cells (x .. x + 3, row y) per thread, 8 x 8 threads per
// tile, from their gas decisions: -1 for liquid, else the smallest index of
// the cell's piece of the tile. Returns whether the tile holds gas (uniform
// over the CTA). Contains barriers: every thread of the CTA calls it.
__device__ __forceinline__ int tile_labels4(const bool (&gas)[4], int x, int y, int nx, int32_t (&lab)[4], int* flags) {
  __shared__ int sp[kTX * kTY];
  const int la = threadIdx.y * kTX + 4 * threadIdx.x;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    sp[la + j] = gas[j] ? la + j : -1;
    lab[j] = -1;
  }
  const int any = __syncthreads_or(gas[0] || gas[1] || gas[2] || gas[3]);
  if (any) {
    int fail = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (!gas[j]) continue;
      if (j < 3 ? gas[j + 1] : (4 * threadIdx.x + 4 < kTX && sp[la + 4] >= 0)) tile_unite(sp, la + j, la + j + 1, &fail);
      if (threadIdx.y + 1 < kTY && sp[la + j + kTX] >= 0) tile_unite(sp, la + j, la + j + kTX, &fail);
    }
    __syncthreads();
    const int x0 = x - 4 * threadIdx.x, y0 = y - threadIdx.y;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (gas[j]) lab[j] = tile_root_index(sp, la + j, x0, y0, nx, &fail);
    if (fail) atomicOr(flags + FLAG_TIMEOUT, 1);
  }
  return any;
}

// Joins the gas cells of tile (x0, y0) to the next tile's across its bottom
// and right borders (periodic wrap included); one warp, `lane` its lane.
__device__ __forceinline__ void tile_union_borders(int32_t* L, int x0, int y0, int nx, int ny, int lane, int* fail) {
  {
    const int x = x0 + lane, y = min(y0 + kTY, ny) - 1;
    if (x < nx) {
      const int c = y * nx + x, down = (y + 1 == ny ? 0 : y + 1) * nx + x;
      if (L[c] >= 0 && L[down] >= 0) unite(L, c, down, fail);
    }
  }
  if (lane < kTY && y0 + lane < ny) {
    const int x = min(x0 + kTX, nx) - 1, y = y0 + lane;
    const int c = y * nx + x, right = y * nx + (x + 1 == nx ? 0 : x + 1);
    if (L[c] >= 0 && L[right] >= 0) unite(L, c, right, fail);
  }
}

}  // namespace
}  // namespace lbm
