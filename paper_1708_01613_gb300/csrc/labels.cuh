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

// Both roots, the two walks side by side (each hop is a load's latency).
__device__ __forceinline__ void find_roots(const int32_t* L, int& a, int& b, int* fail) {
  for (int it = 0; it < kUnionIters; ++it) {
    const int p = L[a], q = L[b];
    if (p == a && q == b) return;
    a = p;
    b = q;
  }
  *fail = 1;
}

__device__ __forceinline__ void unite(int32_t* L, int a, int b, int* fail) {
  for (int it = 0; it < kUnionIters; ++it) {
    find_roots(L, a, b, fail);
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
//
// The gas of a row is a 32-bit mask, so every cell starts with its run's first
// cell as parent, and only the first cell of each overlap with the row below
// unites: a few links per tile instead of two per gas cell.
__device__ __forceinline__ int tile_labels4(const bool (&gas)[4], int x, int y, int nx, int32_t (&lab)[4], int* flags) {
  __shared__ int sp[kTX * kTY];
  __shared__ unsigned rows[kTY];
  const int col = 4 * threadIdx.x, la = threadIdx.y * kTX + col;
  const unsigned own = (gas[0] ? 1u : 0u) | (gas[1] ? 2u : 0u) | (gas[2] ? 4u : 0u) | (gas[3] ? 8u : 0u);
  unsigned row = own << col;
#pragma unroll
  for (int d = 1; d < 8; d *= 2) row |= __shfl_xor_sync(0xffffffffu, row, d);
  if (threadIdx.x == 0) rows[threadIdx.y] = row;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const unsigned liquid = ~row & ((1u << (col + j)) - 1u);  // liquid cells to the left
    sp[la + j] = gas[j] ? (int)threadIdx.y * kTX + 32 - __clz(liquid) : -1;
    lab[j] = -1;
  }
  const int any = __syncthreads_or(own);
  if (any) {
    int fail = 0;
    if (own && threadIdx.y + 1 < kTY) {
      const unsigned both = row & rows[threadIdx.y + 1], first = both & ~(both << 1);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((first >> (col + j)) & 1u) tile_unite(sp, la + j, la + j + kTX, &fail);
    }
    __syncthreads();
    const int x0 = x - col, y0 = y - threadIdx.y;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (gas[j]) lab[j] = tile_root_index(sp, la + j, x0, y0, nx, &fail);
    if (fail) atomicOr(flags + FLAG_TIMEOUT, 1);
  }
  return any;
}

// Joins the gas cells of tile (x0, y0) to the next tile's across its bottom
// and right borders (periodic wrap included); one warp, `lane` its lane, all
// lanes call. One link per run of facing gas cells: the cells of a run are
// joined within each tile already.
__device__ __forceinline__ void tile_union_borders(int32_t* L, int x0, int y0, int nx, int ny, int lane, int* fail) {
  int a = -1, b = -1, ra = -1, rb = -1;
  {
    const int x = x0 + lane, y = min(y0 + kTY, ny) - 1;
    if (x < nx) {
      a = L[y * nx + x];
      b = L[(y + 1 == ny ? 0 : y + 1) * nx + x];
    }
  }
  if (lane < kTY && y0 + lane < ny) {
    const int x = min(x0 + kTX, nx) - 1, y = y0 + lane;
    ra = L[y * nx + x];
    rb = L[y * nx + (x + 1 == nx ? 0 : x + 1)];
  }
  const unsigned down = __ballot_sync(0xffffffffu, a >= 0 && b >= 0),
                 right = __ballot_sync(0xffffffffu, ra >= 0 && rb >= 0);
  if (((down & ~(down << 1)) >> lane) & 1u) unite(L, a, b, fail);
  if (((right & ~(right << 1)) >> lane) & 1u) unite(L, ra, rb, fail);
}

}  // namespace
}  // namespace lbm
