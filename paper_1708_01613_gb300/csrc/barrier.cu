// Film-barrier pipeline of the extended Shan-Chen model (arXiv 1708.01613,
// Sec. 2.1.5): gas labelling, interaction zones, rupture test (Eq. 41),
// blocked-edge mask, the bounce-back across blocked edges after each step;
// and the initialisation of a box. The diagnostics are in fields.cu.
//
// Readings used (the paper is silent on them):
//  - gas cell: rho < threshold (default ln 2, the critical density of
//    Sec. 2.1.2); bubbles are 4-connected gas components on the torus,
//    labelled by the smallest row-major index in the component;
//  - owner of a liquid cell: the bubble of the nearest gas cell within R_z
//    (the nearest-bubble rule of Sec. 2.1.5, which is where the largest
//    |xi_k| of Eq. 38 sits); -1 if there is none; -2 (a wall cell) if gas
//    cells of two or more bubbles are nearest at the same distance (the
//    flowchart places the barrier wall where the bubbles' domains are equal);
//  - rupture: at a cell with a differing-owner neighbour, n = the first such
//    lattice direction, D2 = p(x+n) - 2 p(x) + p(x-n) with p of Eq. 29; the
//    cell opens for good when |D2| <= eps or sign(D2) differs from the sign
//    stored at the previous relabel;
//  - blocked edge: owners differ, both defined (not -1; the wall's -2 is
//    defined), neither end open.
#include <math.h>

#include "labels.cuh"
#include "launch.cuh"
#include "pull.cuh"

namespace lbm {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ int wrapi(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

inline unsigned blocks_for(long long n, int threads = kThreads) {
  long long b = (n + threads - 1) / threads;
  const long long cap = device_sm_count() * 64LL;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (unsigned)b;
}

// --- union-find labelling (min-root hooking: the root is the min index) ---
__global__ void k_label_init(const float* __restrict__ rho, long long N, float th, int32_t* L) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x)
    L[c] = rho[c] < th ? (int32_t)c : -1;
}

// Relabel variant of k_label_init: each new gas cell first parks its label of
// the previous relabel in keep[c] (INT_MAX where it was liquid) for the
// coalescence count; keep is the owner array, which the owner phase
// rewrites afterwards.
__global__ void k_label_init_keep(const float* __restrict__ rho, long long N, float th, int32_t* L,
                                  int32_t* __restrict__ keep) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const bool gas = rho[c] < th;
    if (gas) {
      const int32_t o = L[c];
      keep[c] = o >= 0 ? o : 0x7fffffff;
    }
    L[c] = gas ? (int32_t)c : -1;
  }
}

// Coalescence events (components of the new labelling holding gas of two or
// more components of the previous one). keep[r] of a new root r collects the
// first earlier label seen in its component (the root starts with its own);
// a member with another earlier label marks the component (-3), and the one
// that marks it first counts it, so every merged component counts once.
__device__ __forceinline__ int merge_vote(int32_t* keep, int r, int o) {
  if (o == 0x7fffffff) return 0;
  const int prev = atomicCAS(keep + r, 0x7fffffff, o);
  if (prev == 0x7fffffff || prev == o || prev == -3) return 0;
  return atomicExch(keep + r, -3) != -3;
}

__global__ void k_merge_count(long long N, const int32_t* __restrict__ L, int32_t* keep, int* flags) {
  int n = 0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const int r = L[c];
    if (r >= 0 && r != c) n += merge_vote(keep, r, keep[c]);
  }
  if (n) atomicAdd(flags + FLAG_MERGES, n);
}

__global__ void k_label_union(int nx, int ny, int32_t* L, int* flags) {
  const long long N = (long long)nx * ny;
  int fail = 0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    if (L[c] < 0) continue;
    const int x = (int)(c % nx), y = (int)(c / nx);
    const int right = y * nx + (x + 1 == nx ? 0 : x + 1);
    const int down = (y + 1 == ny ? 0 : y + 1) * nx + x;
    if (L[right] >= 0) unite(L, (int)c, right, &fail);
    if (L[down] >= 0) unite(L, (int)c, down, &fail);
  }
  if (fail) atomicOr(flags + FLAG_TIMEOUT, 1);
}

__global__ void k_label_flatten(long long N, int32_t* L, int* flags) {
  int fail = 0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    if (L[c] >= 0) L[c] = find_root(L, (int)c, &fail);
  }
  if (fail) atomicOr(flags + FLAG_TIMEOUT, 1);
}

// --- interaction zones: nearest gas cell within R; equidistant bubbles: wall (-2) ---
__global__ void k_owner(int nx, int ny, int R, const int32_t* __restrict__ L, int32_t* __restrict__ own) {
  const long long N = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const int lc = L[c];
    if (lc >= 0) {
      own[c] = lc;
      continue;
    }
    const int x = (int)(c % nx), y = (int)(c / nx);
    int best = -1, bd = 0x7fffffff;
    bool tie = false;
    for (int dy = -R; dy <= R; ++dy) {
      const long long row = (long long)wrapi(y + dy, ny) * nx;
      for (int dx = -R; dx <= R; ++dx) {
        const int d2 = dx * dx + dy * dy;
        if (d2 > R * R || d2 > bd) continue;
        const int l = __ldcg(L + row + wrapi(x + dx, nx));
        if (l < 0) continue;
        if (d2 < bd) {
          bd = d2;
          best = l;
          tie = false;
        } else if (l != best) {
          tie = true;
        }
      }
    }
    own[c] = tie ? -2 : best;
  }
}

// Owner of a liquid cell from a window of labels in shared memory (row0 at
// the cell, row stride W): the label of the nearest labelled cell within R,
// -1 if none, -2 if two different labels are nearest at the same distance.
__device__ __forceinline__ int window_owner(const int* row0, int W, int R) {
  int best = -1, bd = 0x7fffffff;
  bool tie = false;
  for (int dy = -R; dy <= R; ++dy) {
    const int* rowp = row0 + dy * W;
    for (int dx = -R; dx <= R; ++dx) {
      const int d2 = dx * dx + dy * dy;
      if (d2 > R * R || d2 > bd) continue;
      const int l = rowp[dx];
      if (l < 0) continue;
      if (d2 < bd) {
        bd = d2;
        best = l;
        tie = false;
      } else if (l != best) {
        tie = true;
      }
    }
  }
  return tie ? -2 : best;
}

// Tiled owner search: a 32 x 8 tile stages the labels of its window (tile
// plus R on every side, wrapped) in shared memory. A tile with no gas cell
// in that window writes -1 everywhere; otherwise each liquid cell scans the
// window from shared memory. Same result as k_owner (same scan order).
constexpr int kOTX = 32, kOTY = 8, kOMaxR = 16;

__global__ void __launch_bounds__(kOTX * kOTY) k_owner_tiled(int nx, int ny, int R, const int32_t* __restrict__ L,
                                                           int32_t* __restrict__ own) {
  __shared__ int32_t sl[(kOTY + 2 * kOMaxR) * (kOTX + 2 * kOMaxR)];
  const int W = kOTX + 2 * R, H = kOTY + 2 * R;
  const int bx0 = blockIdx.x * kOTX, by0 = blockIdx.y * kOTY;
  const int tid = threadIdx.y * kOTX + threadIdx.x;
  int any = 0;
  for (int k = tid; k < W * H; k += kOTX * kOTY) {
    const int yy = k / W, xx = k - yy * W;
    const int gy = wrapi(by0 - R + yy, ny), gx = wrapi(bx0 - R + xx, nx);
    const int l = L[(long long)gy * nx + gx];
    sl[k] = l;
    any |= l >= 0;
  }
  any = __syncthreads_or(any);
  const int x = bx0 + threadIdx.x, y = by0 + threadIdx.y;
  if (x >= nx || y >= ny) return;
  int result = -1;
  if (any) {
    const int* row0 = sl + (threadIdx.y + R) * W + threadIdx.x + R;
    const int lc = row0[0];
    if (lc >= 0) {
      result = lc;
    } else {
      result = window_owner(row0, W, R);
    }
  }
  own[(long long)y * nx + x] = result;
}

__device__ __forceinline__ float pressure_of(float rho, float G, float rho0) {
  const float s = rho0 * (1.0f - expf(-rho / rho0));
  return rho * (1.0f / 3.0f) + G * s * s * (1.0f / 6.0f);
}

__global__ void k_rupture(int nx, int ny, float G, float rho0, float eps,
                          const float* __restrict__ rho, const int32_t* __restrict__ own,
                          int8_t* __restrict__ sgn, uint8_t* __restrict__ open, int* flags) {
  const long long N = (long long)nx * ny;
  int opened = 0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const int o = own[c];
    const int x = (int)(c % nx), y = (int)(c / nx);
    int dir = 0;
    if (o != -1) {
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const int on = own[(long long)wrapi(y + cy(i), ny) * nx + wrapi(x + cx(i), nx)];
        if (dir == 0 && on != -1 && on != o) dir = i;
      }
    }
    if (dir == 0) {
      sgn[c] = 0;
      continue;
    }
    int ex = 0, ey = 0;
#pragma unroll
    for (int i = 1; i < Q; ++i)
      if (i == dir) {
        ex = cx(i);
        ey = cy(i);
      }
    const float pp = pressure_of(rho[(long long)wrapi(y + ey, ny) * nx + wrapi(x + ex, nx)], G, rho0);
    const float p0 = pressure_of(rho[c], G, rho0);
    const float pm = pressure_of(rho[(long long)wrapi(y - ey, ny) * nx + wrapi(x - ex, nx)], G, rho0);
    const float d2 = pp - 2.0f * p0 + pm;
    const int s = (d2 > 0.f) - (d2 < 0.f);
    const int prev = sgn[c];
    if (eps >= 0.f && !open[c] && (fabsf(d2) <= eps || (prev != 0 && s != prev))) {
      open[c] = 1;
      opened += 1;
    }
    sgn[c] = (int8_t)s;
  }
  if (opened) atomicAdd(flags + FLAG_OPENED, opened);
}

__global__ void k_mask(int nx, int ny, int mpitch, const int32_t* __restrict__ own,
                       const uint8_t* __restrict__ open, uint8_t* __restrict__ mask) {
  const long long N = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const int o = own[c];
    const int x = (int)(c % nx), y = (int)(c / nx);
    unsigned m = 0;
    if (o != -1 && !open[c]) {
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const long long nb = (long long)wrapi(y + cy(i), ny) * nx + wrapi(x + cx(i), nx);
        const int on = own[nb];
        if (on != -1 && on != o && !open[nb]) m |= 1u << (i - 1);
      }
    }
    put_cell(mask + (size_t)y * mpitch, x, nx, (uint8_t)m);
  }
}

// --- initialisation: rows by grid coordinates, one column per thread ---
// The stored buffer holds f_i at the source cell of the next pull:
// B_i(y) = f_i(y + e_i).
template <int S>
__global__ void __launch_bounds__(kThreads) k_init_from_rho(const FieldParams fp, typename Store<S>::T* __restrict__ pops,
                                                            const double* __restrict__ rho) {
  const int nx = fp.nx, ny = fp.ny, x = blockIdx.x * kThreads + threadIdx.x;
  if (x >= nx) return;
  const int xm = pull_wrap(x - 1, nx), xp = pull_wrap(x + 1, nx);
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    const size_t r0 = (size_t)y * nx, rm = (size_t)pull_wrap(y - 1, ny) * nx, rp = (size_t)pull_wrap(y + 1, ny) * nx;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const double r = rho[(cy(i) > 0 ? rp : (cy(i) < 0 ? rm : r0)) + (cx(i) > 0 ? xp : (cx(i) < 0 ? xm : x))];
      put_cell(pops + (size_t)i * fp.plane + (size_t)y * fp.pitch, x, nx, Store<S>::of((float)(wq(i) * r), fp.wref[i]));
    }
  }
}

template <int S>
__global__ void __launch_bounds__(kThreads) k_load_plane(const FieldParams fp, typename Store<S>::T* __restrict__ pops,
                                                         const float* __restrict__ f, int plane, int ex, int ey) {
  const int nx = fp.nx, ny = fp.ny, x = blockIdx.x * kThreads + threadIdx.x;
  if (x >= nx) return;
  const int xs = pull_wrap(x + ex, nx);
  for (int y = blockIdx.y; y < ny; y += gridDim.y)
    put_cell(pops + (size_t)plane * fp.plane + (size_t)y * fp.pitch, x, nx,
             Store<S>::of(f[(size_t)pull_wrap(y + ey, ny) * nx + xs], fp.wref[plane]));
}

// Initial density of a bubble set (tanh profile of the signed distance to the
// nearest interface). One CTA per 32 x 32 tile: the bubbles are filtered
// against the tile first, so each cell takes the minimum only over bubbles
// that can come within kSatQ half-widths of it. Beyond that distance the
// correctly rounded tanh is exactly 1 in FP64 (1 - tanh(20) < 1e-17 < 2^-54),
// so the result equals the minimum over all bubbles: the filter drops nothing
// that could change a single bit.
constexpr int kInitTile = 32;
constexpr int kInitChunk = 512;
constexpr double kSatQ = 20.0;

__global__ void __launch_bounds__(kThreads) k_bubbles_rho(const lbm_bubble* __restrict__ b, int n,
                                                         double rho_l, double rho_g, double width,
                                                         int nx, int ny, double* __restrict__ rho) {
  __shared__ double scx[kInitChunk], scy[kInitChunk], sr[kInitChunk];
  __shared__ int cnt;
  const int ntx = (nx + kInitTile - 1) / kInitTile;
  const int x0 = (int)(blockIdx.x % ntx) * kInitTile, y0 = (int)(blockIdx.x / ntx) * kInitTile;
  const double half = 0.5 * width;
  const double reach = kSatQ * half + 2.0;  // margin over the saturation distance
  const double tcx = x0 + 0.5 * (kInitTile - 1), tcy = y0 + 0.5 * (kInitTile - 1);
  const int tx = threadIdx.x % kInitTile, ty = threadIdx.x / kInitTile;
  constexpr int kRows = kInitTile * kInitTile / kThreads;
  double best[kRows];
#pragma unroll
  for (int j = 0; j < kRows; ++j) best[j] = INFINITY;
  for (int k0 = 0; k0 < n; k0 += kInitChunk) {
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    for (int k = k0 + threadIdx.x; k < min(n, k0 + kInitChunk); k += kThreads) {
      // periodic distance from the tile's centre, less the tile's half extent
      double dx = fabs(tcx - b[k].cx), dy = fabs(tcy - b[k].cy);
      dx = fmax(0.0, fmin(dx, nx - dx) - 0.5 * kInitTile);
      dy = fmax(0.0, fmin(dy, ny - dy) - 0.5 * kInitTile);
      if (sqrt(dx * dx + dy * dy) - b[k].r <= reach) {
        const int slot = atomicAdd(&cnt, 1);
        scx[slot] = b[k].cx;
        scy[slot] = b[k].cy;
        sr[slot] = b[k].r;
      }
    }
    __syncthreads();
    const int m = cnt;
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
      const double x = (double)(x0 + tx), y = (double)(y0 + ty + j * (kThreads / kInitTile));
      for (int k = 0; k < m; ++k) {
        double dx = fabs(x - scx[k]), dy = fabs(y - scy[k]);
        dx = fmin(dx, nx - dx);
        dy = fmin(dy, ny - dy);
        const double s = sqrt(dx * dx + dy * dy) - sr[k];
        if (s < best[j]) best[j] = s;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    const int x = x0 + tx, y = y0 + ty + j * (kThreads / kInitTile);
    if (x >= nx || y >= ny) continue;
    const double q = best[j] / half;
    const double v = q >= kSatQ ? 1.0 : tanh(q);
    rho[(size_t)y * nx + x] = 0.5 * (rho_l + rho_g) + 0.5 * (rho_l - rho_g) * v;
  }
}

// ---------------------------------------------------------------------------
// Tiled barrier pipeline. The box is cut into 32 x 8 tiles; where nx or ny is
// not a multiple of the tile, the last tile column or row is ragged and its
// threads outside the box take part in the barriers only. The density pass also joins the gas cells inside
// each tile (a union-find in shared memory: a gas cell's initial label is
// the smallest index of its piece of the tile) and writes one gas flag per
// tile; the union phase then joins the pieces across tile borders. A tile is
// active when a gas cell lies within the tile span that R_z can reach. Owners, rupture signs and masks can only be
// non-trivial in active tiles (a defined owner needs gas within R_z), so the
// later kernels skip every tile that is inactive now and was inactive at the
// previous relabel: its owner/sign/mask are already -1/0/0. A tile that just
// became inactive is reset to those values. Results equal the untiled kernels.
//
// Every phase is one launch over any number of boxes (a lone box is a list
// of one): each box's CTAs follow those of the boxes before it in the entry
// list (RelabelEntry prefix sums), and a CTA finds its box by binary search.
// Mask bits of the directions 1, 2, 5, 6: each blocked edge is seen from the
// one end where its direction is among these.
constexpr unsigned kCanonBits = 0x33u;
// CTAs per box for the tile-list phases, at most: eight per SM
inline int list_ctas() { return device_sm_count() * 8; }

__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

enum { kOffTiles = 0, kOffScan = 1, kOffList = 2 };

template <int F>
__device__ __forceinline__ int entry_off(const RelabelEntry& e) {
  return F == kOffTiles ? e.off_tiles : (F == kOffScan ? e.off_scan : e.off_list);
}

// Entry k owning CTA `b`: the last k < m with off(k) <= b.
template <int F>
__device__ __forceinline__ int find_entry(const RelabelEntry* __restrict__ e, int m, int b) {
  int lo = 0, hi = m - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (entry_off<F>(e[mid]) <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One cell per thread. Used for two-component boxes (TWO, FP32), which also
// get the mixture pressure; one-component boxes take the four-cell kernels
// below, whose per-cell arithmetic is this kernel's.
template <int S, bool TWO>
__global__ void __launch_bounds__(kTX * kTY) kb_density_label(const RelabelBox* __restrict__ boxes,
                                                              const RelabelEntry* __restrict__ e, int m, int parity) {
  grid_begin();
  using T = typename Store<S>::T;
  const int k = find_entry<kOffTiles>(e, m, blockIdx.x);
  const RelabelBox& B = boxes[e[k].box];
  const int t = blockIdx.x - e[k].off_tiles;
  const T* p = static_cast<const T*>(B.pops[B.cur ^ parity]);
  const int nx = B.nx, ny = B.ny;
  const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
  const bool in = x < nx && y < ny;  // a ragged tile's threads outside the box only join the barriers
  const int xi = in ? x : 0, yi = in ? y : 0;
  const size_t P = (size_t)B.plane;
  const size_t r0 = (size_t)yi * B.pitch, rm = (size_t)wrap1(yi - 1, ny) * B.pitch, rp = (size_t)wrap1(yi + 1, ny) * B.pitch;
  float f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const size_t row = cy(i) > 0 ? rm : (cy(i) < 0 ? rp : r0);
    f[i] = Store<S>::load(p + (xi - cx(i)), (size_t)i * P + row, B.wref[i]);
  }
  const float r = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
  const size_t c = (size_t)yi * nx + xi;
  if (in) B.rho[c] = r;
  if (TWO && in) {  // two components (FP32): the gas lattice follows the melt's nine planes
    const float* pg = reinterpret_cast<const float*>(p) + (size_t)Q * P;
    float g = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const size_t row = cy(i) > 0 ? rm : (cy(i) < 0 ? rp : r0);
      g += __ldcg(pg + (size_t)i * P + row + (x - cx(i)));
    }
    const float a = B.rho0 * (1.0f - expf(-r / B.rho0)), b = B.rho0 * (1.0f - expf(-g / B.rho0));
    B.pr[c] = (r + g) * (1.0f / 3.0f) + (B.G * a * a + 2.0f * B.G_mg * a * b + B.G_gg * b * b) * (1.0f / 6.0f);
  }
  const bool gas = in && r < B.threshold;
  // gas cells joined inside the tile here (shared-memory union-find); each
  // starts the global union-find pointing at the smallest index of its piece
  // of the tile, and the union phase joins the pieces across tile borders
  __shared__ int sp[kTX * kTY];
  const int li = threadIdx.y * kTX + threadIdx.x;
  sp[li] = gas ? li : -1;
  const int any = __syncthreads_or(gas);
  int32_t lab = -1;
  if (any) {
    int fail = 0;
    if (gas) {
      if (threadIdx.x + 1 < kTX && sp[li + 1] >= 0) tile_unite(sp, li, li + 1, &fail);
      if (threadIdx.y + 1 < kTY && sp[li + kTX] >= 0) tile_unite(sp, li, li + kTX, &fail);
    }
    __syncthreads();
    if (gas) lab = tile_root_index(sp, li, x - threadIdx.x, y - threadIdx.y, nx, &fail);
    if (fail) atomicOr(B.flags + FLAG_TIMEOUT, 1);
  }
  if (gas) {  // the label of the previous relabel, for the coalescence count
    const int32_t o = B.label[c];
    B.owner[c] = o >= 0 ? o : 0x7fffffff;
  }
  if (in) B.label[c] = lab;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    B.tile_gas[t] = (uint8_t)(any != 0);
    if (t == 0) {  // the tile lists are rebuilt by the next phase and the mask phase
      B.flags[FLAG_TILES] = 0;
      B.flags[FLAG_FILM] = 0;
    }
  }
}

// Four cells (x .. x + 3) of one tile row per thread, 8 x 8 threads per
// 32 x 8 tile: the part after the densities r, shared by the vector density
// kernels. Densities out, gas decision (rho < threshold), tile-local
// union-find, the previous labels of gas cells kept for the coalescence
// count, labels out, tile flags; the same results as kb_density_label's
// one-cell threads. vec: the four cells lie inside the row and the row's
// start is 16-byte aligned (one vector store each for densities and labels).
__device__ __forceinline__ void density_label_tail4(const RelabelBox& B, int t, int x, int y, size_t c,
                                                    const float (&r)[4], bool rowin, bool vec) {
  float* const rho = B.rho;
  int32_t* const label = B.label;
  bool in[4], gas[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    in[j] = rowin && x + j < B.nx;
    gas[j] = in[j] && r[j] < B.threshold;
  }
  if (vec) {
    *reinterpret_cast<float4*>(rho + c) = make_float4(r[0], r[1], r[2], r[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (in[j]) rho[c + j] = r[j];
  }
  int32_t lab[4];
  const int any = tile_labels4(gas, x, y, B.nx, lab, B.flags);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (gas[j]) {  // the label of the previous relabel, for the coalescence count
      const int32_t o = label[c + j];
      B.owner[c + j] = o >= 0 ? o : 0x7fffffff;
    }
  if (vec) {
    *reinterpret_cast<int4*>(label + c) = make_int4(lab[0], lab[1], lab[2], lab[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (in[j]) label[c + j] = lab[j];
  }
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    B.tile_gas[t] = (uint8_t)(any != 0);
    if (t == 0) {  // the tile lists are rebuilt by the next phase and the mask phase
      B.flags[FLAG_TILES] = 0;
      B.flags[FLAG_FILM] = 0;
    }
  }
}

// One component, four cells per thread (pull4): each cell's arithmetic is
// kb_density_label's, so densities, labels and tile flags are bitwise the same.
template <int S>
__global__ void __launch_bounds__(kTX / 4 * kTY, 16) kb_density_label4(const RelabelBox* __restrict__ boxes,
                                                                       const RelabelEntry* __restrict__ e, int m,
                                                                       int parity) {
  grid_begin();
  using T = typename Store<S>::T;
  const int k = find_entry<kOffTiles>(e, m, blockIdx.x);
  const RelabelBox& B = boxes[e[k].box];
  const int t = blockIdx.x - e[k].off_tiles;
  const T* p = static_cast<const T*>(B.pops[B.cur ^ parity]);
  const int nx = B.nx, ny = B.ny;
  const int x = (t % B.ntx) * kTX + 4 * threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
  float2 fa[Q], fb[Q];  // cells (x, x + 1) and (x + 2, x + 3)
  pull4<S>(p, B.plane, B.pitch, B.wref, ny, x < nx ? x : 0, y < ny ? y : 0, fa, fb);
  const float2 ra = rho_pair(fa), rb = rho_pair(fb);
  const float r[4] = {ra.x, ra.y, rb.x, rb.y};
  density_label_tail4(B, t, x, y, (size_t)(y < ny ? y : 0) * nx + x, r, y < ny,
                      y < ny && (nx & 3) == 0 && x + 4 <= nx);
}

// Also appends every tile that needs a visit (active now or at the previous
// relabel) to the box's list; the order of the list does not affect any
// result.
__global__ void kb_active(const RelabelBox* __restrict__ boxes, const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  const int k = find_entry<kOffScan>(e, m, blockIdx.x);
  const RelabelBox& B = boxes[e[k].box];
  const int t = (blockIdx.x - e[k].off_scan) * blockDim.x + threadIdx.x;
  const int ntx = B.ntx, nty = B.nty;
  if (t >= ntx * nty) return;
  // tiles within reach of R cells; across the periodic seam of a box with a
  // ragged last tile one tile more
  const int spx = (B.R + kTX - 1) / kTX + (B.nx % kTX ? 1 : 0);
  const int spy = (B.R + kTY - 1) / kTY + (B.ny % kTY ? 1 : 0);
  const int ty = t / ntx, tx = t - ty * ntx;
  int a = 0;
  for (int dy = -spy; dy <= spy && !a; ++dy) {
    const int yy = wrapi(ty + dy, nty);
    for (int dx = -spx; dx <= spx; ++dx) a |= B.tile_gas[yy * ntx + wrapi(tx + dx, ntx)];
  }
  B.tile_active[t] = (uint8_t)(a != 0);
  if (a || B.tile_prev[t]) B.tile_list[atomicAdd(B.flags + FLAG_TILES, 1)] = t;
}

// CTA `first` of `stride` CTAs that walk box k's tile list.
struct ListWalk {
  const RelabelBox* B;
  int first, stride, n;
};

__device__ __forceinline__ ListWalk list_walk(const RelabelBox* __restrict__ boxes, const RelabelEntry* __restrict__ e,
                                              int m) {
  const int k = find_entry<kOffList>(e, m, blockIdx.x);
  ListWalk w;
  w.B = &boxes[e[k].box];
  w.first = blockIdx.x - e[k].off_list;
  w.stride = e[k + 1].off_list - e[k].off_list;
  w.n = w.B->flags[FLAG_TILES];
  return w;
}

__global__ void __launch_bounds__(kTX * kTY) kb_union(const RelabelBox* __restrict__ boxes,
                                                      const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  const int nx = B.nx, ny = B.ny;
  int32_t* L = B.label;
  int fail = 0;
  for (int w = lw.first; w < lw.n; w += lw.stride) {
    const int t = B.tile_list[w];
    if (!B.tile_gas[t]) continue;
    // edges inside the tile were joined by the density phase: only the
    // right and bottom borders (periodic wrap included) are left
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    if (x >= nx || y >= ny) continue;
    const bool re = threadIdx.x == kTX - 1 || x == nx - 1, be = threadIdx.y == kTY - 1 || y == ny - 1;
    if (!re && !be) continue;
    const int c = y * nx + x;
    if (L[c] < 0) continue;
    if (re) {
      const int right = y * nx + (x + 1 == nx ? 0 : x + 1);
      if (L[right] >= 0) unite(L, c, right, &fail);
    }
    if (be) {
      const int down = (y + 1 == ny ? 0 : y + 1) * nx + x;
      if (L[down] >= 0) unite(L, c, down, &fail);
    }
  }
  if (fail) atomicOr(B.flags + FLAG_TIMEOUT, 1);
}

__global__ void __launch_bounds__(kTX * kTY) kb_flatten(const RelabelBox* __restrict__ boxes,
                                                        const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  int32_t* L = B.label;
  int fail = 0;
  for (int w = lw.first; w < lw.n; w += lw.stride) {
    const int t = B.tile_list[w];
    if (!B.tile_gas[t]) continue;
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    if (x >= B.nx || y >= B.ny) continue;
    const int c = y * B.nx + x;
    if (L[c] >= 0) L[c] = find_root(L, c, &fail);
  }
  if (fail) atomicOr(B.flags + FLAG_TIMEOUT, 1);
}

// Coalescence events of the relabel (merge_vote), over the listed tiles
// with gas; runs between the flatten and the owner phase, whose owner array
// holds the earlier labels the density phase parked there.
__global__ void __launch_bounds__(kTX * kTY) kb_merge(const RelabelBox* __restrict__ boxes,
                                                      const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  int n = 0;
  for (int w = lw.first; w < lw.n; w += lw.stride) {
    const int t = B.tile_list[w];
    if (!B.tile_gas[t]) continue;
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    if (x >= B.nx || y >= B.ny) continue;
    const int c = y * B.nx + x;
    const int r = B.label[c];
    if (r >= 0 && r != c) n += merge_vote(B.owner, r, B.owner[c]);
  }
  n = __syncthreads_count(n);
  if (n && threadIdx.x == 0 && threadIdx.y == 0) atomicAdd(B.flags + FLAG_MERGES, n);
}

// Owner from the labels within radius R of the window position row0 (window
// width W): the label of the nearest labelled cell, -1 if none, -2 if two
// different labels are nearest at the same distance. Shells of equal squared
// distance are scanned in increasing order and the first shell holding a
// label decides: the unsigned minimum of its labels (-1 is the largest
// unsigned value) and the signed maximum (-1 is the smallest) are that
// shell's smallest and largest label, equal unless two bubbles tie. With R
// known at compile time every offset is one shared load, one min and one max.
template <int R>
__device__ __forceinline__ int nearest_label(const int* row0) {
  constexpr int W = kTX + 2 * R;
  unsigned lo = 0xffffffffu;
  int hi = -1;
#pragma unroll
  for (int S = 1; S <= R * R; ++S) {
    bool any = false;
#pragma unroll
    for (int dy = -R; dy <= R; ++dy)
#pragma unroll
      for (int dx = -R; dx <= R; ++dx)
        if (dx * dx + dy * dy == S) {
          const int l = row0[dy * W + dx];
          lo = min(lo, (unsigned)l);
          hi = max(hi, l);
          any = true;
        }
    if (any && lo != 0xffffffffu) break;
  }
  return lo == 0xffffffffu ? -1 : (hi != (int)lo ? -2 : (int)lo);
}

__global__ void __launch_bounds__(kTX * kTY) kb_owner(const RelabelBox* __restrict__ boxes,
                                                      const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  __shared__ int32_t sl[(kTY + 2 * kOMaxR) * (kTX + 2 * kOMaxR)];
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  const int nx = B.nx, ny = B.ny, R = B.R;
  const int32_t* L = B.label;
  for (int w = lw.first; w < lw.n; w += lw.stride) {
    const int t = B.tile_list[w];
    const int tx = t % B.ntx, ty = t / B.ntx;
    const int x = tx * kTX + threadIdx.x, y = ty * kTY + threadIdx.y;
    const bool in = x < nx && y < ny;
    const size_t c = (size_t)y * nx + x;
    if (!B.tile_active[t]) {  // went quiet since the previous relabel
      if (in) B.owner[c] = -1;
      continue;
    }
    const int W = kTX + 2 * R, H = kTY + 2 * R;
    const int bx0 = tx * kTX - R, by0 = ty * kTY - R;
    __syncthreads();  // the previous tile's window is no longer read
    for (int yy = threadIdx.y; yy < H; yy += kTY) {
      const size_t row = (size_t)wrap1(by0 + yy, ny) * nx;
      for (int xx = threadIdx.x; xx < W; xx += kTX) sl[yy * W + xx] = L[row + wrap1(bx0 + xx, nx)];
    }
    __syncthreads();
    const int* row0 = sl + (threadIdx.y + R) * W + threadIdx.x + R;
    int result = row0[0];
    if (result < 0 && R == 4) {  // the default zone radius
      result = nearest_label<4>(row0);
    } else if (result < 0) {
      result = window_owner(row0, W, R);
    }
    if (in) B.owner[c] = result;
  }
}

template <bool TWO>
__global__ void __launch_bounds__(kTX * kTY) kb_rupture(const RelabelBox* __restrict__ boxes,
                                                        const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  const int nx = B.nx, ny = B.ny;
  const int32_t* own = B.owner;
  for (int w = lw.first; w < lw.n; w += lw.stride) {
    const int t = B.tile_list[w];
    const int act = B.tile_active[t];
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    const bool in = x < nx && y < ny;
    const size_t c = (size_t)y * nx + x;
    const int o = act && in ? own[c] : -1;
    int dir = 0;
    if (o != -1) {
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const int on = own[(size_t)wrap1(y + cy(i), ny) * nx + wrap1(x + cx(i), nx)];
        if (dir == 0 && on != -1 && on != o) dir = i;
      }
    }
    int opened = 0;
    if (dir == 0) {
      if (in) B.sgn[c] = 0;
    } else {
      int ex = 0, ey = 0;
#pragma unroll
      for (int i = 1; i < Q; ++i)
        if (i == dir) {
          ex = cx(i);
          ey = cy(i);
        }
      const size_t cp = (size_t)wrap1(y + ey, ny) * nx + wrap1(x + ex, nx);
      const size_t cm = (size_t)wrap1(y - ey, ny) * nx + wrap1(x - ex, nx);
      const float pp = TWO ? B.pr[cp] : pressure_of(B.rho[cp], B.G, B.rho0);
      const float p0 = TWO ? B.pr[c] : pressure_of(B.rho[c], B.G, B.rho0);
      const float pm = TWO ? B.pr[cm] : pressure_of(B.rho[cm], B.G, B.rho0);
      const float d2 = pp - 2.0f * p0 + pm;
      const int sg = (d2 > 0.f) - (d2 < 0.f);
      const int prevs = B.sgn[c];
      if (B.eps >= 0.f && !B.open[c] && (fabsf(d2) <= B.eps || (prevs != 0 && sg != prevs))) {
        B.open[c] = 1;
        opened = 1;
      }
      B.sgn[c] = (int8_t)sg;
    }
    const int n = __syncthreads_count(opened);
    if (n && threadIdx.x == 0 && threadIdx.y == 0) atomicAdd(B.flags + FLAG_OPENED, n);
  }
}

// Also records this relabel's activity as the "previous" one of the next:
// tiles outside the list are inactive in both, so only listed tiles change.
__global__ void __launch_bounds__(kTX * kTY) kb_mask(const RelabelBox* __restrict__ boxes,
                                                     const RelabelEntry* __restrict__ e, int m) {
  grid_begin();
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  const int nx = B.nx, ny = B.ny;
  for (int w = lw.first; w < lw.n; w += lw.stride) {
    const int t = B.tile_list[w];
    const int act = B.tile_active[t];
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    const bool in = x < nx && y < ny;
    const size_t c = (size_t)y * nx + x;
    unsigned msk = 0;
    const int o = act && in ? B.owner[c] : -1;
    if (o != -1 && !B.open[c]) {
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const size_t nb = (size_t)wrap1(y + cy(i), ny) * nx + wrap1(x + cx(i), nx);
        const int on = B.owner[nb];
        if (on != -1 && on != o && !B.open[nb]) msk |= 1u << (i - 1);
      }
    }
    if (in) put_cell(B.mask + (size_t)y * B.mpitch, x, nx, (uint8_t)msk);
    // tiles holding a blocked edge go to the bounce-back's list
    const int film = __syncthreads_or((msk & kCanonBits) != 0);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      B.tile_prev[t] = (uint8_t)act;
      if (film) B.film_list[atomicAdd(B.flags + FLAG_FILM, 1)] = t;
    }
  }
}

// --- halfway bounce-back across blocked edges (the barrier of Sec. 2.1.5) ---
// The step kernels store every outgoing population in its own slot: slot
// (plane i, x) holds f_i^out(x), which the next step pulls into x + e_i. For
// a blocked edge (x, x + e_i) the wall sends it back instead: f_i^out(x)
// returns to x as population opp(i), which the next step pulls from
// x - e_opp(i) = x + e_i in plane opp(i), and f_opp(i)^out(x + e_i) returns to
// x + e_i as population i, pulled from slot (plane i, x). So after the step
// the two slots of every blocked edge trade their values. The mask is
// symmetric; each edge is handled once, from its end whose direction is
// 1, 2, 5 or 6 (mask bits 0, 1, 4, 5), and every slot belongs to one edge
// only, so no two threads touch the same slot. T is the raw storage word
// (4 or 2 bytes: the values move bit for bit); TWO: a second lattice follows
// the first nine planes.
template <typename T, bool TWO>
__device__ __forceinline__ void bounce_cell(T* __restrict__ pops, size_t plane, int pitch, int x, int y, int nx, int ny,
                                            unsigned m) {
  m &= kCanonBits;
  if (!m) return;
#pragma unroll
  for (int i = 1; i <= 6; ++i) {
    if (i == 3 || i == 4 || !((m >> (i - 1)) & 1u)) continue;
    const int xb = wrap1(x + cx(i), nx);
    T* ra = pops + (size_t)i * plane + (size_t)y * pitch;
    T* rb = pops + (size_t)opp(i) * plane + (size_t)wrap1(y + cy(i), ny) * pitch;
#pragma unroll
    for (int k = 0; k < (TWO ? 2 : 1); ++k, ra += Q * plane, rb += Q * plane) {
      const T va = ra[x], vb = rb[xb];
      put_cell(ra, x, nx, vb);
      put_cell(rb, xb, nx, va);
    }
  }
}

// Every cell of a box (boxes that do not use the tiled pipeline).
template <typename T, bool TWO>
__global__ void k_bounce(T* __restrict__ pops, const uint8_t* __restrict__ mask, int nx, int ny, int pitch,
                         long long plane, int mpitch) {
  const long long N = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % nx), y = (int)(c / nx);
    const unsigned m = mask[(size_t)y * mpitch + x];
    if (m & kCanonBits) bounce_cell<T, TWO>(pops, (size_t)plane, pitch, x, y, nx, ny, m);
  }
}

// Tiled boxes: the mask phase of the latest relabel listed the tiles that
// hold a blocked edge (a short list: film tiles only). Buffer
// B.pops[B.cur ^ q] of every box in the entry list.
template <typename T, bool TWO>
__global__ void __launch_bounds__(kTX * kTY) kb_bounce(const RelabelBox* __restrict__ boxes,
                                                       const RelabelEntry* __restrict__ e, int m, int q) {
  grid_begin();
  const ListWalk lw = list_walk(boxes, e, m);
  const RelabelBox& B = *lw.B;
  T* pops = static_cast<T*>(const_cast<void*>(B.pops[B.cur ^ q]));
  const int nfilm = B.flags[FLAG_FILM];
  for (int w = lw.first; w < nfilm; w += lw.stride) {
    const int t = B.film_list[w];
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    if (x >= B.nx || y >= B.ny) continue;
    const unsigned msk = B.mask[(size_t)y * B.mpitch + x];
    if (msk & kCanonBits) bounce_cell<T, TWO>(pops, (size_t)B.plane, B.pitch, x, y, B.nx, B.ny, msk);
  }
}

}  // namespace

cudaError_t launch_labels(const FieldParams& fp, const float* rho, float threshold, int32_t* label,
                          int* flags, cudaStream_t s, int32_t* keep) {
  const unsigned b = blocks_for(fp.N);
  if (keep) k_label_init_keep<<<b, kThreads, 0, s>>>(rho, fp.N, threshold, label, keep);
  else k_label_init<<<b, kThreads, 0, s>>>(rho, fp.N, threshold, label);
  k_label_union<<<b, kThreads, 0, s>>>(fp.nx, fp.ny, label, flags);
  k_label_flatten<<<b, kThreads, 0, s>>>(fp.N, label, flags);
  if (keep) k_merge_count<<<b, kThreads, 0, s>>>(fp.N, label, keep, flags);
  return cudaGetLastError();
}

cudaError_t launch_owner(int nx, int ny, int R, const int32_t* label, int32_t* owner, cudaStream_t s) {
  if (R <= kOMaxR) {
    dim3 grid((nx + kOTX - 1) / kOTX, (ny + kOTY - 1) / kOTY);
    k_owner_tiled<<<grid, dim3(kOTX, kOTY), 0, s>>>(nx, ny, R, label, owner);
  } else {
    k_owner<<<blocks_for((long long)nx * ny), kThreads, 0, s>>>(nx, ny, R, label, owner);
  }
  return cudaGetLastError();
}

cudaError_t launch_rupture(int nx, int ny, float G, float rho0, float eps, const float* rho,
                           const int32_t* owner, int8_t* sgn, uint8_t* open, int* flags,
                           cudaStream_t s) {
  k_rupture<<<blocks_for((long long)nx * ny), kThreads, 0, s>>>(nx, ny, G, rho0, eps, rho, owner, sgn,
                                                                open, flags);
  return cudaGetLastError();
}

cudaError_t launch_mask(int nx, int ny, int mpitch, const int32_t* owner, const uint8_t* open, uint8_t* mask,
                        cudaStream_t s) {
  k_mask<<<blocks_for((long long)nx * ny), kThreads, 0, s>>>(nx, ny, mpitch, owner, open, mask);
  return cudaGetLastError();
}

static dim3 init_grid(const FieldParams& fp) {
  return dim3((fp.nx + kThreads - 1) / kThreads, fp.ny < 65535 ? fp.ny : 65535);
}

#define LBM_BY_STORAGE(storage, CALL)                           \
  switch (storage) {                                            \
    case LBM_F32: CALL(LBM_F32, float); break;                  \
    case LBM_F16_DEV: CALL(LBM_F16_DEV, __half); break;         \
    case LBM_BF16_DEV: CALL(LBM_BF16_DEV, __nv_bfloat16); break; \
    default: return cudaErrorInvalidValue;                      \
  }

cudaError_t launch_init_from_rho(const FieldParams& fp, const double* rho, cudaStream_t s) {
#define CALL(S, T) k_init_from_rho<S><<<init_grid(fp), kThreads, 0, s>>>(fp, static_cast<T*>(const_cast<void*>(fp.pops)), rho)
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_load_plane(const FieldParams& fp, const float* f, int plane, cudaStream_t s) {
#define CALL(S, T)                                                                                                   \
  k_load_plane<S><<<init_grid(fp), kThreads, 0, s>>>(fp, static_cast<T*>(const_cast<void*>(fp.pops)), f, plane, cx(plane), \
                                                     cy(plane))
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_bubbles_rho(const lbm_bubble* d_bubbles, int n, double rho_l, double rho_g,
                               double width, int nx, int ny, double* rho, cudaStream_t s) {
  const unsigned tiles = (unsigned)((nx + kInitTile - 1) / kInitTile) * ((ny + kInitTile - 1) / kInitTile);
  k_bubbles_rho<<<tiles, kThreads, 0, s>>>(d_bubbles, n, rho_l, rho_g, width, nx, ny, rho);
  return cudaGetLastError();
}

bool relabel_tiled_ok(int nx, int ny, int R) { return nx > 2 * R && ny > 2 * R && R <= kOMaxR; }

int relabel_tile_count(int nx, int ny) { return ((nx + kTX - 1) / kTX) * ((ny + kTY - 1) / kTY); }

void relabel_entry_sizes(int nx, int ny, int* tiles, int* scan, int* list) {
  const int t = relabel_tile_count(nx, ny);
  *tiles = t;
  *scan = (t + kThreads - 1) / kThreads;
  const int cap = list_ctas();
  *list = t < cap ? t : cap;
}

cudaError_t launch_relabel_boxes(int storage, const RelabelBox* boxes, const RelabelEntry* entries, int m,
                                 const int totals[3], int parity, cudaStream_t s, bool two) {
  if (m <= 0) return cudaSuccess;
  const dim3 block(kTX, kTY);
  if (two) {  // two components: FP32 only
    if (storage != LBM_F32) return cudaErrorInvalidValue;
    LBM_TRY(launch_chain(kb_density_label<LBM_F32, true>, dim3(totals[0]), block, 0, s, boxes, entries, m, parity));
  } else {
    switch (storage) {
      case LBM_F32: 
        LBM_TRY(launch_chain(kb_density_label4<LBM_F32>, dim3(totals[0]), dim3(kTX / 4, kTY), 0, s, boxes, entries, m, parity));
        break;
      case LBM_F16_DEV:
        LBM_TRY(launch_chain(kb_density_label4<LBM_F16_DEV>, dim3(totals[0]), dim3(kTX / 4, kTY), 0, s, boxes, entries, m, parity));
        break;
      case LBM_BF16_DEV:
        LBM_TRY(launch_chain(kb_density_label4<LBM_BF16_DEV>, dim3(totals[0]), dim3(kTX / 4, kTY), 0, s, boxes, entries, m, parity));
        break;
      default: return cudaErrorInvalidValue;
    }
  }
  LBM_TRY(launch_chain(kb_active, dim3(totals[1]), dim3(kThreads), 0, s, boxes, entries, m));
  LBM_TRY(launch_chain(kb_union, dim3(totals[2]), block, 0, s, boxes, entries, m));
  LBM_TRY(launch_chain(kb_flatten, dim3(totals[2]), block, 0, s, boxes, entries, m));
  LBM_TRY(launch_chain(kb_merge, dim3(totals[2]), block, 0, s, boxes, entries, m));
  LBM_TRY(launch_chain(kb_owner, dim3(totals[2]), block, 0, s, boxes, entries, m));
  if (two) LBM_TRY(launch_chain(kb_rupture<true>, dim3(totals[2]), block, 0, s, boxes, entries, m));
  else LBM_TRY(launch_chain(kb_rupture<false>, dim3(totals[2]), block, 0, s, boxes, entries, m));
  LBM_TRY(launch_chain(kb_mask, dim3(totals[2]), block, 0, s, boxes, entries, m));
  return cudaGetLastError();
}

cudaError_t launch_bounce(const FieldParams& fp, bool two, void* pops, const uint8_t* mask, cudaStream_t s) {
  const unsigned b = blocks_for(fp.N);
  if (two && fp.storage != LBM_F32) return cudaErrorInvalidValue;
#define CALL(T, TWO) \
  k_bounce<T, TWO><<<b, kThreads, 0, s>>>(static_cast<T*>(pops), mask, fp.nx, fp.ny, fp.pitch, fp.plane, fp.mpitch)
  if (two) CALL(uint32_t, true);
  else if (fp.storage == LBM_F32) CALL(uint32_t, false);
  else CALL(uint16_t, false);
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_bounce_boxes(int storage, bool two, const RelabelBox* boxes, const RelabelEntry* entries, int m,
                                int total_list, int q, cudaStream_t s) {
  if (m <= 0 || total_list <= 0) return cudaSuccess;
  const dim3 block(kTX, kTY);
  if (two) {
    if (storage != LBM_F32) return cudaErrorInvalidValue;
    LBM_TRY(launch_chain(kb_bounce<uint32_t, true>, dim3(total_list), block, 0, s, boxes, entries, m, q));
  } else if (storage == LBM_F32) {
    LBM_TRY(launch_chain(kb_bounce<uint32_t, false>, dim3(total_list), block, 0, s, boxes, entries, m, q));
  } else {
    LBM_TRY(launch_chain(kb_bounce<uint16_t, false>, dim3(total_list), block, 0, s, boxes, entries, m, q));
  }
  return cudaGetLastError();
}

}  // namespace lbm
