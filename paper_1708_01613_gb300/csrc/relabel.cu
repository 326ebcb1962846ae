// Film-barrier pipeline (arXiv 1708.01613, Sec. 2.1.5) over 32 x 8 tiles, for
// R_z <= 16; the readings are listed in barrier.cu. Four launches per relabel,
// over one box or over all boxes of a batch that are due:
//
//  1. kb_label: densities of every cell; the gas cells of each tile joined in
//     shared memory (a gas cell's initial label is the smallest index of its
//     piece of the tile), their labels of the previous relabel parked in
//     B.old, one gas flag per tile. The only pass over the populations:
//     36 bytes per cell (FP32), 18 (16-bit), and 4 more in tiles with gas now
//     or before.
//  2. kb_scan: the tiles to visit listed (gas within the span R_z can reach,
//     now or at the previous relabel); the pieces of gas tiles joined across
//     tile borders.
//  3. kb_zone: one CTA per listed tile. It takes a window of labels around
//     the tile, each followed to its root, into shared memory, with the gas
//     of each window row as a bit mask; stores the tile's final labels, counts
//     its coalescence votes, adds its gas to the growth source's census; finds
//     the owners of the tile and its one-cell border (the nearest gas, by bit
//     operations) and makes the rupture test, whose pressures are formed from
//     the populations (at film cells only).
//  4. kb_mask: blocked edges of the film tiles.
//
// Owners, rupture signs and masks can only be non-trivial in active tiles (a
// defined owner needs gas within R_z), so tiles that are inactive now and were
// at the previous relabel are skipped: their owner, sign and mask are -1, 0 and
// 0 already. A tile that just became inactive is reset to those values. Results
// equal the untiled kernels.
//
// What bounds them: the label phase by its read of the populations (8192^2 FP32
// 380 us, 6.4 TB/s; FP16 270 us); the others, over 10 % of the tiles of a box at
// most, by the chain of dependent loads of each tile. Microseconds of the
// phases 1 to 4, and in brackets of the whole with a launch for each of the eight
// things they do (densities written and read, every listed tile visited by five
// kernels): 160 x 80 5.1 + 4.6 + 8.0 + 2.9 (36); 1024^2 FP16 8.3 + 6.2 + 11 + 3.6
// (41); 4096^2 FP32 104 + 9.2 + 37 + 3.3 (212); 8192^2 FP32 384 + 17 + 145 + 4
// (705). Final labels in a launch of their own cost 5 to 45 us more, the mask over
// all listed tiles in place of the film tiles 4 to 100 us. Walks to roots go side
// by side, and a cell's own state is loaded with the window (one after the other:
// scan 6.4 and zone 9.1 us at 160 x 80).
#include <algorithm>

#include "bounce.cuh"
#include "labels.cuh"
#include "launch.cuh"
#include "pull.cuh"

namespace lbm {
namespace {

constexpr int kMaxR = 16;
constexpr int kScanTiles = 32;  // tiles of a scan CTA
constexpr int kTileThreads = kTX * kTY, kTileWarps = kTileThreads / 32;

enum Phase { kTiles, kScan, kList, kFilm };

template <int F>
__host__ __device__ __forceinline__ int entry_off(const RelabelEntry& e) {
  return F == kTiles ? e.off_tiles : (F == kScan ? e.off_scan : (F == kList ? e.off_list : e.off_film));
}

// The boxes of a launch: one, its descriptor a kernel argument, or a list of
// them in device memory (a batch), each with the CTAs of the boxes before it.
struct Lone {
  RelabelBox box;
  template <int F>
  __device__ __forceinline__ int find(int) const { return 0; }
  __device__ __forceinline__ const RelabelBox& get(int) const { return box; }
  template <int F>
  __device__ __forceinline__ int first(int) const { return blockIdx.x; }
  template <int F>
  __device__ __forceinline__ int stride(int) const { return gridDim.x; }
};

struct Many {
  const RelabelBox* boxes;
  const RelabelEntry* e;
  int m;
  // entry owning CTA b: the last k < m with off(k) <= b
  template <int F>
  __device__ __forceinline__ int find(int b) const {
    int lo = 0, hi = m - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (entry_off<F>(e[mid]) <= b) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  }
  __device__ __forceinline__ const RelabelBox& get(int k) const { return boxes[e[k].box]; }
  template <int F>
  __device__ __forceinline__ int first(int k) const { return blockIdx.x - entry_off<F>(e[k]); }
  template <int F>
  __device__ __forceinline__ int stride(int k) const { return entry_off<F>(e[k + 1]) - entry_off<F>(e[k]); }
};

// --- 1: densities, labels inside each tile (8 x 8 threads, four cells each) ---
template <int S, class Src>
__global__ void __launch_bounds__(kTX / 4 * kTY, 16) kb_label(const __grid_constant__ Src src, int parity) {
  using T = typename Store<S>::T;
  const int k = src.template find<kTiles>(blockIdx.x);
  const RelabelBox& B = src.get(k);
  const int t = src.template first<kTiles>(k);
  grid_begin();
  const T* p = static_cast<const T*>(B.pops[B.cur ^ parity]);
  const int nx = B.nx, ny = B.ny;
  const int x = (t % B.ntx) * kTX + 4 * threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
  float2 fa[Q], fb[Q];  // cells (x, x + 1) and (x + 2, x + 3)
  pull4<S>(p, B.plane, B.pitch, B.wref, ny, x < nx ? x : 0, y < ny ? y : 0, fa, fb);
  const float2 ra = rho_pair(fa), rb = rho_pair(fb);
  const float r[4] = {ra.x, ra.y, rb.x, rb.y};
  bool in[4], gas[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    in[j] = y < ny && x + j < nx;
    gas[j] = in[j] && r[j] < B.threshold;
  }
  // whether the previous relabel may have left labels here. (Its gas flags
  // would say so too, but they are being written: reading them took the
  // relabel of 8192^2 from 645 us to 880.)
  const int before = B.tile_active[t];
  int32_t lab[4];
  const int any = tile_labels4(gas, x, y, nx, lab, B.flags);
  const size_t c = (size_t)(y < ny ? y : 0) * nx + x;
  int32_t* const label = B.label;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (gas[j]) {  // the label of the previous relabel, for the coalescence count
      const int32_t o = label[c + j];
      B.old[c + j] = o >= 0 ? o : 0x7fffffff;
    }
  if (any || before) {  // elsewhere the labels are -1 already
    if (in[3] && (nx & 3) == 0) {
      *reinterpret_cast<int4*>(label + c) = make_int4(lab[0], lab[1], lab[2], lab[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (in[j]) label[c + j] = lab[j];
    }
  }
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    B.tile_gas[t] = (uint8_t)(any != 0);
    if (t == 0) {  // what the next phases count up
      B.flags[FLAG_TILES] = 0;
      B.flags[FLAG_FILM] = 0;
      B.flags[FLAG_GAS] = 0;
    }
  }
}

// Position of a true predicate among the warp's, the counter advanced by one
// addition per warp (all lanes call).
__device__ __forceinline__ int warp_slot(bool want, int* counter) {
  const unsigned b = __ballot_sync(0xffffffffu, want);
  if (!b) return 0;
  const int lane = threadIdx.x & 31, lead = __ffs(b) - 1;
  int base = 0;
  if (lane == lead) base = atomicAdd(counter, __popc(b));
  return __shfl_sync(0xffffffffu, base, lead) + __popc(b & ((1u << lane) - 1u));
}

__device__ __forceinline__ int wrap_any(int a, int n) {
  a %= n;
  return a < 0 ? a + n : a;
}

// --- 2: tile lists (their order does not affect any result), borders joined ---
template <class Src>
__global__ void __launch_bounds__(32 * kScanTiles) kb_scan(const __grid_constant__ Src src) {
  __shared__ int gas_tiles[kScanTiles], ngas;
  const int k = src.template find<kScan>(blockIdx.x);
  const RelabelBox& B = src.get(k);
  const int ntx = B.ntx, nty = B.nty, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = src.template first<kScan>(k) * kScanTiles + lane;
  grid_begin();
  const bool in = t < ntx * nty;
  bool gas = false;
  if (warp == 0) {
    gas = in && B.tile_gas[t] != 0;
    const unsigned g = __ballot_sync(0xffffffffu, gas);
    if (gas) gas_tiles[__popc(g & ((1u << lane) - 1u))] = t;
    if (lane == 0) ngas = __popc(g);
  }
  __syncthreads();
  if (warp == 0) {  // the list, while the other warps unite
    int a = 0;
    if (in) {
      // tiles within reach of R cells; across the periodic seam of a box with a
      // ragged last tile one tile more
      const int spx = (B.R + kTX - 1) / kTX + (B.nx % kTX ? 1 : 0);
      const int spy = (B.R + kTY - 1) / kTY + (B.ny % kTY ? 1 : 0);
      const int ty = t / ntx, tx = t - ty * ntx;
      for (int dy = -spy; dy <= spy; ++dy) {
        const int row = wrap_any(ty + dy, nty) * ntx;
        for (int dx = -spx; dx <= spx; ++dx) a |= B.tile_gas[row + wrap_any(tx + dx, ntx)];
      }
      B.tile_active[t] = (uint8_t)(a != 0);
    }
    const bool visit = in && (a || B.tile_prev[t]);
    const int slot = warp_slot(visit, B.flags + FLAG_TILES);
    if (visit) B.tile_list[slot] = a ? t : ~t;
  }
  int fail = 0;
  const int warps = blockDim.x / 32;
  for (int w = warp == 0 ? warps - 1 : warp - 1; w < ngas; w += warps) {
    const int g = gas_tiles[w];
    tile_union_borders(B.label, (g % ntx) * kTX, (g / ntx) * kTY, B.nx, B.ny, lane, &fail);
  }
  if (fail) atomicOr(B.flags + FLAG_TIMEOUT, 1);
}

// Coalescence events (components of the new labelling holding gas of two or
// more components of the previous one). keep[r] of a new root r collects the
// first earlier label seen in its component (the root starts with its own);
// a member with another earlier label marks the component (-3), and the one
// that marks it first counts it, so every merged component counts once.
__device__ __forceinline__ int merge_vote(int32_t* keep, int r, int o) {
  if (o == 0x7fffffff) return 0;
  int prev = keep[r];  // a slot only goes from empty to a label to -3, so a value read late decides too
  if (prev == o || prev == -3) return 0;
  prev = atomicCAS(keep + r, 0x7fffffff, o);
  if (prev == 0x7fffffff || prev == o || prev == -3) return 0;
  return atomicExch(keep + r, -3) != -3;
}

// --- 3: final labels, votes, census; owners and rupture ---
// Label of the nearest labelled cell within R of a window position, -1 if
// none, -2 if two different labels are nearest at the same distance. Bit q of
// `row(dy)` says that the cell at dx = q - R of the row dy away is gas. Rows
// go outwards until they are further off than the nearest cell found.
template <typename RowBits>
__device__ __forceinline__ int nearest_label(const int* at, int W, int R, RowBits row) {
  const unsigned keep = (2u << (2 * R)) - 1u;
  int best = R * R, owner = -1;
  for (int d = 0; d * d <= best && d <= R; ++d) {
    for (int dy = -d; dy <= d; dy += max(2 * d, 1)) {
      const unsigned m = row(dy) & keep;
      if (!m) continue;
      const unsigned right = m >> R, left = m << (31 - R);  // bit 0, bit 31: dx = 0
      const int dr = right ? __ffs(right) - 1 : 64, dl = left ? __clz(left) : 64;
      const int dx = min(dr, dl), d2 = dx * dx + dy * dy;
      if (d2 > best) continue;
      if (d2 < best) owner = -1;
      best = d2;
      if (dr == dx) {
        const int l = at[dy * W + dx];
        owner = owner == -1 || owner == l ? l : -2;
      }
      if (dl == dx) {
        const int l = at[dy * W - dx];
        owner = owner == -1 || owner == l ? l : -2;
      }
    }
  }
  return owner;
}

// The same by a scan of the whole window (R = 16, whose rows have 33 cells).
__device__ __forceinline__ int window_owner(const int* at, int W, int R) {
  int best = -1, bd = 0x7fffffff;
  bool tie = false;
  for (int dy = -R; dy <= R; ++dy) {
    const int* rowp = at + dy * W;
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

// Pressure of cell (x, y) of the state the relabel sees (Eq. 29; two
// components: of the mixture).
template <int S, bool TWO>
__device__ __forceinline__ float pressure_at(const RelabelBox& B, const typename Store<S>::T* p, int x, int y) {
  const size_t P = (size_t)B.plane;
  const size_t r0 = (size_t)y * B.pitch + x, rm = (size_t)(y == 0 ? B.ny - 1 : y - 1) * B.pitch + x,
               rp = (size_t)(y == B.ny - 1 ? 0 : y + 1) * B.pitch + x;
  float f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i)
    f[i] = Store<S>::load(p - cx(i), (size_t)i * P + (cy(i) > 0 ? rm : (cy(i) < 0 ? rp : r0)), B.wref[i]);
  const float r = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
  if (TWO) {
    const float* pg = reinterpret_cast<const float*>(p) + (size_t)Q * P;
    float g = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) g += __ldcg(pg - cx(i) + ((size_t)i * P + (cy(i) > 0 ? rm : (cy(i) < 0 ? rp : r0))));
    const float a = B.rho0 * (1.0f - expf(-r / B.rho0)), b = B.rho0 * (1.0f - expf(-g / B.rho0));
    return (r + g) * (1.0f / 3.0f) + (B.G * a * a + 2.0f * B.G_mg * a * b + B.G_gg * b * b) * (1.0f / 6.0f);
  }
  const float s = B.rho0 * (1.0f - expf(-r / B.rho0));
  return r * (1.0f / 3.0f) + B.G * s * s * (1.0f / 6.0f);
}

template <int S, bool TWO, class Src>
__global__ void __launch_bounds__(kTileThreads, 5) kb_zone(const __grid_constant__ Src src, int parity) {
  using T = typename Store<S>::T;
  constexpr int MW = kTX + 2 + 2 * kMaxR, MH = kTY + 2 + 2 * kMaxR;  // largest window
  __shared__ int32_t win[MH * MW];
  __shared__ unsigned bits[MH][4];  // gas of each window row (the last word zero)
  __shared__ int own[kTY + 2][kTX + 2];
  const int k = src.template find<kList>(blockIdx.x);
  const RelabelBox& B = src.get(k);
  const int first = src.template first<kList>(k), step = src.template stride<kList>(k);
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  grid_begin();
  const T* p = static_cast<const T*>(B.pops[B.cur ^ parity]);
  const int nx = B.nx, ny = B.ny, R = B.R, n = B.flags[FLAG_TILES];
  const int W = kTX + 2 + 2 * R, H = kTY + 2 + 2 * R;
  const int32_t* L = B.label;
  const int head = B.tile_list[first];  // along with n: garbage, and unused, where first >= n
  int fail = 0, merged = 0, opened = 0;
  for (int w = first; w < n; w += step) {
    const int entry = w == first ? head : B.tile_list[w];
    const bool act = entry >= 0;
    const int t = act ? entry : ~entry;
    const int x0 = (t % B.ntx) * kTX, y0 = (t / B.ntx) * kTY;
    const int x = x0 + lane, y = y0 + warp;
    const bool in = x < nx && y < ny;
    const int c = y * nx + x;
    bool any = false;
    // this cell's own state, on its way while the window is
    const int was = act && in ? B.old[c] : 0, prevs = act && in ? B.sgn[c] : 0, open = act && in ? B.open[c] : 0;
    if (act) {
      for (int yb = warp; yb < H; yb += 3 * kTileWarps) {  // six loads in flight (R = 4: the whole window)
        for (int q = 0; 32 * q < W; q += 2) {
          int l[3][2];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            // (beyond a ragged end of a tiny box the window may go round
            // twice: no cell of the box looks there)
            const int yy = yb + k * kTileWarps, row = min(wrap1(y0 - R - 1 + yy, ny), ny - 1) * nx;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int xx = 32 * (q + u) + lane;
              l[k][u] = yy < H && xx < W ? L[row + min(wrap1(x0 - R - 1 + xx, nx), nx - 1)] : -1;
            }
          }
          // every label to its root, the six walks side by side
          bool walk = true;
          for (int it = 0; walk && it < kUnionIters; ++it) {
            walk = false;
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int up = l[k][u] >= 0 ? L[l[k][u]] : -1;
                walk |= up != l[k][u];
                l[k][u] = up;
              }
          }
          if (walk) fail = 1;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const int yy = yb + k * kTileWarps;
            if (yy >= H) break;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int xx = 32 * (q + u) + lane;
              if (xx < W) win[yy * W + xx] = l[k][u];
              const unsigned b = __ballot_sync(0xffffffffu, l[k][u] >= 0);
              if (lane == 0 && q + u < 4) bits[yy][q + u] = b;
              any |= b != 0;
            }
            if (lane == 0 && q == 0) bits[yy][2] = 0u;  // (W <= 64; the wider ones write it next)
          }
        }
      }
    }
    // (also: the previous tile's window and owners are no longer read)
    any = __syncthreads_or(any);
    if (tid == 0) B.tile_prev[t] = (uint8_t)act;  // for the scan of the next relabel
    uint8_t* const mrow = B.mask + (size_t)y * B.mpitch;
    if (!any) {  // no gas in reach, or it went quiet since the previous relabel
      if (in) {
        B.owner[c] = -1;
        B.sgn[c] = 0;
        put_cell(mrow, x, nx, (uint8_t)0);
      }
      continue;
    }
    const int root = in ? win[(warp + R + 1) * W + lane + R + 1] : -1;
    if (root >= 0) {
      B.label[c] = root;
      if (root != c) merged += merge_vote(B.old, root, was);
    }
    if (B.gas_list) {
      const int slot = warp_slot(root >= 0, B.flags + FLAG_GAS);
      if (root >= 0) B.gas_list[slot] = c;
    }
    for (int q = tid; q < (kTX + 2) * (kTY + 2); q += kTileThreads) {
      const int oy = q / (kTX + 2), ox = q - oy * (kTX + 2);
      const int* at = win + (oy + R) * W + ox + R;
      int o = *at;
      if (o < 0) {
        // columns ox .. ox + 2 R of the window rows oy + R + dy
        auto row = [&](int dy) {
          const unsigned* rb = bits[oy + R + dy];
          return __funnelshift_r(rb[ox >> 5], rb[(ox >> 5) + 1], ox & 31);
        };
        if (R == 4) o = nearest_label(at, W, 4, row);  // the default zone radius
        else if (R < kMaxR) o = nearest_label(at, W, R, row);
        else o = window_owner(at, W, R);
      }
      own[oy][ox] = o;
    }
    __syncthreads();
    const int o = own[warp + 1][lane + 1];
    int dir = 0;
    if (o != -1) {
#pragma unroll
      for (int i = Q - 1; i >= 1; --i) {  // the first direction with another owner
        const int on = own[warp + 1 + cy(i)][lane + 1 + cx(i)];
        if (on != -1 && on != o) dir = i;
      }
    }
    if (in) {
      B.owner[c] = o;
      if (dir == 0) {
        B.sgn[c] = 0;
      } else {
        int ex = 0, ey = 0;
#pragma unroll
        for (int i = 1; i < Q; ++i)
          if (i == dir) {
            ex = cx(i);
            ey = cy(i);
          }
        const float pp = pressure_at<S, TWO>(B, p, wrap1(x + ex, nx), wrap1(y + ey, ny));
        const float p0 = pressure_at<S, TWO>(B, p, x, y);
        const float pm = pressure_at<S, TWO>(B, p, wrap1(x - ex, nx), wrap1(y - ey, ny));
        const float d2 = pp - 2.0f * p0 + pm;
        const int sg = (d2 > 0.f) - (d2 < 0.f);
        if (B.eps >= 0.f && !open && (fabsf(d2) <= B.eps || (prevs != 0 && sg != prevs))) {
          B.open[c] = 1;
          ++opened;
        }
        B.sgn[c] = (int8_t)sg;
      }
    }
    // tiles where owners meet go to the list of the mask and the bounce-back
    const int film = __syncthreads_or(in && dir != 0);
    if (film) {
      if (tid == 0) B.film_list[atomicAdd(B.flags + FLAG_FILM, 1)] = t;
    } else if (in) {
      put_cell(mrow, x, nx, (uint8_t)0);
    }
  }
  merged = __reduce_add_sync(0xffffffffu, merged);
  opened = __reduce_add_sync(0xffffffffu, opened);
  if (merged && lane == 0) atomicAdd(B.flags + FLAG_MERGES, merged);
  if (opened && lane == 0) atomicAdd(B.flags + FLAG_OPENED, opened);
  if (fail) atomicOr(B.flags + FLAG_TIMEOUT, 1);
}

// --- 4: the mask of the film tiles (it needs the neighbours' opened cells, so
// it is a launch of its own; everywhere else the zone phase wrote zeros) ---
template <class Src>
__global__ void __launch_bounds__(kTileThreads) kb_mask(const __grid_constant__ Src src) {
  const int k = src.template find<kFilm>(blockIdx.x);
  const RelabelBox& B = src.get(k);
  const int first = src.template first<kFilm>(k), step = src.template stride<kFilm>(k);
  grid_begin();
  const int nx = B.nx, ny = B.ny, n = B.flags[FLAG_FILM];
  for (int w = first; w < n; w += step) {
    const int t = B.film_list[w];
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    if (x >= nx || y >= ny) continue;
    const size_t c = (size_t)y * nx + x;
    unsigned msk = 0;
    const int o = B.owner[c];
    if (o != -1 && !B.open[c]) {
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const size_t nb = (size_t)wrap1(y + cy(i), ny) * nx + wrap1(x + cx(i), nx);
        const int on = B.owner[nb];
        if (on != -1 && on != o && !B.open[nb]) msk |= 1u << (i - 1);
      }
    }
    put_cell(B.mask + (size_t)y * B.mpitch, x, nx, (uint8_t)msk);
  }
}

// Bounce-back over the film tiles of the latest relabel, on buffer
// B.pops[B.cur ^ q].
template <typename T, bool TWO, class Src>
__global__ void __launch_bounds__(kTileThreads) kb_bounce(const __grid_constant__ Src src, int q) {
  const int k = src.template find<kFilm>(blockIdx.x);
  const RelabelBox& B = src.get(k);
  const int first = src.template first<kFilm>(k), step = src.template stride<kFilm>(k);
  grid_begin();
  T* pops = static_cast<T*>(const_cast<void*>(B.pops[B.cur ^ q]));
  const int n = B.flags[FLAG_FILM];
  for (int w = first; w < n; w += step) {
    const int t = B.film_list[w];
    const int x = (t % B.ntx) * kTX + threadIdx.x, y = (t / B.ntx) * kTY + threadIdx.y;
    if (x >= B.nx || y >= B.ny) continue;
    const unsigned msk = B.mask[(size_t)y * B.mpitch + x];
    if (msk & kCanonBits) bounce_cell<T, TWO>(pops, (size_t)B.plane, B.pitch, x, y, B.nx, B.ny, msk);
  }
}

template <class Src>
cudaError_t launch_relabel(int storage, const Src& src, const RelabelEntry& total, int parity, bool two, cudaStream_t s) {
  const dim3 quad(kTX / 4, kTY), tile(kTX, kTY);
  if (two && storage != LBM_F32) return cudaErrorInvalidValue;
#define CALL(S) LBM_TRY(launch_chain(kb_label<S, Src>, dim3(total.off_tiles), quad, 0, s, src, parity))
  switch (storage) {
    case LBM_F32: CALL(LBM_F32); break;
    case LBM_F16_DEV: CALL(LBM_F16_DEV); break;
    case LBM_BF16_DEV: CALL(LBM_BF16_DEV); break;
    default: return cudaErrorInvalidValue;
  }
#undef CALL
  // a warp per tile while the grid is small (the unions of a CTA's tiles are a
  // serial chain then), four warps beyond
  const dim3 scan(total.off_scan <= 2 * device_sm_count() ? 32 * kScanTiles : 128);
  LBM_TRY(launch_chain(kb_scan<Src>, dim3(total.off_scan), scan, 0, s, src));
#define CALL(S, TWO) LBM_TRY(launch_chain(kb_zone<S, TWO, Src>, dim3(total.off_list), tile, 0, s, src, parity))
  switch (storage) {
    case LBM_F32:
      if (two) CALL(LBM_F32, true);
      else CALL(LBM_F32, false);
      break;
    case LBM_F16_DEV: CALL(LBM_F16_DEV, false); break;
    default: CALL(LBM_BF16_DEV, false); break;
  }
#undef CALL
  return launch_chain(kb_mask<Src>, dim3(total.off_film), tile, 0, s, src);
}

template <class Src>
cudaError_t launch_bounce_src(int storage, const Src& src, int ctas, int q, bool two, cudaStream_t s) {
  const dim3 grid(ctas), tile(kTX, kTY);
  if (two && storage != LBM_F32) return cudaErrorInvalidValue;
  if (two) return launch_chain(kb_bounce<uint32_t, true, Src>, grid, tile, 0, s, src, q);
  if (storage == LBM_F32) return launch_chain(kb_bounce<uint32_t, false, Src>, grid, tile, 0, s, src, q);
  return launch_chain(kb_bounce<uint16_t, false, Src>, grid, tile, 0, s, src, q);
}

}  // namespace

bool relabel_tiled_ok(int nx, int ny, int R) { return nx > 2 * R && ny > 2 * R && R <= kMaxR; }

int relabel_tile_count(int nx, int ny) { return ((nx + kTX - 1) / kTX) * ((ny + kTY - 1) / kTY); }

RelabelEntry relabel_entry_sizes(int nx, int ny) {
  RelabelEntry e{};
  const int t = relabel_tile_count(nx, ny), cap = device_sm_count() * 8;
  auto share = [&](int least, int part, int most) { return std::min(std::min(t, most), std::max(least, t / part)); };
  e.off_tiles = t;
  e.off_scan = (t + kScanTiles - 1) / kScanTiles;
  // the listed tiles are a few to a few tens of percent of a large box
  e.off_list = share(64, 8, cap);
  e.off_film = share(64, 64, cap / 4);
  return e;
}

cudaError_t launch_relabel_lone(int storage, const RelabelBox& box, bool two, cudaStream_t s) {
  return launch_relabel(storage, Lone{box}, relabel_entry_sizes(box.nx, box.ny), 0, two, s);
}

cudaError_t launch_relabel_boxes(int storage, const RelabelBox* boxes, const RelabelEntry* entries, int m,
                                 const RelabelEntry& totals, int parity, cudaStream_t s) {
  if (m <= 0) return cudaSuccess;
  return launch_relabel(storage, Many{boxes, entries, m}, totals, parity, false, s);
}

cudaError_t launch_bounce_lone(int storage, const RelabelBox& box, bool two, cudaStream_t s) {
  return launch_bounce_src(storage, Lone{box}, relabel_entry_sizes(box.nx, box.ny).off_film, 0, two, s);
}

cudaError_t launch_bounce_boxes(int storage, const RelabelBox* boxes, const RelabelEntry* entries, int m, int ctas,
                                int q, cudaStream_t s) {
  if (m <= 0 || ctas <= 0) return cudaSuccess;
  return launch_bounce_src(storage, Many{boxes, entries, m}, ctas, q, false, s);
}

}  // namespace lbm
