// Film-barrier pipeline of the extended Shan-Chen model (arXiv 1708.01613,
// Sec. 2.1.5) for boxes with R_z > 16: gas labelling, interaction zones, rupture
// test (Eq. 41), blocked-edge mask, bounce-back, over every cell of the box
// (relabel.cu does the same over tiles near gas for R_z <= 16); and the
// initialisation of a box. The diagnostics are in fields.cu.
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

#include "bounce.cuh"
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
// Each new gas cell parks its label of the previous relabel in keep[c] (INT_MAX
// where it was liquid) for the coalescence count; keep is the owner array, which
// the owner phase rewrites afterwards.
__global__ void k_label_init(const float* __restrict__ rho, long long N, float th, int32_t* L,
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

}  // namespace

cudaError_t launch_labels(const FieldParams& fp, const float* rho, float threshold, int32_t* label,
                          int* flags, cudaStream_t s, int32_t* keep) {
  const unsigned b = blocks_for(fp.N);
  k_label_init<<<b, kThreads, 0, s>>>(rho, fp.N, threshold, label, keep);
  k_label_union<<<b, kThreads, 0, s>>>(fp.nx, fp.ny, label, flags);
  k_label_flatten<<<b, kThreads, 0, s>>>(fp.N, label, flags);
  k_merge_count<<<b, kThreads, 0, s>>>(fp.N, label, keep, flags);
  return cudaGetLastError();
}

cudaError_t launch_owner(int nx, int ny, int R, const int32_t* label, int32_t* owner, cudaStream_t s) {
  k_owner<<<blocks_for((long long)nx * ny), kThreads, 0, s>>>(nx, ny, R, label, owner);
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

}  // namespace lbm
