// Diagnostics of a state: fields, populations, FP64 mass, gas labels, bubble
// statistics and areas (arXiv 1708.01613, Eqs. 11, 29; Sec. 5 statistics).
//
// Every one of these is bound by memory, so each reads the populations once
// and keeps what it needs on the chip:
//  - the fields rho, u and p come from one pass that forms the densities of a
//    tile with its halo in shared memory (4096^2 FP32 all four 190 us; a pass per
//    field after a density pass takes 730);
//  - all population planes are written by one launch, rows by grid
//    coordinates (no division per cell);
//  - labels, areas, statistics and the mass come from one density pass over
//    32 x 8 tiles that joins the gas cells of each tile in shared memory and
//    flags the tiles holding gas; the passes after it visit only those.
#include <math.h>

#include <algorithm>

#include "cellmath.cuh"
#include "labels.cuh"
#include "pull.cuh"

namespace lbm {
namespace {

constexpr int kThreads = 256;

// --- densities (untiled relabel, growth census without the barrier) ---
constexpr int kRows = 4;  // rows per thread of the row kernels: four cells' loads in flight

template <int S>
__global__ void __launch_bounds__(kThreads) k_density(const FieldParams fp, float* __restrict__ rho) {
  using T = typename Store<S>::T;
  const T* p = static_cast<const T*>(fp.pops);
  const int nx = fp.nx, ny = fp.ny;
  const int x = blockIdx.x * kThreads + threadIdx.x;
  if (x >= nx) return;
  for (int yb = blockIdx.y * kRows; yb < ny; yb += gridDim.y * kRows) {
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const int y = yb + r;
      if (y >= ny) break;
      float f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const int ys = cy(i) > 0 ? pull_wrap(y - 1, ny) : (cy(i) < 0 ? pull_wrap(y + 1, ny) : y);
        f[i] = Store<S>::load(p + (x - cx(i)), (size_t)i * fp.plane + (size_t)ys * fp.pitch, fp.wref[i]);
      }
      rho[(size_t)y * nx + x] = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
    }
  }
}

// --- populations: plane i of the incoming state, f_i(x) = B_i(x - e_i) ---
// Four columns of a few rows per thread. The source row's four columns start
// at x - e_x: an aligned vector load, and the word beside it for a shifted
// plane. Dense output rows of a width that is not a multiple of four are
// written one value at a time. Bound by HBM (FP32) and by bytes in flight
// (16-bit words: 8192^2 with 1, 2, 4, 8 rows 2001, 1183, 811, 1060 us, FP32
// 804, 772, 881, 1175). All planes of 8192^2 take 772 us (FP32, 6.3 TB/s) and
// 811 us (FP16; 861 without the streaming hint, which costs FP32 nothing and
// gives it nothing); a launch per plane with a 64-bit division per cell takes 2452
// and 2330 us.
template <int S>
constexpr int pop_rows() {
  return S == LBM_F32 ? 2 : 4;
}

template <int S>
__device__ __forceinline__ float4 load4(const typename Store<S>::T* q, int ex, float base) {
  if constexpr (S == LBM_F32) {
    const float4 w = __ldg(reinterpret_cast<const float4*>(q));
    if (ex > 0) return make_float4(__ldg(q - 1), w.x, w.y, w.z);
    if (ex < 0) return make_float4(w.y, w.z, w.w, __ldg(q + 4));
    return w;
  } else {
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(q));
    uint32_t lo = w.x, hi = w.y;
    if (ex > 0) {
      lo = __byte_perm(__ldg(reinterpret_cast<const uint32_t*>(q - 2)), w.x, 0x5432);
      hi = __byte_perm(w.x, w.y, 0x5432);
    } else if (ex < 0) {
      lo = __byte_perm(w.x, w.y, 0x5432);
      hi = __byte_perm(w.y, __ldg(reinterpret_cast<const uint32_t*>(q + 4)), 0x5432);
    }
    const float2 wr = make_float2(base, base), a = __fadd2_rn(wr, dec16x2<S>(lo)), b = __fadd2_rn(wr, dec16x2<S>(hi));
    return make_float4(a.x, a.y, b.x, b.y);
  }
}

template <int S>
__global__ void __launch_bounds__(kThreads) k_pops_out(const FieldParams fp, int plane0, bool vec,
                                                       float* __restrict__ out) {
  using T = typename Store<S>::T;
  constexpr int ROWS = pop_rows<S>();
  const int nx = fp.nx, ny = fp.ny;
  const int x = 4 * (blockIdx.x * kThreads + threadIdx.x);
  if (x >= nx) return;
  const int i = plane0 + blockIdx.z;
  const int ex = (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
  const int ey = (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
  const T* p = static_cast<const T*>(fp.pops) + (size_t)i * fp.plane + x;
  float* o = out + (size_t)blockIdx.z * fp.N + x;
  const float base = fp.wref[i];
  for (int yb = blockIdx.y * ROWS; yb < ny; yb += gridDim.y * ROWS) {
    float4 v[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
      if (yb + r < ny) v[r] = load4<S>(p + (size_t)pull_wrap(yb + r - ey, ny) * fp.pitch, ex, base);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      if (yb + r >= ny) continue;
      float* q = o + (size_t)(yb + r) * nx;
      if (vec) {
        if (S == LBM_F32) *reinterpret_cast<float4*>(q) = v[r];
        else __stcs(reinterpret_cast<float4*>(q), v[r]);
      } else {
        q[0] = v[r].x;
        if (x + 1 < nx) q[1] = v[r].y;
        if (x + 2 < nx) q[2] = v[r].z;
        if (x + 3 < nx) q[3] = v[r].w;
      }
    }
  }
}

// --- mask: its rows without their padding, 16 cells per thread ---
// (8192^2 20 us; a 2-D device copy takes 67.)
__global__ void __launch_bounds__(kThreads) k_mask_out(const uint8_t* __restrict__ mask, int mpitch, int nx, int ny,
                                                       int vec, uint8_t* __restrict__ out) {
  const int x = 16 * (blockIdx.x * kThreads + threadIdx.x);
  if (x >= nx) return;
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    const uint4 v = *reinterpret_cast<const uint4*>(mask + (size_t)y * mpitch + x);
    uint8_t* q = out + (size_t)y * nx + x;
    if (vec == 16) {
      *reinterpret_cast<uint4*>(q) = v;
      continue;
    }
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (vec == 4 && x + 4 * k + 4 <= nx) {
        *reinterpret_cast<uint32_t*>(q + 4 * k) = w[k];
      } else {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (x + 4 * k + b < nx) q[4 * k + b] = (uint8_t)(w[k] >> (8 * b));
      }
    }
  }
}

// --- rho, u = (j + F/2)/rho, p (Eq. 29): any of the four in one pass ---
// A 64 x 8 tile per CTA, two cells per thread. With a velocity asked for, the
// CTA also forms the densities of the tile's one-cell halo (148 cells beside
// 512) and shares psi; without one, nothing is shared.
constexpr int kFX = 64, kFY = 8;

template <int S>
__device__ __forceinline__ float pulled9(const FieldParams& fp, int x, int y, float (&f)[Q]) {
  using T = typename Store<S>::T;
  const T* p = static_cast<const T*>(fp.pops);
  const int ny = fp.ny;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int ys = pull_wrap(y - cy(i), ny);
    f[i] = Store<S>::load(p + (x - cx(i)), (size_t)i * fp.plane + (size_t)ys * fp.pitch, fp.wref[i]);
  }
  return ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
}

template <int S, bool VEL>
__global__ void __launch_bounds__(kThreads) k_fields(const FieldParams fp, const uint8_t* __restrict__ mask,
                                                     const FieldOuts out) {
  __shared__ float psi[VEL ? kFY + 2 : 1][VEL ? kFX + 2 : 1];
  const int nx = fp.nx, ny = fp.ny;
  const int ntx = (nx + kFX - 1) / kFX;
  const int x0 = (int)(blockIdx.x % ntx) * kFX, y0 = (int)(blockIdx.x / ntx) * kFY;
  const int lx = threadIdx.x % kFX, ly = threadIdx.x / kFX;  // cells (lx, ly) and (lx, ly + 4)
  float rho[2], jx[2], jy[2], ps[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int x = x0 + lx, y = y0 + ly + 4 * q;
    if (x >= nx || y >= ny) continue;
    float f[Q];
    const float r = pulled9<S>(fp, x, y, f);
    rho[q] = r;
    jx[q] = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
    jy[q] = (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7]);
    ps[q] = fp.rho0 * (1.0f - expf(-r * fp.inv_rho0));
    if (VEL) psi[ly + 4 * q + 1][lx + 1] = ps[q];
  }
  if (VEL) {
    // the halo of the cells inside the box: rows -1 and h, columns -1 and w
    const int w = min(kFX, nx - x0), h = min(kFY, ny - y0);
    const int n = 2 * (w + 2) + 2 * h;
    for (int k = threadIdx.x; k < n; k += kThreads) {
      int hx, hy;
      if (k < 2 * (w + 2)) {
        hy = k < w + 2 ? -1 : h;
        hx = (k < w + 2 ? k : k - (w + 2)) - 1;
      } else {
        const int m = k - 2 * (w + 2);
        hx = m < h ? -1 : w;
        hy = m < h ? m : m - h;
      }
      float f[Q];
      const float r = pulled9<S>(fp, pull_wrap(x0 + hx, nx), pull_wrap(y0 + hy, ny), f);
      psi[hy + 1][hx + 1] = fp.rho0 * (1.0f - expf(-r * fp.inv_rho0));
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int x = x0 + lx, y = y0 + ly + 4 * q;
    if (x >= nx || y >= ny) continue;
    const size_t c = (size_t)y * nx + x;
    const float r = rho[q], psi_c = ps[q];
    if (out.rho) out.rho[c] = r;
    if (out.p) out.p[c] = r * (1.0f / 3.0f) + fp.G * psi_c * psi_c * (1.0f / 6.0f);
    if (VEL) {
      const unsigned m = mask ? mask[(size_t)y * fp.mpitch + x] : 0u;
      float sx = 0.f, sy = 0.f;
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        float s = psi[ly + 4 * q + 1 + cy(i)][lx + 1 + cx(i)];
        if ((m >> (i - 1)) & 1u) s = psi_c;
        // explicit roundings: left to the compiler, a component asked for
        // without the other is contracted differently and rounds differently
        if (i < 5) {
          const float t = __fmul_rn(wqf(i), s);
          sx = __fmaf_rn(t, (float)cx(i), sx);
          sy = __fmaf_rn(t, (float)cy(i), sy);
        } else {
          sx = __fmaf_rn(wqf(i) * cx(i), s, sx);
          sy = __fmaf_rn(wqf(i) * cy(i), s, sy);
        }
      }
      const float g = -fp.G * psi_c;
      if (out.ux) out.ux[c] = (jx[q] + 0.5f * (g * sx)) / r;
      if (out.uy) out.uy[c] = (jy[q] + 0.5f * (g * sy)) / r;
    }
  }
}

// --- FP64 sums of FP32 values ---
// A running sum as an unevaluated triple s + e + r of FP32 values: s takes the
// values, e the rounding error of every addition to s and r that of every
// addition to e, both exact (Knuth's TwoSum; the cascade is the K-fold summation
// of Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26, 2005). A chain of n
// additions is within n^3 2^-72 of the sum of the magnitudes (n is 24 at most
// here: 2^-58), less than the rounding of one FP64 addition. FP64 adds run at
// 1/64 of the FP32 rate here: one per value took 0.61 ms at 4096^2 (FP32
// storage) where the bytes take 0.09 ms. With V = float2 two sums run side by
// side in packed instructions (6.5 per value): the statistics of 4096^2 take 236
// us (FP32) and 235 (FP16, whose density pass they bound), those of 8192^2 656
// and 651; a pair s + e, which loses what e cannot hold, took 233, 202, 634 and
// 532. A sum that leaves the FP32 range or meets an infinity or NaN is no longer
// finite, and its values are added in FP64 instead.
template <typename V>
struct Sum3 {
  V s{}, e{}, r{};
  // a + b rounded, and its error
  static __device__ __forceinline__ V two_sum(V a, V b, V& err) {
    using O = VOps<V>;
    const V t = O::add(a, b), z = O::sub(t, a);
    err = O::add(O::sub(a, O::sub(t, z)), O::sub(b, z));
    return t;
  }
  __device__ __forceinline__ void add_error(V q) {
    V d;
    e = two_sum(e, q, d);
    r = VOps<V>::add(r, d);
  }
  __device__ __forceinline__ void add(V b) {
    V q;
    s = two_sum(s, b, q);
    add_error(q);
  }
  __device__ __forceinline__ void add(const Sum3& o) {
    add(o.s);
    add_error(o.e);
    r = VOps<V>::add(r, o.r);
  }
};

__device__ __forceinline__ Sum3<float> both(const Sum3<float2>& p) {
  Sum3<float> a, b;
  a.s = p.s.x, a.e = p.e.x, a.r = p.r.x;
  b.s = p.s.y, b.e = p.e.y, b.r = p.r.y;
  a.add(b);
  return a;
}
__device__ __forceinline__ bool finite(const Sum3<float>& a) { return fabsf(a.s) < INFINITY; }
__device__ __forceinline__ double value(const Sum3<float>& a) { return (double)a.s + ((double)a.e + (double)a.r); }

// Sum of a sum over the warp, in a fixed order (valid in lane 0).
__device__ __forceinline__ Sum3<float> warp_sum(Sum3<float> a) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    Sum3<float> b;
    b.s = __shfl_down_sync(0xffffffffu, a.s, d);
    b.e = __shfl_down_sync(0xffffffffu, a.e, d);
    b.r = __shfl_down_sync(0xffffffffu, a.r, d);
    a.add(b);
  }
  return a;
}

// FP64 sum of the populations of the cells (x .. x + n, y).
template <int S>
__device__ __forceinline__ double cells_sum64(const FieldParams& fp, int x, int y, int n) {
  using T = typename Store<S>::T;
  double sum = 0.0;
#pragma unroll 1
  for (int i = 0; i < Q; ++i) {
    const T* row = static_cast<const T*>(fp.pops) + (size_t)i * fp.plane + (size_t)pull_wrap(y - cy(i), fp.ny) * fp.pitch;
#pragma unroll 1
    for (int j = 0; j < n; ++j) sum += (double)Store<S>::load(row + (x + j - cx(i)), 0, fp.wref[i]);
  }
  return sum;
}

// --- fixed-order FP64 reductions ---
// A fixed number of block partials (not tied to the device's SM count), so the
// summation order, and with it every reduced value, is the same on any GPU.
constexpr int kRedBlocks = 608;

template <int NV>
__device__ void block_reduce_store(double (&v)[NV], double* __restrict__ out) {
  __shared__ double sh[NV][kThreads];
#pragma unroll
  for (int j = 0; j < NV; ++j) sh[j][threadIdx.x] = v[j];
  __syncthreads();
  for (int s = kThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
#pragma unroll
      for (int j = 0; j < NV; ++j) sh[j][threadIdx.x] += sh[j][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int j = 0; j < NV; ++j) out[j * gridDim.x + blockIdx.x] = sh[j][0];
}

// Sum of all stored populations: rows of one plane after another, eight
// values of a row in flight per thread (8192^2 FP32 562 us, FP16 575; with the
// four rows' 32 values loaded first 480 and 1043).
template <int S>
__global__ void __launch_bounds__(kThreads) k_mass_partial(const __grid_constant__ FieldParams fp, double* partials) {
  using T = typename Store<S>::T;
  const T* p = static_cast<const T*>(fp.pops);
  const long long rows = (long long)Q * fp.ny;
  double acc[1] = {0.0};
  for (long long r0 = (long long)blockIdx.x * kRows; r0 < rows; r0 += (long long)gridDim.x * kRows) {
    for (int xb = 0; xb < fp.nx; xb += 8 * kThreads) {
      const int x = xb + threadIdx.x;
      auto row_at = [&](int r, float& base) {  // column 0 of the r-th row, nullptr beyond the last
        const long long row = r0 + r;
        const int i = (int)(row / fp.ny);
        base = fp.wref[i < Q ? i : 0];
        return row < rows ? p + (size_t)i * fp.plane + (size_t)(row - (long long)i * fp.ny) * fp.pitch : nullptr;
      };
      Sum3<float2> pair;
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        float base, v[8];
        const T* q = row_at(r, base);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          v[k] = q && x + k * kThreads < fp.nx ? Store<S>::load(q, (size_t)(x + k * kThreads), base) : 0.f;
#pragma unroll
        for (int k = 0; k < 8; k += 2) pair.add(make_float2(v[k], v[k + 1]));
      }
      const Sum3<float> a = both(pair);
      if (finite(a)) {
        acc[0] += value(a);
      } else {
#pragma unroll 1
        for (int r = 0; r < kRows; ++r) {
          float base;
          const T* q = row_at(r, base);
#pragma unroll 1
          for (int k = 0; q && k < 8 && x + k * kThreads < fp.nx; ++k)
            acc[0] += (double)Store<S>::load(q, (size_t)(x + k * kThreads), base);
        }
      }
    }
  }
  block_reduce_store<1>(acc, partials);
}

template <int NV>
__global__ void __launch_bounds__(kThreads) k_sum_partials(const double* partials, int nparts, double* out) {
  double acc[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) acc[j] = 0.0;
  for (int k = threadIdx.x; k < nparts; k += blockDim.x)
#pragma unroll
    for (int j = 0; j < NV; ++j) acc[j] += partials[j * nparts + k];
  block_reduce_store<NV>(acc, out);
}

// --- labels, areas, statistics ---
// Density pass over 32 x 8 tiles (8 x 8 threads, four cells each): the labels
// of each tile's own gas pieces (the smallest index of the piece), one gas
// flag per tile; with AREA the area slots of its gas cells cleared; with MASS
// the FP64 sum of the tile's populations.
template <int S, bool AREA, bool MASS>
__global__ void __launch_bounds__(kTX / 4 * kTY, MASS ? 16 : 0) kd_label(const __grid_constant__ FieldParams fp, float threshold, bool vec4,
                                                          int32_t* __restrict__ label, int32_t* __restrict__ area,
                                                          uint8_t* __restrict__ tile_gas, double* __restrict__ tile_mass,
                                                          int* __restrict__ flags) {
  using T = typename Store<S>::T;
  const int nx = fp.nx, ny = fp.ny;
  const int ntx = (nx + kTX - 1) / kTX, t = blockIdx.x;
  const int x = (t % ntx) * kTX + 4 * threadIdx.x, y = (t / ntx) * kTY + threadIdx.y;
  float2 fa[Q], fb[Q];
  pull4<S>(static_cast<const T*>(fp.pops), fp.plane, fp.pitch, fp.wref, ny, x < nx ? x : 0, y < ny ? y : 0, fa, fb);
  const float2 ra = rho_pair(fa), rb = rho_pair(fb);
  const float r[4] = {ra.x, ra.y, rb.x, rb.y};
  const bool rowin = y < ny;
  bool in[4], gas[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    in[j] = rowin && x + j < nx;
    gas[j] = in[j] && r[j] < threshold;
  }
  if (MASS) {
    Sum3<float2> pair;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      pair.add(make_float2(in[0] ? fa[i].x : 0.f, in[1] ? fa[i].y : 0.f));
      pair.add(make_float2(in[2] ? fb[i].x : 0.f, in[3] ? fb[i].y : 0.f));
    }
    __shared__ double wm[2];
    const Sum3<float> a = warp_sum(both(pair));
    double v = value(a);
    if (!__shfl_sync(0xffffffffu, finite(a), 0)) {
      v = in[0] ? cells_sum64<S>(fp, x, y, min(4, nx - x)) : 0.0;
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    }
    const int tid = threadIdx.y * (kTX / 4) + threadIdx.x;
    if ((tid & 31) == 0) wm[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) tile_mass[t] = wm[0] + wm[1];
  }
  int32_t lab[4];
  const int any = tile_labels4(gas, x, y, nx, lab, flags);
  const size_t c = (size_t)y * nx + x;
  if (vec4 && in[3]) {
    *reinterpret_cast<int4*>(label + c) = make_int4(lab[0], lab[1], lab[2], lab[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (in[j]) label[c + j] = lab[j];
  }
  if (AREA)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (gas[j]) area[c + j] = 0;
  if (threadIdx.x == 0 && threadIdx.y == 0) tile_gas[t] = (uint8_t)(any != 0);
}

// One warp per tile with gas: its right and bottom borders joined to the
// neighbouring tiles (periodic wrap included).
constexpr int kTileWarps = 8;

__global__ void __launch_bounds__(32 * kTileWarps) kd_union(int nx, int ny, int ntx, int ntiles,
                                                            const uint8_t* __restrict__ tile_gas, int32_t* L,
                                                            int* __restrict__ flags) {
  int fail = 0;
  for (int t = blockIdx.x * kTileWarps + (threadIdx.x >> 5); t < ntiles; t += gridDim.x * kTileWarps)
    if (tile_gas[t]) tile_union_borders(L, (t % ntx) * kTX, (t / ntx) * kTY, nx, ny, threadIdx.x & 31, &fail);
  if (fail) atomicOr(flags + FLAG_TIMEOUT, 1);
}

// Final labels of the gas tiles; with AREA the cells counted per root, one
// atomic for the cells of a warp's row that share a root.
template <bool AREA>
__global__ void __launch_bounds__(32 * kTileWarps) kd_flatten(int nx, int ny, int ntx, int ntiles,
                                                              const uint8_t* __restrict__ tile_gas, int32_t* L,
                                                              int32_t* __restrict__ area, int* __restrict__ flags) {
  int fail = 0;
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x * kTileWarps + (threadIdx.x >> 5); t < ntiles; t += gridDim.x * kTileWarps) {
    if (!tile_gas[t]) continue;
    const int x = (t % ntx) * kTX + lane, y0 = (t / ntx) * kTY;
    int run = -1, n = 0;  // cells of this column so far that share the root `run`
    for (int j = 0; j < kTY; ++j) {
      const int y = y0 + j;
      const int c = y * nx + x;
      int r = -1;
      if (x < nx && y < ny && L[c] >= 0) {
        r = find_root(L, c, &fail);
        L[c] = r;
      }
      if (AREA && r >= 0) {
        if (r != run) {
          if (n) atomicAdd(area + run, n);
          run = r;
          n = 0;
        }
        ++n;
      }
    }
    if (AREA) {  // one addition per root and warp
      const unsigned peers = __match_any_sync(0xffffffffu, run);
      const int total = __reduce_add_sync(peers, n);
      if (run >= 0 && lane == __ffs(peers) - 1) atomicAdd(area + run, total);
    }
  }
  if (fail) atomicOr(flags + FLAG_TIMEOUT, 1);
}

// partial sums: [0] bubbles, [1] gas cells, [2] sum of equivalent diameters;
// histogram counts are integers, accumulated exactly with atomics
constexpr int kMaxBins = 64;
constexpr int kStatVals = 4;  // and [3] the mass (the tiles' partial sums)

__global__ void __launch_bounds__(kThreads) kd_stats(int nx, int ny, int ntx, int ntiles,
                                                     const uint8_t* __restrict__ tile_gas,
                                                     const int32_t* __restrict__ L, const int32_t* __restrict__ area,
                                                     const double* __restrict__ tile_mass, int nbins, double ldmin,
                                                     double ldspan, double* partials, int* hist) {
  double v[kStatVals] = {0.0, 0.0, 0.0, 0.0};
  const int lane = threadIdx.x & 31;
  int gas = 0;
  for (int t = blockIdx.x * kTileWarps + (threadIdx.x >> 5); t < ntiles; t += gridDim.x * kTileWarps) {
    if (!tile_gas[t]) continue;
    const int x = (t % ntx) * kTX + lane, y0 = (t / ntx) * kTY;
    for (int j = 0; j < kTY; ++j) {
      const int y = y0 + j;
      if (x >= nx || y >= ny) break;
      const int c = y * nx + x, l = L[c];
      if (l < 0) continue;
      ++gas;
      if (l == c) {
        const double d = 2.0 * sqrt((double)area[c] / M_PI);
        v[0] += 1.0;
        v[2] += d;
        if (nbins > 0) {
          int b = (int)floor((log(d) - ldmin) / ldspan * nbins);
          b = b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
          atomicAdd(hist + b, 1);
        }
      }
    }
  }
  v[1] = (double)gas;
  for (int t = blockIdx.x * kThreads + threadIdx.x; t < ntiles; t += gridDim.x * kThreads) v[3] += tile_mass[t];
  block_reduce_store<kStatVals>(v, partials);
}

// Roots with their areas appended to list (warp-aggregated slots).
__global__ void __launch_bounds__(32 * kTileWarps) kd_list(int nx, int ny, int ntx, int ntiles,
                                                           const uint8_t* __restrict__ tile_gas,
                                                           const int32_t* __restrict__ L,
                                                           const int32_t* __restrict__ area, int32_t* __restrict__ list,
                                                           int* count) {
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x * kTileWarps + (threadIdx.x >> 5); t < ntiles; t += gridDim.x * kTileWarps) {
    if (!tile_gas[t]) continue;
    const int x = (t % ntx) * kTX + lane, y0 = (t / ntx) * kTY;
    for (int j = 0; j < kTY; ++j) {
      const int y = y0 + j, c = y * nx + x;
      const bool root = x < nx && y < ny && L[c] == c;
      const unsigned b = __ballot_sync(0xffffffffu, root);
      if (!b) continue;
      int base = 0;
      if (lane == __ffs(b) - 1) base = atomicAdd(count, __popc(b));
      base = __shfl_sync(0xffffffffu, base, __ffs(b) - 1);
      if (root) {
        const int k = base + __popc(b & ((1u << lane) - 1u));
        list[2 * k] = c;
        list[2 * k + 1] = area[c];
      }
    }
  }
}

inline dim3 row_grid(int nx, int ny, int planes) {
  const int gy = (ny + kRows - 1) / kRows;
  return dim3((nx + kThreads - 1) / kThreads, gy < 65535 ? gy : 65535, planes);
}

inline int tile_grid(int ntiles) {
  const int n = (ntiles + kTileWarps - 1) / kTileWarps, cap = device_sm_count() * 8;
  return n < cap ? n : cap;
}

inline bool base16(const void* a) { return (reinterpret_cast<uintptr_t>(a) & 15u) == 0; }

}  // namespace

#define LBM_BY_STORAGE(storage, CALL)              \
  switch (storage) {                               \
    case LBM_F32: CALL(LBM_F32); break;            \
    case LBM_F16_DEV: CALL(LBM_F16_DEV); break;    \
    case LBM_BF16_DEV: CALL(LBM_BF16_DEV); break;  \
    default: return cudaErrorInvalidValue;         \
  }

int mass_partials_needed() { return kRedBlocks * kStatVals; }

cudaError_t launch_density(const FieldParams& fp, float* rho, cudaStream_t s) {
#define CALL(S) k_density<S><<<row_grid(fp.nx, fp.ny, 1), kThreads, 0, s>>>(fp, rho)
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_pops_out(const FieldParams& fp, int plane0, int planes, float* out, cudaStream_t s) {
  const bool vec = fp.nx % 4 == 0 && base16(out) && fp.N % 4 == 0;
  const int rows = fp.storage == LBM_F32 ? pop_rows<LBM_F32>() : pop_rows<LBM_F16_DEV>();
  dim3 grid = row_grid((fp.nx + 3) / 4, fp.ny, planes);
  grid.y = std::min((fp.ny + rows - 1) / rows, 65535);
#define CALL(S) k_pops_out<S><<<grid, kThreads, 0, s>>>(fp, plane0, vec, out)
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  return cudaGetLastError();
}

cudaError_t launch_mask_out(const FieldParams& fp, const uint8_t* mask, uint8_t* out, cudaStream_t s) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(out);
  const int vec = fp.nx % 16 == 0 && a % 16 == 0 ? 16 : (fp.nx % 4 == 0 && a % 4 == 0 ? 4 : 1);
  const dim3 grid((fp.nx + 16 * kThreads - 1) / (16 * kThreads), fp.ny < 65535 ? fp.ny : 65535);
  k_mask_out<<<grid, kThreads, 0, s>>>(mask, fp.mpitch, fp.nx, fp.ny, vec, out);
  return cudaGetLastError();
}

cudaError_t launch_fields(const FieldParams& fp, const uint8_t* mask, const FieldOuts& out, cudaStream_t s) {
  const unsigned tiles = (unsigned)((fp.nx + kFX - 1) / kFX) * (unsigned)((fp.ny + kFY - 1) / kFY);
  if (out.ux || out.uy) {
#define CALL(S) k_fields<S, true><<<tiles, kThreads, 0, s>>>(fp, mask, out)
    LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  } else {
#define CALL(S) k_fields<S, false><<<tiles, kThreads, 0, s>>>(fp, mask, out)
    LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  }
  return cudaGetLastError();
}

cudaError_t launch_mass(const FieldParams& fp, double* partials, int nparts, double* out_dev, cudaStream_t s) {
  if (nparts < kRedBlocks) return cudaErrorInvalidValue;
#define CALL(S) k_mass_partial<S><<<kRedBlocks, kThreads, 0, s>>>(fp, partials)
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  k_sum_partials<1><<<1, kThreads, 0, s>>>(partials, kRedBlocks, out_dev);
  return cudaGetLastError();
}

size_t diag_scratch_bytes(int nx, int ny) {
  const size_t nt = (size_t)relabel_tile_count(nx, ny);
  return nt * sizeof(double) + nt;
}

// Tile sums first (8-byte aligned scratch), then the flags.
static uint8_t* diag_flags(void* scratch, int nt) { return static_cast<uint8_t*>(scratch) + (size_t)nt * sizeof(double); }

template <bool AREA, bool MASS>
static cudaError_t labels_pass(const FieldParams& fp, float threshold, int32_t* label, int32_t* area, void* scratch,
                               int* flags, cudaStream_t s) {
  const int nt = relabel_tile_count(fp.nx, fp.ny), ntx = (fp.nx + kTX - 1) / kTX;
  uint8_t* tg = diag_flags(scratch, nt);
  double* tm = static_cast<double*>(scratch);
#define CALL(S) \
  kd_label<S, AREA, MASS><<<nt, dim3(kTX / 4, kTY), 0, s>>>(fp, threshold, fp.nx % 4 == 0 && base16(label), label, area, tg, tm, flags)
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  kd_union<<<tile_grid(nt), 32 * kTileWarps, 0, s>>>(fp.nx, fp.ny, ntx, nt, tg, label, flags);
  kd_flatten<AREA><<<tile_grid(nt), 32 * kTileWarps, 0, s>>>(fp.nx, fp.ny, ntx, nt, tg, label, area, flags);
  return cudaGetLastError();
}

cudaError_t launch_diag_labels(const FieldParams& fp, float threshold, int32_t* label, void* scratch, int* flags,
                               cudaStream_t s) {
  return labels_pass<false, false>(fp, threshold, label, nullptr, scratch, flags, s);
}

cudaError_t launch_diag_stats(const FieldParams& fp, float threshold, int32_t* label, int32_t* area, void* scratch,
                              int* flags, double* partials, int nparts, double* out_dev, int* hist, int nbins,
                              double dmin, double dmax, cudaStream_t s) {
  if (nparts < kRedBlocks * kStatVals || nbins > kMaxBins) return cudaErrorInvalidValue;
  const int nt = relabel_tile_count(fp.nx, fp.ny), ntx = (fp.nx + kTX - 1) / kTX;
  cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(int) * kMaxBins, s);
  if (e != cudaSuccess) return e;
  if ((e = labels_pass<true, true>(fp, threshold, label, area, scratch, flags, s)) != cudaSuccess) return e;
  const double ldmin = log(dmin > 0 ? dmin : 1.0);
  const double ldspan = log(dmax > dmin && dmin > 0 ? dmax : 2.0 * (dmin > 0 ? dmin : 1.0)) - ldmin;
  kd_stats<<<kRedBlocks, kThreads, 0, s>>>(fp.nx, fp.ny, ntx, nt, diag_flags(scratch, nt), label, area,
                                           static_cast<const double*>(scratch), nbins, ldmin, ldspan, partials, hist);
  k_sum_partials<kStatVals><<<1, kThreads, 0, s>>>(partials, kRedBlocks, out_dev);
  return cudaGetLastError();
}

cudaError_t launch_diag_areas(const FieldParams& fp, float threshold, int32_t* label, int32_t* area, int32_t* list,
                              int* count, void* scratch, int* flags, cudaStream_t s) {
  const int nt = relabel_tile_count(fp.nx, fp.ny), ntx = (fp.nx + kTX - 1) / kTX;
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  if ((e = labels_pass<true, false>(fp, threshold, label, area, scratch, flags, s)) != cudaSuccess) return e;
  kd_list<<<tile_grid(nt), 32 * kTileWarps, 0, s>>>(fp.nx, fp.ny, ntx, nt, diag_flags(scratch, nt), label, area, list,
                                                    count);
  return cudaGetLastError();
}

}  // namespace lbm
