// Many steps of a small box in one launch: k_steps_resident.
//
// A launch per step costs a small box 2.7 us whatever its size (launch, load
// latency, drain), with most of the GPU idle. Here one thread-block cluster
// keeps the box in its CTAs' shared memory for all steps between two events
// of the host loop (a relabel, the end of the call): each CTA holds a strip of
// rows with one halo row above and below, and hands its outermost rows' psi
// and outgoing populations to its neighbours through distributed shared
// memory. Two cluster barriers per step replace the launch: one after psi
// (which also says that every pull has been read), one after the new
// populations.
//
// A thread owns pairs of cells (x, x + nx/2) of a row for the packed
// arithmetic, so that a warp's shared-memory accesses are consecutive words.
// Same per-cell arithmetic as every step kernel: bitwise the same
// populations. 128^2 FP32: 2.7 us per step with a launch each, 1.45
// here (64^2 0.93): two barriers, and the latency of a psi and a population
// read between them.
#include "cellmath.cuh"
#include "launch.cuh"

namespace lbm {
namespace {

constexpr int kResThreads = 512, kResCtas = 16;
constexpr size_t kResSmem = 227 * 1024;

struct Resident {
  const void* src;  // column 0
  void* dst;
  const uint8_t* mask;  // nullptr: plain Shan-Chen
  int* flags;
  int nx, ny, pitch, mpitch;
  long long plane;
  int rows;   // per CTA (the last ones may hold fewer, or none)
  int steps;  // >= 1
  StepParams s;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t smem_address(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// *p of CTA `cta` of the cluster
__device__ __forceinline__ void put_remote(const float* p, int cta, float v) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_address(p)), "r"(cta));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

template <int S>
__device__ __forceinline__ float stored(float v) {  // the value the next step reads back
  const typename Store<S>::T w = Store<S>::enc(v);
  return Store<S>::raw_smem(&w, 0);
}

// PAIRS: pairs of cells per thread at most.
template <int S, bool MASKED, bool TAU_ONE, int PAIRS>
__global__ void __launch_bounds__(kResThreads, 1) k_steps_resident(const Resident b) {
  using T = typename Store<S>::T;
  extern __shared__ float smem[];
  grid_begin();
  const int nx = b.nx, ny = b.ny, h = b.rows, half = (nx + 1) / 2;
  const int cta = blockIdx.x, live = (ny + h - 1) / h;  // CTAs holding rows
  const int y0 = cta * h, hc = max(0, min(h, ny - y0));
  const int up = cta == 0 ? live - 1 : cta - 1, down = cta + 1 == live ? 0 : cta + 1;
  const int last_up = min(h, ny - up * h);  // rows of the CTA above
  const int ps = (h + 2) * nx;              // one plane: halo row, rows, halo row
  float* const F = smem;
  float* const psi = smem + Q * ps;
  if (hc > 0) {
    for (int k = threadIdx.x; k < (hc + 2) * nx; k += kResThreads) {
      const int r = k / nx, x = k - r * nx;
      int y = y0 + r - 1;
      y = y < 0 ? ny - 1 : (y >= ny ? 0 : y);
      const T* row = static_cast<const T*>(b.src) + (size_t)y * b.pitch;
      float v[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) v[i] = Store<S>::raw(row + (size_t)i * b.plane, x);
#pragma unroll
      for (int i = 0; i < Q; ++i) F[i * ps + k] = v[i];
    }
  }
  // this thread's pairs: offset of the row in a plane, columns and their neighbours
  int at[PAIRS], xa[PAIRS], xb[PAIRS];
  unsigned mask[PAIRS];
#pragma unroll
  for (int k = 0; k < PAIRS; ++k) {
    const int p = threadIdx.x + k * kResThreads, r = p / half;
    at[k] = r < hc ? (r + 1) * nx : 0;  // 0: no pair
    xa[k] = p - r * half;
    xb[k] = xa[k] + half < nx ? xa[k] + half : xa[k];  // an odd width's middle column: twice the same cell
    mask[k] = 0;
    if (MASKED && at[k]) {
      const uint8_t* m = b.mask + (size_t)(y0 + r) * b.mpitch;
      mask[k] = (unsigned)__ldcg(m + xa[k]) | (unsigned)__ldcg(m + xb[k]) << 8;
    }
  }
  uint32_t worst = 0;
  cluster_arrive();  // every CTA of the cluster runs; own rows are loaded
  cluster_wait();
  for (int s = 0; s < b.steps; ++s) {
    const bool last = s + 1 == b.steps;
    float2 rho[PAIRS], jx[PAIRS], jy[PAIRS], own[PAIRS], g[PAIRS][TAU_ONE ? 1 : Q];
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
      if (!at[k]) continue;
      const int a = xa[k], c = xb[k];
      const int am = a == 0 ? nx - 1 : a - 1, ap = a + 1 == nx ? 0 : a + 1, cm = c == 0 ? nx - 1 : c - 1,
                cp = c + 1 == nx ? 0 : c + 1;
      float2 f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const float* row = F + i * ps + at[k] - cy(i) * nx;
        f[i] = make_float2(row[cx(i) > 0 ? am : (cx(i) < 0 ? ap : a)], row[cx(i) > 0 ? cm : (cx(i) < 0 ? cp : c)]);
      }
      if (MASKED && s > 0 && mask[k]) {
        // what would have come across a blocked edge is the cell's own
        // outgoing population (the launch's first step reads slots that the
        // host loop has bounced back already)
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          const float* row = F + i * ps + at[k];
          if ((mask[k] >> (i - 1)) & 1u) f[opp(i)].x = row[a];
          if ((mask[k] >> (i + 7)) & 1u) f[opp(i)].y = row[c];
        }
      }
      moments9(f, rho[k], jx[k], jy[k]);
      own[k] = psi_of(full_rho<S != LBM_F32>(rho[k], b.s), b.s);
      if (!TAU_ONE) {
#pragma unroll
        for (int i = 0; i < Q; ++i) g[k][TAU_ONE ? 0 : i] = f[i];
      }
      psi[at[k] + a] = own[k].x;
      psi[at[k] + c] = own[k].y;
      if (at[k] == nx) {
        put_remote(psi + (last_up + 1) * nx + a, up, own[k].x);
        put_remote(psi + (last_up + 1) * nx + c, up, own[k].y);
      }
      if (at[k] == hc * nx) {
        put_remote(psi + a, down, own[k].x);
        put_remote(psi + c, down, own[k].y);
      }
    }
    cluster_arrive();
    cluster_wait();
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
      if (!at[k]) continue;
      const int a = xa[k], c = xb[k];
      const int am = a == 0 ? nx - 1 : a - 1, ap = a + 1 == nx ? 0 : a + 1, cm = c == 0 ? nx - 1 : c - 1,
                cp = c + 1 == nx ? 0 : c + 1;
      float2 n[Q], Fx, Fy, f[Q];
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const float* row = psi + at[k] + cy(i) * nx;
        n[i] = make_float2(row[cx(i) > 0 ? ap : (cx(i) < 0 ? am : a)], row[cx(i) > 0 ? cp : (cx(i) < 0 ? cm : c)]);
      }
      if (MASKED && mask[k]) {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          if ((mask[k] >> (i - 1)) & 1u) n[i].x = own[k].x;
          if ((mask[k] >> (i + 7)) & 1u) n[i].y = own[k].y;
        }
      }
      force_of(n, own[k], b.s.G, Fx, Fy);
      if (!TAU_ONE) {
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = g[k][TAU_ONE ? 0 : i];
      }
      collide<TAU_ONE, S != LBM_F32>(f, rho[k], jx[k], jy[k], Fx, Fy, b.s, worst);
      if (last) {
        const int y = y0 + at[k] / nx - 1;
        T* row = static_cast<T*>(b.dst) + (size_t)y * b.pitch;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          put_cell(row + (size_t)i * b.plane, a, nx, Store<S>::enc(f[i].x));
          put_cell(row + (size_t)i * b.plane, c, nx, Store<S>::enc(f[i].y));
        }
        continue;
      }
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        float* row = F + i * ps;
        const float2 v = make_float2(stored<S>(f[i].x), stored<S>(f[i].y));
        row[at[k] + a] = v.x;
        row[at[k] + c] = v.y;
        if (cy(i) < 0 && at[k] == nx) {  // leaves upwards: the halo row below the last row there
          put_remote(row + (last_up + 1) * nx + a, up, v.x);
          put_remote(row + (last_up + 1) * nx + c, up, v.y);
        }
        if (cy(i) > 0 && at[k] == hc * nx) {
          put_remote(row + a, down, v.x);
          put_remote(row + c, down, v.y);
        }
      }
    }
    if (!last) {
      cluster_arrive();
      cluster_wait();
    }
  }
  report_faults(worst, b.flags);
}

int rows_of(int ny) { return (ny + kResCtas - 1) / kResCtas; }
size_t smem_of(int nx, int ny) { return (size_t)(Q + 1) * (rows_of(ny) + 2) * nx * sizeof(float); }
int pairs_of(int nx, int ny) { return (rows_of(ny) * ((nx + 1) / 2) + kResThreads - 1) / kResThreads; }

template <int S, bool MASKED, bool TAU_ONE, int PAIRS>
cudaError_t launch_pairs(const Resident& b, cudaStream_t s) {
  return launch_cluster(k_steps_resident<S, MASKED, TAU_ONE, PAIRS>, kResCtas, dim3(kResCtas), dim3(kResThreads),
                        smem_of(b.nx, b.ny), s, b);
}

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_tau(const Resident& b, cudaStream_t s) {
  switch (pairs_of(b.nx, b.ny)) {
    case 1: return launch_pairs<S, MASKED, TAU_ONE, 1>(b, s);
    case 2: return launch_pairs<S, MASKED, TAU_ONE, 2>(b, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int S>
cudaError_t launch_s(const Resident& b, cudaStream_t s) {
  const bool one = b.s.tau == 1.0f;
  if (b.mask) return one ? launch_tau<S, true, true>(b, s) : launch_tau<S, true, false>(b, s);
  return one ? launch_tau<S, false, true>(b, s) : launch_tau<S, false, false>(b, s);
}

}  // namespace

// Whether `steps` steps of the box go in one launch: up to two pairs per thread
// (32768 cells; beyond, a CTA's share of a step takes as long as a launch over
// the whole GPU), and enough steps to pay for loading and storing the box (3 us
// for one pair, 9 for two). Microseconds per step with a launch each and here:
// 128^2 FP32 (one pair) in calls of 4 steps 3.2 and 2.2, of 100 2.7 and 1.45;
// 256 x 128 (two) in calls of 5 steps 2.9 and 3.1, of 10 2.8 and 2.7, of 100 2.8
// and 2.3; 1024 x 32, the longest halos, of 10 2.8 and 3.0, of 100 2.8 and 2.5.
bool steps_resident(const StepParams& p, long long steps) {
  if (p.force_generic != 0 || pairs_of(p.nx, p.ny) > 2 || smem_of(p.nx, p.ny) > kResSmem) return false;
  if (steps < (pairs_of(p.nx, p.ny) == 1 ? 4 : 16)) return false;
  return cluster_fits(k_steps_resident<LBM_F32, true, false, 2>, kResCtas, kResThreads, kResSmem);
}

cudaError_t launch_resident(int storage, const StepParams& p, int steps, cudaStream_t s) {
  Resident b{};
  b.src = p.src;
  b.dst = p.dst;
  b.mask = p.mask;
  b.flags = p.flags;
  b.nx = p.nx;
  b.ny = p.ny;
  b.pitch = p.pitch;
  b.mpitch = p.mpitch;
  b.plane = p.plane;
  b.rows = rows_of(p.ny);
  b.steps = steps;
  b.s = p;
  switch (storage) {
    case LBM_F32: return launch_s<LBM_F32>(b, s);
    case LBM_F16_DEV: return launch_s<LBM_F16_DEV>(b, s);
    case LBM_BF16_DEV: return launch_s<LBM_BF16_DEV>(b, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbm
