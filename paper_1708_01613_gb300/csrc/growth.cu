// Nucleation and bubble growth (Sec. 2.1.3; main flowchart boxes "Random
// Nucleation" and "Bubble growth").
//
// Growth: the paper adds the released hydrogen to every gas point as a
// pressure increment, dp/dt = A (dn/dt) / N (Eq. 34). The increment is taken
// on the ideal-gas part of the equation of state (dp = c_s^2 drho), so a
// release is a density source split equally over the N gas points of the
// latest census and added at rest to their post-collision populations:
// f_i^out(x) += w_i drho. Buffer convention: the buffer a step writes holds
// f_i^out(x) at x (the next step pulls it from x + e_i).
//
// Nucleation: cells within a nucleus radius become gas at rest, incoming
// f_i(x) = w_i rho_g, i.e. B_i(x - e_i) in the buffer the next step reads.
#include "launch.cuh"
#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int kThreadsG = 256;

struct FieldWref {
  float w[Q];  // w_i rho_ref of 16-bit deviations (0 for FP32)
};

__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

__global__ void k_gas_census(const float* __restrict__ rho, long long N, float th, int32_t* __restrict__ list,
                             int* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  // every lane of a warp runs the same number of iterations (bounds tested inside)
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long c0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); c0 < N; c0 += stride) {
    const long long c = c0 + lane;
    const bool gas = c < N && rho[c] < th;
    const unsigned b = __ballot_sync(0xffffffffu, gas);
    if (!b) continue;
    int base = 0;
    if (lane == 0) base = atomicAdd(count, __popc(b));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (gas) list[base + __popc(b & ((1u << lane) - 1u))] = (int32_t)c;
  }
}

// The release is worked out in FP64 by nine lanes of each CTA that has cells
// (FP64 runs at 1/64 of the FP32 rate: 1024^2 with 3 % gas takes 3.1 us, with
// the release worked out by every thread 11.5), while the cells' nine loads, all
// issued before the first store, are on their way. Six CTAs per SM (five fit at
// its 48 registers; capped to 40, with a spill, it is slower at every size):
// 8192^2 with 1.8 % gas 39 us, 4096^2 9.3; two CTAs per SM 71 and 20.
template <int S>
__global__ void __launch_bounds__(kThreadsG) k_growth(typename Store<S>::T* pops, const int32_t* list, const int* count,
                                                      int nx, int pitch, long long plane, double rate, double budget,
                                                      double* released, int parity) {
  __shared__ float add[Q];
  __shared__ int some;
  grid_begin();
  const int n = *count;
  StridedIndex k{(int)(blockIdx.x * blockDim.x + threadIdx.x), (int)(gridDim.x * blockDim.x), n};
  if (blockIdx.x != 0 && (int)(blockIdx.x * blockDim.x) >= n) return;
  float f[Q];
  typename Store<S>::T* cell = pops;  // row of the cell, and its column
  int x = 0;
  auto fetch = [&]() {
    const int c = list[k.at], y = c / nx;
    x = c - y * nx;
    cell = pops + (size_t)y * pitch;
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = Store<S>::raw(cell + (size_t)i * plane, x);
  };
  if (k.in()) fetch();
  if (threadIdx.x < Q) {
    const double before = released[parity];
    double release = 0.0;
    if (n > 0) {
      const double left = budget - before;
      release = rate < left ? rate : left;
      if (!(release > 0.0)) release = 0.0;
    }
    if (k.at == 0) released[parity ^ 1] = before + release;
    if (threadIdx.x == 0) some = release != 0.0;
    if (release != 0.0) add[threadIdx.x] = (float)(wq(threadIdx.x) * (release / (double)n));
  }
  __syncthreads();
  if (!some) return;
  while (k.in()) {
#pragma unroll
    for (int i = 0; i < Q; ++i) put_cell(cell + (size_t)i * plane, x, nx, Store<S>::enc(__fadd_rn(f[i], add[i])));
    k.next();
    if (k.in()) fetch();
  }
}

// Inside test of one cell against the nuclei, in FP64 without contraction
// (the same decision as the oracle's plain expression).
__device__ __forceinline__ bool in_nucleus(const lbm_bubble* __restrict__ nu, int n, int x, int y, int nx,
                                           int ny) {
  for (int k = 0; k < n; ++k) {
    double dx = fabs((double)x - nu[k].cx), dy = fabs((double)y - nu[k].cy);
    dx = fmin(dx, __dsub_rn((double)nx, dx));
    dy = fmin(dy, __dsub_rn((double)ny, dy));
    if (__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)) <= __dmul_rn(nu[k].r, nu[k].r)) return true;
  }
  return false;
}

template <int S>
__global__ void k_nucleate(typename Store<S>::T* __restrict__ pops, const lbm_bubble* __restrict__ nu, int n,
                           double rho_g, int nx, int ny, int pitch, long long plane, FieldWref wr) {
  const long long N = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
       c += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(c % nx), y = (int)(c / nx);
    if (!in_nucleus(nu, n, x, y, nx, ny)) continue;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      // incoming f_i(x) lives at B_i(x - e_i)
      const int xs = wrap1(x - cx(i), nx);
      typename Store<S>::T* row = pops + (size_t)i * plane + (size_t)wrap1(y - cy(i), ny) * pitch;
      put_cell(row, xs, nx, Store<S>::of((float)(wq(i) * rho_g), wr.w[i]));
    }
  }
}

unsigned grid_for(long long n) {
  long long b = (n + kThreadsG - 1) / kThreadsG;
  if (b > device_sm_count() * 8LL) b = device_sm_count() * 8LL;
  return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t launch_gas_census(const float* rho, long long N, float threshold, int32_t* list, int* count,
                              cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  k_gas_census<<<grid_for(N), kThreadsG, 0, s>>>(rho, N, threshold, list, count);
  return cudaGetLastError();
}

#define LBM_BY_STORAGE(storage, CALL)                    \
  switch (storage) {                                     \
    case LBM_F32: CALL(LBM_F32, float); break;           \
    case LBM_F16_DEV: CALL(LBM_F16_DEV, __half); break;  \
    case LBM_BF16_DEV: CALL(LBM_BF16_DEV, __nv_bfloat16); break; \
    default: return cudaErrorInvalidValue;               \
  }

cudaError_t launch_growth(const FieldParams& fp, void* pops, const int32_t* list, const int* count, double rate,
                          double budget, double* released, int parity, cudaStream_t s) {
  const unsigned g = (unsigned)device_sm_count() * 6;
#define CALL(S, T)                                                                                                   \
  LBM_TRY(launch_chain(k_growth<S>, dim3(g), dim3(kThreadsG), 0, s, static_cast<T*>(pops), list, count, fp.nx, fp.pitch, \
                       fp.plane, rate, budget, released, parity))
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  return cudaSuccess;
}

cudaError_t launch_nucleate(const FieldParams& fp, void* pops, const lbm_bubble* nuclei, int n, double rho_g,
                            cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  FieldWref wr;
  for (int i = 0; i < Q; ++i) wr.w[i] = fp.wref[i];
  const unsigned g = grid_for(fp.N);
#define CALL(S, T)                                                                                              \
  k_nucleate<S><<<g, kThreadsG, 0, s>>>(static_cast<T*>(pops), nuclei, n, rho_g, fp.nx, fp.ny, fp.pitch, fp.plane, \
                                        wr)
  LBM_BY_STORAGE(fp.storage, CALL)
#undef CALL
  return cudaGetLastError();
}

}  // namespace lbm
