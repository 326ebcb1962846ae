// Launches with programmatic dependent launch: a kernel of a chain is put on
// the SMs while the one before it finishes, and waits there for it
// (grid_begin) before it touches memory, which hides the 2 - 2.5 us between
// dependent launches. Every kernel launched through launch_chain calls
// grid_begin in every thread before its first access to data that an earlier
// kernel writes, so completion still means that all work before it is done.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>
#include <vector>

namespace lbm {
namespace {

// Waits for the kernels before this one, then lets the next one be placed.
// Data the earlier kernels wrote is read by ordinary or L2 loads only after
// this (not ld.global.nc, which the compiler may move up).
__device__ __forceinline__ void grid_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_chain(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &attr;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}

// The same as one cluster of `size` CTAs (more than 8: not portable, so ask
// cluster_fits first).
template <typename... P, typename... A>
inline cudaError_t launch_cluster(void (*kern)(P...), int size, dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && smem > 48 * 1024)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = attr;
  c.numAttrs = 2;
  return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}

// A kernel's permission for more than 48 KB of dynamic shared memory and its
// occupancy belong to a device, so a launcher keeps them per device. Threads
// that ask for the first time together both ask, and store the same number.
class PerDevice {
 public:
  // *out = what ask(out) found (> 0) on the current device
  template <typename F>
  cudaError_t get(F ask, int* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool kept = dev >= 0 && dev < kDevices;
    if (kept && (*out = found_[dev].load(std::memory_order_acquire)) > 0) return cudaSuccess;
    e = ask(out);
    if (e == cudaSuccess && kept) found_[dev].store(*out, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> found_[kDevices] = {};
};

// CTAs of a kernel that one SM of the current device holds, after allowing the
// kernel its dynamic shared memory there.
template <typename... P>
inline cudaError_t ctas_per_sm(void (*kern)(P...), int threads, size_t smem, int* out) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kern, threads, smem);
  if (e == cudaSuccess && *out < 1) *out = 1;
  return e;
}

// Whether the current device holds such a cluster (asked once per device and kernel).
template <typename... P>
inline bool cluster_fits(void (*kern)(P...), int size, int threads, size_t smem) {
  struct Seen {
    void (*kern)(P...);
    int dev;
    bool fits;
  };
  static std::mutex lock;
  static std::vector<Seen> seen;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> g(lock);
  for (const Seen& v : seen)
    if (v.kern == kern && v.dev == dev) return v.fits;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess && smem > 48 * 1024)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = size;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(size);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.attrs = &attr;
  c.numAttrs = 1;
  int n = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, kern, &c);
  if (e != cudaSuccess) cudaGetLastError();  // not an error of the caller's
  seen.push_back({kern, dev, e == cudaSuccess && n > 0});
  return seen.back().fits;
}

}  // namespace
}  // namespace lbm

#define LBM_TRY(expr)                      \
  do {                                     \
    const cudaError_t try_ = (expr);       \
    if (try_ != cudaSuccess) return try_;  \
  } while (0)
