// Launches with programmatic dependent launch: a kernel of a chain is put on
// the SMs while the one before it finishes, and waits there for it
// (grid_begin) before it touches memory, which hides the 2 - 2.5 us between
// dependent launches. Every kernel launched through launch_chain calls
// grid_begin in every thread before its first access to data that an earlier
// kernel writes, so completion still means that all work before it is done.
#pragma once
#include <cuda_runtime.h>

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

}  // namespace
}  // namespace lbm

#define LBM_TRY(expr)                      \
  do {                                     \
    const cudaError_t try_ = (expr);       \
    if (try_ != cudaSuccess) return try_;  \
  } while (0)
