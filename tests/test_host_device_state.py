"""What the step launchers keep about a device is kept per device: on every
device a staged kernel is allowed its shared memory there before it is
launched, and its grid follows that device's occupancy and SM count, also when
threads step boxes of several devices for the first time together. The
library's launchers run against a stand-in for the CUDA runtime that records
the calls (two devices of 152 and 132 SMs); no GPU is needed."""
import os
import subprocess

import pytest

from paper_1708_01613_gb300 import build as B

RUNTIME = r"""
#include <cuda_runtime_api.h>
#include <cstdio>
#include <map>
#include <mutex>
#include <set>
#include <utility>

thread_local int device = 0;
static std::mutex lock;
static std::map<std::pair<int, const void*>, int> allowed;  // dynamic shared memory by device and kernel
static std::map<int, std::set<unsigned>> grids;             // grid sizes by device
static int launches = 0, refused = 0;
static const int sms[2] = {152, 132}, ctas[2] = {3, 2};

extern "C" {
cudaError_t cudaGetDevice(int* d) { return *d = device, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { return *v = sms[d], cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> g(lock);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) allowed[{device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = ctas[device], cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  std::lock_guard<std::mutex> g(lock);
  ++launches;
  const auto it = allowed.find({device, f});
  if (c->dynamicSmemBytes > 48 * 1024 && (it == allowed.end() || it->second < (int)c->dynamicSmemBytes)) ++refused;
  grids[device].insert(c->gridDim.x);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { return *k = (cudaKernel_t)f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
}

void report() {
  for (int d = 0; d < 2; ++d)  // full grids of the persistent kernels
    printf("device %d own %d other %d\n", d, (int)grids[d].count(sms[d] * ctas[d]),
           (int)grids[d].count(sms[1 - d] * ctas[1 - d]));
  printf("launches %d refused %d\n", launches, refused);
}
"""

PROGRAM = r"""
#include <thread>
#include <vector>
#include "lbm_internal.cuh"

extern thread_local int device;
void report();

// every staged launcher once on the current device
static void step_all() {
  using namespace lbm;
  static uint8_t mask;
  for (int storage : {LBM_F32, LBM_F16_DEV, LBM_BF16_DEV})
    for (float tau : {1.0f, 0.8f})
      for (int masked : {0, 1}) {
        StepParams p{};
        p.nx = p.ny = 8192;
        p.tau = tau;
        p.mask = masked ? &mask : nullptr;
        for (int variant : {2, 3, 4}) {
          p.force_generic = variant;
          launch_step(storage, p, 0);
        }
        launch_step_batch(storage, masked, tau == 1.0f, nullptr, nullptr, 1 << 20, nullptr, 0, 0);
        if (storage == LBM_F32) {
          Step2Params q{};
          q.nx = q.ny = 8192;
          q.tau_m = q.tau_g = tau;
          q.mask = p.mask;
          launch_step2(q, 0);
        }
      }
}

int main() {
  std::vector<std::thread> t;
  for (int k = 0; k < 8; ++k)
    t.emplace_back([k] {
      device = k & 1;
      step_all();
    });
  for (auto& x : t) x.join();
  report();
  return 0;
}
"""


def test_launch_state_is_kept_per_device(tmp_path):
    if not os.path.exists(B.nvcc()):
        pytest.skip("nvcc not available")
    B.build()
    names = ["step", "step2", "tile"]
    objs = [os.path.join(B.BUILD, n + ".o") for n in names]
    newest = max(os.path.getmtime(p) for p in B._deps())
    for n, o in zip(names, objs):
        if not os.path.exists(o) or os.path.getmtime(o) < newest:
            os.makedirs(B.BUILD, exist_ok=True)
            B._compile(os.path.join(B.CSRC, n + ".cu"), [])
    src, rt, exe = tmp_path / "launch.cu", tmp_path / "runtime.cpp", tmp_path / "launch"
    src.write_text(PROGRAM)
    rt.write_text(RUNTIME)
    r = subprocess.run([B.nvcc(), "-std=c++17", "-O1", "-I", B.INCLUDE, "-I", B.CSRC, str(src), str(rt), *objs,
                        "-o", str(exe), "-cudart", "none", "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stderr
    lines = out.stdout.splitlines()
    # 12 combinations of three step variants and the batch, 4 two-component ones, on 8 threads
    assert lines == ["device 0 own 1 other 0", "device 1 own 1 other 0", "launches 416 refused 0"], lines
