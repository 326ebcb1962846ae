"""The step's reciprocal and exponential against CUDA's own, over every
argument of their range, and a step of a box whose density is subnormal."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_1708_01613_gb300 import Simulation, build as B, make_config

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "cellmath.cuh"
using namespace lbm;

// every positive float with bits in [lo, hi): the scalar and both packed reciprocals
__global__ void k_recip(unsigned lo, unsigned hi, unsigned long long* bad) {
  unsigned long long n = 0;
  for (unsigned long long b = lo + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b < hi;
       b += (unsigned long long)gridDim.x * blockDim.x) {
    const float a = __uint_as_float((unsigned)b), c = __uint_as_float((unsigned)(b ^ 1));  // a neighbour beside it
    const float2 p = VOps<float2>::rcp(make_float2(__fmul_rn(a, kRhoScale), __fmul_rn(c, kRhoScale)));
    n += __float_as_uint(recip(__fmul_rn(a, kRhoScale))) != __float_as_uint(__frcp_rn(a));
    n += __float_as_uint(p.x) != __float_as_uint(__frcp_rn(a));
    n += c > 0.f && __float_as_uint(p.y) != __float_as_uint(__frcp_rn(c));
  }
  if (n) atomicAdd(bad, n);
}

// 1 - e^x for every float x in [-0x1p127, -0]
__global__ void k_exp(unsigned long long* bad) {
  unsigned long long n = 0;
  for (unsigned long long b = 0x80000000ull + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b <= 0xff000000ull;
       b += (unsigned long long)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((unsigned)b);
    const float got = __fsub_rn(1.0f, exp2_approx(__fmul_rn(x, 1.4426950408889634f)));
    n += __float_as_uint(got) != __float_as_uint(__fsub_rn(1.0f, __expf(x)));
  }
  if (n) atomicAdd(bad, n);
}

extern "C" long long mismatches(int what) {
  unsigned long long *d, h = 0;
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
  cudaMemset(d, 0, sizeof(h));
  // 1 .. bits(2^102): from the smallest subnormal
  if (what == 0) k_recip<<<2048, 256>>>(1u, (102u + 127u) << 23, d);
  else k_exp<<<2048, 256>>>(d);
  const cudaError_t e = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? (long long)h : -2;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cellmath")
    src, so = d / "cellmath.cu", d / "libcellmath.so"
    src.write_text(PROGRAM)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", str(src), "-o", str(so)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = C.CDLL(str(so))
    out.mismatches.restype = C.c_longlong
    return out


def test_reciprocal_of_every_density(lib):
    assert lib.mismatches(0) == 0


def test_exponential_of_every_argument(lib):
    assert lib.mismatches(1) == 0


@pytest.mark.parametrize("variant,nx,steps", [(0, 64, 1), (0, 64, 8), (0, 1200, 2), (1, 64, 2), (2, 272, 2), (3, 67, 2), (4, 272, 2)])
@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_subnormal_density_stays(variant, nx, steps, tau):
    rho = 5e-39  # 1 / rho is finite
    sim = Simulation(make_config(nx, 600 if nx == 1200 else 20, tau=tau))
    sim.set_step_variant(variant)
    sim.init_density(np.full((sim.ny, nx), rho))
    sim.step(steps)
    sim.sync()
    w = np.array([4 / 9] + 4 * [1 / 9] + 4 * [1 / 36])[:, None, None]
    f = sim.read("pops")["pops"].astype(np.float64)
    # at rest, every operation of a step exact or within half the spacing 2^-149:
    # ten of them on the way to a population
    assert np.abs(f - w * rho).max() <= steps * 10 * 2.0**-150, np.abs(f - w * rho).max() / 2.0**-150
