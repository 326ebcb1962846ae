// Pulled populations of four cells (x .. x + 3, x a multiple of 4) of row y
// per thread, shared by the relabel's density phase and the diagnostics:
// f_i(x) = B_i(x - e_i). A plane arrives in one vector load (16 bytes FP32, 8
// bytes 16-bit), a plane the pull shifts by one column adds the value (or
// 4-byte word) beside it; the ghost columns stand in for the periodic wrap.
#pragma once
#include "lbm_internal.cuh"

namespace lbm {
namespace {

template <int S>
__device__ __forceinline__ float dec16(unsigned short v) {
  if constexpr (S == LBM_F16_DEV) return __half2float(__ushort_as_half(v));
  else return __bfloat162float(__ushort_as_bfloat16(v));
}

template <int S>
__device__ __forceinline__ float2 dec16x2(uint32_t bits) {
  return make_float2(dec16<S>((unsigned short)(bits & 0xffffu)), dec16<S>((unsigned short)(bits >> 16)));
}

__device__ __forceinline__ int pull_wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Cells (x, x + 1) in fa and (x + 2, x + 3) in fb; 0 <= x < nx, 0 <= y < ny.
// Cells beyond the box's last column take whatever lies there.
template <int S>
__device__ __forceinline__ void pull4(const typename Store<S>::T* __restrict__ pops, long long plane, int pitch,
                                      const float (&wref)[Q], int ny, int x, int y, float2 (&fa)[Q], float2 (&fb)[Q]) {
  const size_t r0 = (size_t)y * pitch + x;
  const size_t rm = (size_t)(y == 0 ? ny - 1 : y - 1) * pitch + x, rp = (size_t)(y == ny - 1 ? 0 : y + 1) * pitch + x;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const size_t at = (size_t)i * plane + (cy(i) > 0 ? rm : (cy(i) < 0 ? rp : r0));
    if constexpr (S == LBM_F32) {
      const float* q = pops + at;
      const float4 w = __ldcg(reinterpret_cast<const float4*>(q));  // columns x .. x + 3
      if (cx(i) > 0) {  // columns x - 1 .. x + 2
        fa[i] = make_float2(__ldcg(q - 1), w.x);
        fb[i] = make_float2(w.y, w.z);
      } else if (cx(i) < 0) {  // columns x + 1 .. x + 4
        fa[i] = make_float2(w.y, w.z);
        fb[i] = make_float2(w.w, __ldcg(q + 4));
      } else {
        fa[i] = make_float2(w.x, w.y);
        fb[i] = make_float2(w.z, w.w);
      }
    } else {
      const unsigned short* q = reinterpret_cast<const unsigned short*>(pops) + at;
      const uint2 w = __ldcg(reinterpret_cast<const uint2*>(q));  // columns x .. x + 3
      uint32_t lo = w.x, hi = w.y;
      if (cx(i) > 0) {  // columns x - 1 .. x + 2
        const uint32_t wm = __ldcg(reinterpret_cast<const uint32_t*>(q - 2));
        lo = __byte_perm(wm, w.x, 0x5432);
        hi = __byte_perm(w.x, w.y, 0x5432);
      } else if (cx(i) < 0) {  // columns x + 1 .. x + 4
        const uint32_t wp = __ldcg(reinterpret_cast<const uint32_t*>(q + 4));
        lo = __byte_perm(w.x, w.y, 0x5432);
        hi = __byte_perm(w.y, wp, 0x5432);
      }
      const float2 wr = make_float2(wref[i], wref[i]);
      fa[i] = __fadd2_rn(wr, dec16x2<S>(lo));
      fb[i] = __fadd2_rn(wr, dec16x2<S>(hi));
    }
  }
}

// Sum of the nine values in the order every density of the library takes
// (the packed adds round per component like the scalar ones).
__device__ __forceinline__ float2 rho_pair(const float2 (&f)[Q]) {
  return __fadd2_rn(__fadd2_rn(__fadd2_rn(__fadd2_rn(f[0], f[1]), __fadd2_rn(f[2], f[3])),
                               __fadd2_rn(__fadd2_rn(f[4], f[5]), __fadd2_rn(f[6], f[7]))),
                    f[8]);
}

}  // namespace
}  // namespace lbm
