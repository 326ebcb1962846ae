// The bounce-back of a blocked edge, shared by the tiled pipeline (relabel.cu)
// and the boxes outside it (barrier.cu).
#pragma once
#include "lbm_internal.cuh"

namespace lbm {
namespace {

// Mask bits of the directions 1, 2, 5, 6: each blocked edge is seen from the
// one end where its direction is among these.
constexpr unsigned kCanonBits = 0x33u;

__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// --- halfway bounce-back across blocked edges (the barrier of Sec. 2.1.5) ---
// The step kernels store every outgoing population in its own slot: slot
// (plane i, x) holds f_i^out(x), which the next step pulls into x + e_i. For
// a blocked edge (x, x + e_i) the wall sends it back instead: f_i^out(x)
// returns to x as population opp(i), which the next step pulls from
// x - e_opp(i) = x + e_i in plane opp(i), and f_opp(i)^out(x + e_i) returns to
// x + e_i as population i, pulled from slot (plane i, x). So after the step
// the two slots of every blocked edge trade their values. The mask is
// symmetric; each edge is handled once, from its end whose direction is
// 1, 2, 5 or 6 (mask bits 0, 1, 4, 5), and every slot belongs to one edge
// only, so no two threads touch the same slot. T is the raw storage word
// (4 or 2 bytes: the values move bit for bit); TWO: a second lattice follows
// the first nine planes.
template <typename T, bool TWO>
__device__ __forceinline__ void bounce_cell(T* __restrict__ pops, size_t plane, int pitch, int x, int y, int nx, int ny,
                                            unsigned m) {
  m &= kCanonBits;
  if (!m) return;
#pragma unroll
  for (int i = 1; i <= 6; ++i) {
    if (i == 3 || i == 4 || !((m >> (i - 1)) & 1u)) continue;
    const int xb = wrap1(x + cx(i), nx);
    T* ra = pops + (size_t)i * plane + (size_t)y * pitch;
    T* rb = pops + (size_t)opp(i) * plane + (size_t)wrap1(y + cy(i), ny) * pitch;
#pragma unroll
    for (int k = 0; k < (TWO ? 2 : 1); ++k, ra += Q * plane, rb += Q * plane) {
      const T va = ra[x], vb = rb[xb];
      put_cell(ra, x, nx, vb);
      put_cell(rb, xb, nx, va);
    }
  }
}

}  // namespace
}  // namespace lbm
