// Fused time step of the extended Shan-Chen lattice Boltzmann method
// (arXiv 1708.01613): pull streaming (Sec. 2.1.1, Eq. 19), moments (Eq. 11),
// pseudopotential (Sec. 2.1.2, Eq. 30), masked neighbour-sum force (Eq. 22;
// barrier of Sec. 2.1.5), velocity-shift equilibrium (Eqs. 39-40 with
// Eq. 14) and BGK collision (Eq. 18), in one pass over the populations.
//
// Layout: structure of arrays, padded rows with two ghost columns on either
// side (PopShape), x fastest. The buffer read by a step holds the
// post-collision populations of the previous step at their source cell; the
// step pulls f_i(x) from x - e_i, and writes the ghosts of the outer columns
// it stores, so no kernel here wraps along x.
//
// Every kernel marches a strip of columns down a chunk of rows. For every
// row it pulls the populations of the strip's cells and of one halo column
// on each side, forms rho and psi once per cell, and puts psi into a
// four-row ring in shared memory; one barrier later the ring holds psi for
// rows r-2..r and the force and collision of row r-1 run on the moments kept
// in registers. All per-cell arithmetic lives in the shared device functions
// of cellmath.cuh (one cell or two), so every kernel gives bitwise the same
// populations.
//
//  - k_step_strip: plain global loads, one cell per thread; any box size.
//  - k_step_tma: the nine source rows of every output row (with halo) are
//    copied into a ring of shared-memory stages by cp.async.bulk, issued
//    NSTAGE-1 rows ahead by a ninth warp that also computes the two halo
//    cells, so the eight compute warps are balanced and the bytes in flight
//    do not depend on occupancy.
//  - k_step_tma2: the same staging over 512-column strips with two cells per
//    thread (march2); one static row chunk per CTA.
//  - k_step_dyn: march2 over row chunks that the resident CTAs draw from a
//    device counter (the automatic choice for the boxes that the tile kernel,
//    tile.cu, steps more slowly).
//  - k_step_batch: march2 over work items (box, strip, row chunk) of many
//    boxes in one launch (batch.cu).
//
// A staged window is copied whole: in a ragged last strip, and up to the next
// 16 bytes, it runs past the box's last column, whose neighbours in memory
// (the rest of the row, the next row, after the last row the workspace's next
// slice) are never used.
#include "cellmath.cuh"
#include "launch.cuh"
#include "tma.cuh"

namespace lbm {
namespace {

constexpr int kBX = 256;           // columns per strip (= compute threads)
constexpr int kTmaThreads = kBX + 32;

__device__ __forceinline__ int wrapi(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// Rows r - 1, r, r + 1 of the torus for r in [-1, ny].
struct Rows3 {
  int m, c, p;
  __device__ __forceinline__ Rows3(int r, int ny) {
    c = wrapi(r, ny);
    m = c == 0 ? ny - 1 : c - 1;
    p = c == ny - 1 ? 0 : c + 1;
  }
};

// Force + collision + store of one cell from the psi ring.
template <int S, bool MASKED, bool TAU_ONE>
__device__ __forceinline__ void finish_cell(float f[Q], float rho, float jx, float jy, unsigned m,
                                            const float (*ring)[kBX + 2], int sm, int s0, int sp, int jc,
                                            const StepParams& p, typename Store<S>::T* __restrict__ row, int x,
                                            uint32_t& worst) {
  const float psi_c = ring[s0][jc];
  float s[Q];
#pragma unroll
  for (int i = 1; i < Q; ++i) s[i] = ring[cy(i) > 0 ? sp : (cy(i) < 0 ? sm : s0)][jc + cx(i)];
  if (MASKED && m) {
#pragma unroll
    for (int i = 1; i < Q; ++i)
      if ((m >> (i - 1)) & 1u) s[i] = psi_c;
  }
  float Fx, Fy;
  force_of(s, psi_c, p.G, Fx, Fy);
  collide<TAU_ONE, S != LBM_F32>(f, rho, jx, jy, Fx, Fy, p, worst);
#pragma unroll
  for (int i = 0; i < Q; ++i) put_cell(row + (size_t)i * p.plane, x, p.nx, Store<S>::enc(f[i]));
}

// ---------------------------------------------------------------- plain-load kernel
template <int S>
__device__ __forceinline__ void pull_cell(const typename Store<S>::T* __restrict__ src, const StepParams& p,
                                          const Rows3& r, int x, float f[Q]) {
  // f_i(x, r) = f_i^out(x - c_ix, r - c_iy): rows r-1 (c_iy = +1), r, r+1 (c_iy = -1)
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const long long row = (long long)(cy(i) > 0 ? r.m : (cy(i) < 0 ? r.p : r.c)) * p.pitch;
    f[i] = Store<S>::raw(src + ((long long)i * p.plane + row), x - cx(i));
  }
}

template <int S, bool MASKED, bool TAU_ONE>
__global__ void __launch_bounds__(kBX) k_step_strip(const StepParams p) {
  using T = typename Store<S>::T;
  const T* __restrict__ src = static_cast<const T*>(p.src);
  T* __restrict__ dst = static_cast<T*>(p.dst);
  __shared__ float ring[4][kBX + 2];

  const int nx = p.nx, ny = p.ny;
  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * kBX;
  const int x = x0 + tid;
  const bool active = x < nx;
  const int last = min(x0 + kBX, nx) - 1;
  const int y0 = blockIdx.y * p.rows_per_chunk;
  const int y1 = min(y0 + p.rows_per_chunk, ny);
  grid_begin();
  if (y0 >= y1) return;  // uniform over the block
  const int jc = tid + 1;

  float fprev[Q];
  float rho_prev = 1.f, jx_prev = 0.f, jy_prev = 0.f;
  uint32_t worst = 0;
  for (int r = y0 - 1, k = 0; r <= y1; ++r, ++k) {
    const Rows3 rows(r, ny);
    float f[Q];
    float rho = 1.f, jx = 0.f, jy = 0.f;
    if (active) {
      pull_cell<S>(src, p, rows, x, f);
      moments9(f, rho, jx, jy);
      ring[k & 3][jc] = psi_of(full_rho<S != LBM_F32>(rho, p), p);
    }
    if (tid == 0) {
      float h[Q], rh, hx, hy;
      pull_cell<S>(src, p, rows, x0 - 1, h);
      moments9(h, rh, hx, hy);
      ring[k & 3][0] = psi_of(full_rho<S != LBM_F32>(rh, p), p);
    }
    if (x == last) {
      float h[Q], rh, hx, hy;
      pull_cell<S>(src, p, rows, last + 1, h);
      moments9(h, rh, hx, hy);
      ring[k & 3][last - x0 + 2] = psi_of(full_rho<S != LBM_F32>(rh, p), p);
    }
    __syncthreads();
    if (k >= 2 && active) {
      const int rc = r - 1;
      const unsigned m = MASKED ? p.mask[(size_t)rc * p.mpitch + x] : 0u;
      finish_cell<S, MASKED, TAU_ONE>(fprev, rho_prev, jx_prev, jy_prev, m, ring, (k - 2) & 3, (k - 1) & 3,
                                      k & 3, jc, p, dst + (size_t)rc * p.pitch, x, worst);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) fprev[i] = f[i];
    rho_prev = rho;
    jx_prev = jx;
    jy_prev = jy;
  }
  report_faults(worst, p.flags);
}

// ---------------------------------------------------------------- TMA-staged kernel
template <int S>
struct TmaGeom {
  using T = typename Store<S>::T;
  static constexpr int E = sizeof(T);
  static constexpr int PAD = 16 / E;         // halo pad in elements: 16 bytes
  static constexpr int WIN = kBX + 2 * PAD;  // elements per staged plane row
  static constexpr int ROW_BYTES = WIN * E;  // multiple of 16
};

// Issued by the lanes of the ninth warp: lane 0 arms the stage's mbarrier,
// lanes 0..8 copy plane `lane`, lane 9 copies the mask row.
template <int S, bool MASKED, int NSTAGE>
__device__ __forceinline__ void issue_stage(const StepParams& p, const typename Store<S>::T* src,
                                            unsigned char* stages, uint64_t* bars, int k, int y0, int x0,
                                            int lane) {
  using G = TmaGeom<S>;
  using T = typename G::T;
  constexpr uint32_t STAGE_BYTES = Q * G::ROW_BYTES + (MASKED ? kBX : 0);
  const int slot = k % NSTAGE;
  unsigned char* st = stages + (size_t)slot * STAGE_BYTES;
  uint64_t* bar = bars + slot;
  const Rows3 rows(y0 - 1 + k, p.ny);
  if (lane < Q + (MASKED ? 1 : 0)) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (lane == 0) mbar_expect_tx(bar, STAGE_BYTES);
  __syncwarp();
  if (lane < Q) {
    const int i = lane;
    const int g = (i == 2 || i == 5 || i == 6) ? rows.m : ((i == 4 || i == 7 || i == 8) ? rows.p : rows.c);
    bulk_g2s(st + i * G::ROW_BYTES, src + (long long)i * p.plane + (long long)g * p.pitch + (x0 - G::PAD), G::ROW_BYTES,
             bar);
  } else if (MASKED && lane == Q) {
    bulk_g2s(st + Q * G::ROW_BYTES, p.mask + (long long)rows.c * p.mpitch + x0, kBX, bar);
  }
}

template <int S, bool MASKED, int NSTAGE>
constexpr size_t tma_smem_bytes_c() {
  return (size_t)NSTAGE * (Q * TmaGeom<S>::ROW_BYTES + (MASKED ? kBX : 0)) + 4 * (kBX + 2) * 4 + NSTAGE * 8 + 16;
}

template <int S, bool MASKED, bool TAU_ONE, int NSTAGE, int MINB>
__global__ void __launch_bounds__(kTmaThreads, MINB) k_step_tma(const StepParams p) {
  using G = TmaGeom<S>;
  using T = typename G::T;
  constexpr int STAGE_BYTES = Q * G::ROW_BYTES + (MASKED ? kBX : 0);
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char* stages = smem;
  float(*ring)[kBX + 2] = reinterpret_cast<float(*)[kBX + 2]>(smem + (size_t)NSTAGE * STAGE_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)NSTAGE * STAGE_BYTES + 4 * (kBX + 2) * 4);
  int* abort_flag = reinterpret_cast<int*>(bars + NSTAGE);

  const T* __restrict__ src = static_cast<const T*>(p.src);
  T* __restrict__ dst = static_cast<T*>(p.dst);
  const int nx = p.nx, ny = p.ny;
  const int tid = threadIdx.x;
  const bool helper = tid >= kBX;  // the ninth warp
  const int lane = tid & 31;
  const int x0 = blockIdx.x * kBX;
  const int width = min(kBX, nx - x0);
  const bool active = !helper && tid < width;
  const int y0 = blockIdx.y * p.rows_per_chunk;
  const int y1 = min(y0 + p.rows_per_chunk, ny);
  const int nst = (y1 - y0) + 2;  // stages = rows y0-1 .. y1

  if (tid == 0) {
    for (int s = 0; s < NSTAGE; ++s) mbar_init(bars + s, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  grid_begin();
  if (y0 >= y1) return;  // uniform over the block
  if (helper)
    for (int k = 0; k < NSTAGE - 1 && k < nst; ++k) issue_stage<S, MASKED, NSTAGE>(p, src, stages, bars, k, y0, x0, lane);

  // halo lanes of the helper warp: lanes 0..8 pull plane `lane` of the left
  // halo cell (column x0-1), lanes 16..24 of the right one (column x0+width)
  const int hplane = lane & 15;
  const bool hlane = helper && hplane < Q;
  const int hcx = (hplane == 1 || hplane == 5 || hplane == 8) ? 1 : ((hplane == 3 || hplane == 6 || hplane == 7) ? -1 : 0);
  const int hpos = (lane < 16 ? G::PAD - 1 : G::PAD + width) - hcx;

  const int jc = tid + 1;
  const int pos = G::PAD + tid;
  float fprev[Q];
  float rho_prev = 1.f, jx_prev = 0.f, jy_prev = 0.f;
  unsigned m_prev = 0;
  uint32_t worst = 0;
  int k_abort = 0;
  for (int k = 0; k < nst; ++k) {
    const int slot = k % NSTAGE;
    const unsigned char* st = stages + (size_t)slot * STAGE_BYTES;
    if (!mbar_wait(bars + slot, (uint32_t)((k / NSTAGE) & 1))) *abort_flag = 1;
    float f[Q];
    float rho = 1.f, jx = 0.f, jy = 0.f;
    unsigned m = 0;
    if (active) {
#pragma unroll
      for (int i = 0; i < Q; ++i)
        f[i] = Store<S>::raw_smem(reinterpret_cast<const T*>(st + i * G::ROW_BYTES), pos - cx(i));
      moments9(f, rho, jx, jy);
      ring[k & 3][jc] = psi_of(full_rho<S != LBM_F32>(rho, p), p);
      if (MASKED) m = st[Q * G::ROW_BYTES + tid];
    } else if (helper) {
      // same summation order as moments9: ((f0+f1)+(f2+f3)) + ((f4+f5)+(f6+f7)) + f8
      const float v = hlane ? Store<S>::raw_smem(reinterpret_cast<const T*>(st + hplane * G::ROW_BYTES), hpos) : 0.f;
      const float t1 = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 1));
      const float t2 = __fadd_rn(t1, __shfl_xor_sync(0xffffffffu, t1, 2));
      const float t3 = __fadd_rn(t2, __shfl_xor_sync(0xffffffffu, t2, 4));
      const float rh = full_rho<S != LBM_F32>(__fadd_rn(t3, __shfl_xor_sync(0xffffffffu, t2, 8)), p);
      if (lane == 0) ring[k & 3][0] = psi_of(rh, p);
      if (lane == 16) ring[k & 3][width + 1] = psi_of(rh, p);
    }
    __syncthreads();
    if (*abort_flag) {
      k_abort = k;
      break;
    }
    if (helper) {
      if (k + NSTAGE - 1 < nst) issue_stage<S, MASKED, NSTAGE>(p, src, stages, bars, k + NSTAGE - 1, y0, x0, lane);
    } else if (k >= 2 && active) {
      const int rc = y0 + k - 2;  // row collided now
      finish_cell<S, MASKED, TAU_ONE>(fprev, rho_prev, jx_prev, jy_prev, m_prev, ring, (k - 2) & 3, (k - 1) & 3,
                                      k & 3, jc, p, dst + (size_t)rc * p.pitch, x0 + tid, worst);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) fprev[i] = f[i];
    rho_prev = rho;
    jx_prev = jx;
    jy_prev = jy;
    m_prev = m;
  }
  if (*abort_flag) {
    // a stage never completed: record it, then wait (bounded) for the copies
    // of every stage issued and not consumed before the CTA leaves
    if (tid == 0) {
      atomicOr(p.flags + FLAG_TIMEOUT, 1);
      const int issued = min(nst, k_abort + NSTAGE - 1);
      for (int q = k_abort; q < issued; ++q) mbar_wait(bars + q % NSTAGE, (uint32_t)((q / NSTAGE) & 1), 500000000ull);
    }
    __syncthreads();
    return;
  }
  report_faults(worst, p.flags);
}

// ---------------------------------------------------------------- two-cell staged kernel
// The staged march with two neighbouring cells per thread: a CTA owns a
// strip of kBX2 = 512 columns, 256 compute threads (cells 2t and 2t+1) plus
// the helper warp. Pairs are read from the stage with one 32-bit (16-bit
// storage) or 64-bit (FP32) shared load where aligned, and with two loads and
// a byte permute where the pull shifts them by one column; the arithmetic
// runs on float2 (packed FP32); outputs leave as half2/bfloat162/float2.
constexpr int kBX2 = 512;

template <int S>
struct TmaGeom2 {
  using T = typename Store<S>::T;
  static constexpr int E = sizeof(T);
  static constexpr int PAD = 16 / E;
  static constexpr int WIN = kBX2 + 2 * PAD;
  static constexpr int ROW_BYTES = WIN * E;
};

// Two consecutive staged raw values (window positions pos, pos+1) as floats.
template <int S>
__device__ __forceinline__ float2 load_pair(const unsigned char* row, int pos, int shift);

template <>
__device__ __forceinline__ float2 load_pair<LBM_F32>(const unsigned char* row, int pos, int shift) {
  const float* r = reinterpret_cast<const float*>(row);
  if (shift == 0) return *reinterpret_cast<const float2*>(r + pos);  // pos even: 8-byte aligned
  return make_float2(r[pos], r[pos + 1]);
}

__device__ __forceinline__ uint32_t pair_bits_16(const unsigned char* row, int pos, int shift) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(row);
  if (shift == 0) return w[pos >> 1];  // pos even
  // pos odd: high half of the word at pos-1 and low half of the word at pos+1
  return __byte_perm(w[(pos - 1) >> 1], w[(pos + 1) >> 1], 0x5432);
}

// 16-bit pairs are converted element by element with the same conversion as
// the one-cell kernels (the packed conversions gave different results for
// small deviations), so all kernels agree bitwise.
template <>
__device__ __forceinline__ float2 load_pair<LBM_F16_DEV>(const unsigned char* row, int pos, int shift) {
  const uint32_t b = pair_bits_16(row, pos, shift);
  const __half2 h = *reinterpret_cast<const __half2*>(&b);
  return make_float2(__low2float(h), __high2float(h));
}

template <>
__device__ __forceinline__ float2 load_pair<LBM_BF16_DEV>(const unsigned char* row, int pos, int shift) {
  const uint32_t b = pair_bits_16(row, pos, shift);
  const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&b);
  return make_float2(__low2float(h), __high2float(h));
}

template <int S>
__device__ __forceinline__ void store_pair(typename Store<S>::T* dst, size_t idx, float2 v);

template <>
__device__ __forceinline__ void store_pair<LBM_F32>(float* dst, size_t idx, float2 v) {
  *reinterpret_cast<float2*>(dst + idx) = v;  // idx even
}

template <>
__device__ __forceinline__ void store_pair<LBM_F16_DEV>(__half* dst, size_t idx, float2 v) {
  *reinterpret_cast<__half2*>(dst + idx) = __halves2half2(__float2half_rn(v.x), __float2half_rn(v.y));
}

template <>
__device__ __forceinline__ void store_pair<LBM_BF16_DEV>(__nv_bfloat16* dst, size_t idx, float2 v) {
  *reinterpret_cast<__nv_bfloat162*>(dst + idx) = __halves2bfloat162(__float2bfloat16_rn(v.x), __float2bfloat16_rn(v.y));
}

// Layout of one stage slot of the two-cell march: nine plane rows, the mask row.
template <int S, bool MASKED>
struct Slot2 {
  static constexpr int RB = TmaGeom2<S>::ROW_BYTES;  // plane row stride
  static constexpr int BYTES = Q * RB + (MASKED ? kBX2 : 0);
};

// One stage of the two-cell march: for output row r = y0 - 1 + k, plane i's
// source row r - c_iy, columns x0 - PAD .. x0 + width + PAD with the width
// rounded up to 16, and the mask row r, columns x0 .. x0 + width.
template <int S, bool MASKED, int NSTAGE>
__device__ __forceinline__ void issue_stage2(const StepParams& p, const typename Store<S>::T* src,
                                             unsigned char* stages, uint64_t* bars, unsigned gk, int k, int y0,
                                             int x0, int width, int lane) {
  using G = TmaGeom2<S>;
  const int w16 = (width + 15) & ~15;
  const uint32_t row_bytes = (uint32_t)((w16 + 2 * G::PAD) * G::E);
  const int slot = (int)(gk % NSTAGE);
  unsigned char* st = stages + (size_t)slot * Slot2<S, MASKED>::BYTES;
  uint64_t* bar = bars + slot;
  const Rows3 rows(y0 - 1 + k, p.ny);
  if (lane < Q + (MASKED ? 1 : 0)) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (lane == 0) mbar_expect_tx(bar, Q * row_bytes + (MASKED ? w16 : 0));
  __syncwarp();
  if (lane < Q) {
    const int i = lane;
    const int g = (i == 2 || i == 5 || i == 6) ? rows.m : ((i == 4 || i == 7 || i == 8) ? rows.p : rows.c);
    bulk_g2s(st + i * Slot2<S, MASKED>::RB, src + (long long)i * p.plane + (long long)g * p.pitch + (x0 - G::PAD),
             row_bytes, bar);
  } else if (MASKED && lane == Q) {
    bulk_g2s(st + Q * Slot2<S, MASKED>::RB, p.mask + (long long)rows.c * p.mpitch + x0, (uint32_t)w16, bar);
  }
}

template <int S, bool MASKED, int NSTAGE>
constexpr size_t tma2_smem_bytes_c() {
  return (size_t)NSTAGE * Slot2<S, MASKED>::BYTES + 4 * (kBX2 + 4) * 4 + NSTAGE * 8 + 16;
}

template <int S, bool MASKED, int NSTAGE>
struct Tma2Smem {
  static constexpr int RB = Slot2<S, MASKED>::RB;  // plane row stride
  static constexpr int SLOT_BYTES = Slot2<S, MASKED>::BYTES;
  static constexpr int RW = kBX2 + 4;  // ring row: cell column c at index c + 2, halos at 1 and width + 2
  unsigned char* stages;
  float (*ring)[RW];
  uint64_t* bars;
  int* abort_flag;
  __device__ __forceinline__ explicit Tma2Smem(unsigned char* smem) {
    stages = smem;
    ring = reinterpret_cast<float(*)[RW]>(smem + (size_t)NSTAGE * SLOT_BYTES);
    bars = reinterpret_cast<uint64_t*>(smem + (size_t)NSTAGE * SLOT_BYTES + 4 * RW * 4);
    abort_flag = reinterpret_cast<int*>(bars + NSTAGE);
  }
};

// The two-cell march of one work item: columns x0 .. x0 + width (x0 a multiple
// of 16, width at most kBX2) and rows y0 .. y1 of one box. `gstage` counts the
// stages this CTA consumed before (mbarrier phases continue across items).
// Returns false if a stage wait timed out (the CTA must then leave).
template <int S, bool MASKED, bool TAU_ONE, int NSTAGE, bool FULL = false>
__device__ __forceinline__ bool march2(const StepParams& p, const Tma2Smem<S, MASKED, NSTAGE>& sm, int x0,
                                       int width_, int y0, int y1, unsigned& gstage, uint32_t& worst) {
  const int width = FULL ? kBX2 : width_;  // FULL: a whole strip (known at compile time)
  using G = TmaGeom2<S>;
  using T = typename G::T;
  constexpr int SLOT_BYTES = Tma2Smem<S, MASKED, NSTAGE>::SLOT_BYTES;
  constexpr int RB = Tma2Smem<S, MASKED, NSTAGE>::RB;
  const T* __restrict__ src = static_cast<const T*>(p.src);
  T* __restrict__ dst = static_cast<T*>(p.dst);
  const int nx = p.nx;
  const int tid = threadIdx.x;
  const bool helper = tid >= kBX;
  const int lane = tid & 31;
  const int x = x0 + 2 * tid;  // the pair's first column
  const bool active = !helper && 2 * tid < width;
  // with an odd width the last pair's second cell is the right halo cell
  // (computed for its psi only); pairs in the outer columns write ghosts
  const bool edge = active && (x < 2 || x + 1 >= nx - 2);
  const int nst = (y1 - y0) + 2;  // stages = rows y0-1 .. y1
  const unsigned g0 = gstage;

  if (helper)
    for (int k = 0; k < NSTAGE - 1 && k < nst; ++k)
      issue_stage2<S, MASKED, NSTAGE>(p, src, sm.stages, sm.bars, g0 + k, k, y0, x0, width, lane);

  const int hplane = lane & 15;
  const bool hlane = helper && hplane < Q;
  const int hcx = (hplane == 1 || hplane == 5 || hplane == 8) ? 1 : ((hplane == 3 || hplane == 6 || hplane == 7) ? -1 : 0);
  const int hpos = (lane < 16 ? G::PAD - 1 : G::PAD + width) - hcx;

  const int jc = 2 * tid + 2;        // ring index of the first cell of the pair
  const int pos = G::PAD + 2 * tid;  // window position of the first cell
  float2 fprev[Q];
  float2 rho_prev = make_float2(1.f, 1.f), jx_prev = make_float2(0.f, 0.f), jy_prev = make_float2(0.f, 0.f);
  unsigned m_prev = 0;
  int k_abort = -1;
  for (int k = 0; k < nst; ++k) {
    const unsigned gk = g0 + k;
    const unsigned char* st = sm.stages + (size_t)(gk % NSTAGE) * SLOT_BYTES;
    if (!mbar_wait(sm.bars + gk % NSTAGE, (gk / NSTAGE) & 1u)) *sm.abort_flag = 1;
    float2 f[Q];
    float2 rho = make_float2(1.f, 1.f), jx = make_float2(0.f, 0.f), jy = make_float2(0.f, 0.f);
    unsigned m = 0;
    if (active) {
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = load_pair<S>(st + i * RB, pos - cx(i), cx(i));
      moments9(f, rho, jx, jy);
      *reinterpret_cast<float2*>(&sm.ring[k & 3][jc]) = psi_of(full_rho<S != LBM_F32>(rho, p), p);
      if (MASKED) m = *reinterpret_cast<const uint16_t*>(st + Q * RB + 2 * tid);
    } else if (helper) {
      const float v = hlane ? Store<S>::raw_smem(reinterpret_cast<const T*>(st + hplane * RB), hpos) : 0.f;
      const float t1 = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 1));
      const float t2 = __fadd_rn(t1, __shfl_xor_sync(0xffffffffu, t1, 2));
      const float t3 = __fadd_rn(t2, __shfl_xor_sync(0xffffffffu, t2, 4));
      const float rh = full_rho<S != LBM_F32>(__fadd_rn(t3, __shfl_xor_sync(0xffffffffu, t3, 8)), p);
      if (lane == 0) sm.ring[k & 3][1] = psi_of(rh, p);
      if (lane == 16) sm.ring[k & 3][width + 2] = psi_of(rh, p);
    }
    __syncthreads();
    if (*sm.abort_flag) {
      k_abort = k;
      break;
    }
    if (helper) {
      if (k + NSTAGE - 1 < nst)
        issue_stage2<S, MASKED, NSTAGE>(p, src, sm.stages, sm.bars, gk + NSTAGE - 1, k + NSTAGE - 1, y0, x0, width,
                                        lane);
    } else if (k >= 2 && active) {
      const int rc = y0 + k - 2;
      const int srow[3] = {(k - 2) & 3, (k - 1) & 3, k & 3};  // rows rc-1, rc, rc+1
      float2 nb[3][3];  // [row][left, centre, right] for the pair
#pragma unroll
      for (int r3 = 0; r3 < 3; ++r3) {
        const float* rr = sm.ring[srow[r3]];
        const float2 c2 = *reinterpret_cast<const float2*>(rr + jc);
        nb[r3][0] = make_float2(rr[jc - 1], c2.x);
        nb[r3][1] = c2;
        nb[r3][2] = make_float2(c2.y, rr[jc + 2]);
      }
      const float2 psi_c = nb[1][1];
      float2 sv[Q];
#pragma unroll
      for (int i = 1; i < Q; ++i) sv[i] = nb[cy(i) + 1][cx(i) + 1];
      if (MASKED && m_prev) {
        const unsigned ma = m_prev & 0xffu, mb = m_prev >> 8;
#pragma unroll
        for (int i = 1; i < Q; ++i) {
          if ((ma >> (i - 1)) & 1u) sv[i].x = psi_c.x;
          if ((mb >> (i - 1)) & 1u) sv[i].y = psi_c.y;
        }
      }
      float2 Fx, Fy;
      force_of(sv, psi_c, p.G, Fx, Fy);
      collide<TAU_ONE, S != LBM_F32>(fprev, rho_prev, jx_prev, jy_prev, Fx, Fy, p, worst);
      T* row = dst + (size_t)rc * p.pitch;
      if (!edge) {
#pragma unroll
        for (int i = 0; i < Q; ++i) store_pair<S>(row + (size_t)i * p.plane, x, fprev[i]);
      } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
          T* q = row + (size_t)i * p.plane;
          put_cell(q, x, nx, Store<S>::enc(fprev[i].x));
          if (x + 1 < nx) put_cell(q, x + 1, nx, Store<S>::enc(fprev[i].y));
        }
      }
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) fprev[i] = f[i];
    rho_prev = rho;
    jx_prev = jx;
    jy_prev = jy;
    m_prev = m;
  }
  if (k_abort >= 0) {
    // a stage never completed: record it, then wait (bounded) for the copies
    // of every stage issued and not consumed before the CTA leaves
    if (tid == 0) {
      atomicOr(p.flags + FLAG_TIMEOUT, 1);
      const int issued = min(nst, k_abort + NSTAGE - 1);
      for (int q = k_abort; q < issued; ++q)
        mbar_wait(sm.bars + (g0 + q) % NSTAGE, ((g0 + q) / NSTAGE) & 1u, 500000000ull);
    }
    __syncthreads();
    return false;
  }
  gstage = g0 + nst;
  return true;
}

template <int S, bool MASKED, int NSTAGE>
__device__ __forceinline__ void march2_init(const Tma2Smem<S, MASKED, NSTAGE>& sm) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) mbar_init(sm.bars + s, 1);
    *sm.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  grid_begin();
}

// One box, one work item per CTA: strip blockIdx.x (kBX2 columns), row chunk blockIdx.y.
template <int S, bool MASKED, bool TAU_ONE, int NSTAGE, int MINB>
__global__ void __launch_bounds__(kTmaThreads, MINB) k_step_tma2(const StepParams p) {
  extern __shared__ __align__(128) unsigned char smem[];
  const Tma2Smem<S, MASKED, NSTAGE> sm(smem);
  const int x0 = blockIdx.x * kBX2;
  const int y0 = blockIdx.y * p.rows_per_chunk;
  const int y1 = min(y0 + p.rows_per_chunk, p.ny);
  march2_init(sm);
  if (y0 >= y1) return;
  unsigned gstage = 0;
  uint32_t worst = 0;
  const int width = min(kBX2, p.nx - x0);
  const bool ok = width == kBX2
                      ? march2<S, MASKED, TAU_ONE, NSTAGE, true>(p, sm, x0, width, y0, y1, gstage, worst)
                      : march2<S, MASKED, TAU_ONE, NSTAGE, false>(p, sm, x0, width, y0, y1, gstage, worst);
  if (!ok) return;
  report_faults(worst, p.flags);
}

// One box, dynamically scheduled: as many CTAs as fit take row chunks (of
// `rows` rows, gx strips) from a device counter until all are done. With
// chunks a few times shorter than a static split, CTAs that march fast take
// more chunks and the launch does not wait for the slowest of
// one-chunk-per-CTA (8192^2: FP32 0.817 -> 0.757 ms, FP16 0.509 -> 0.481
// ms). The counters are zero between launches: the last CTA to finish
// resets them.
template <int S, bool MASKED, bool TAU_ONE, int NSTAGE, int MINB>
__global__ void __launch_bounds__(kTmaThreads, MINB) k_step_dyn(const StepParams p, int rows, int gx, int nitems) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int item_sh;
  const Tma2Smem<S, MASKED, NSTAGE> sm(smem);
  march2_init(sm);
  int* counter = p.flags + FLAG_ITEM;
  unsigned gstage = 0;
  uint32_t worst = 0;
  for (int guard = 0; guard < nitems + 1; ++guard) {
    __syncthreads();  // the previous chunk's ring and item index are no longer read
    if (threadIdx.x == 0) item_sh = atomicAdd(counter, 1);
    __syncthreads();
    const int w = item_sh;
    if (w >= nitems) break;
    // row-major chunk order: the strips of a chunk row run together, so
    // the halo columns a strip shares with its neighbours are read while
    // still in L2 (measured for 16-bit storage at 8192^2 after the packed
    // arithmetic: 0.459 ms strip by strip, 0.450 row-major)
    const int sx = w % gx, cyk = w / gx;
    const int x0 = sx * kBX2, y0 = cyk * rows;
    const int y1 = min(y0 + rows, p.ny), width = min(kBX2, p.nx - x0);
    // full strips take the compile-time-width march (with tau != 1 the two
    // inlined copies would spill at this kernel's register budget)
    const bool ok = TAU_ONE && width == kBX2
                        ? march2<S, MASKED, TAU_ONE, NSTAGE, TAU_ONE>(p, sm, x0, width, y0, y1, gstage, worst)
                        : march2<S, MASKED, TAU_ONE, NSTAGE, false>(p, sm, x0, width, y0, y1, gstage, worst);
    if (!ok) break;  // a stage wait timed out (recorded); no further chunks
  }
  report_faults(worst, p.flags);
  __syncthreads();
  if (threadIdx.x == 0) {
    // every CTA arrives here after its last draw from the counter
    if (atomicAdd(p.flags + FLAG_DONE, 1) == (int)gridDim.x - 1) {
      *counter = 0;
      p.flags[FLAG_DONE] = 0;
    }
  }
}

// Many boxes in one launch: persistent CTAs take work items (box, strip,
// row chunk) from a device counter until the list is exhausted. Each box
// reads buffer `cur ^ parity` and writes the other. Launches alternate
// parity, so two counters take turns: this launch draws from
// counters[parity] and zeroes counters[parity ^ 1] for the next one (which
// starts only after this one has finished), so no reset is launched.
template <int S, bool MASKED, bool TAU_ONE, int NSTAGE, int MINB>
__global__ void __launch_bounds__(kTmaThreads, MINB)
    k_step_batch(const BatchInst* __restrict__ insts, const BatchItem* __restrict__ items, int nitems,
                 int* __restrict__ counters, int parity) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int item_sh;
  const Tma2Smem<S, MASKED, NSTAGE> sm(smem);
  march2_init(sm);
  int* counter = counters + parity;
  if (blockIdx.x == 0 && threadIdx.x == 0) counters[parity ^ 1] = 0;
  unsigned gstage = 0;
  for (int guard = 0; guard < nitems + 1; ++guard) {
    __syncthreads();  // the previous item's ring and item index are no longer read
    if (threadIdx.x == 0) item_sh = atomicAdd(counter, 1);
    __syncthreads();
    const int w = item_sh;
    if (w >= nitems) break;
    const BatchItem it = items[w];
    const BatchInst& in = insts[it.inst];
    StepParams p{};
    const int c = in.cur ^ parity;
    p.src = c ? in.pops1 : in.pops0;
    p.dst = c ? in.pops0 : in.pops1;
    p.mask = in.mask;
    p.flags = in.flags;
    p.nx = in.nx;
    p.ny = in.ny;
    p.pitch = in.pitch;
    p.mpitch = in.mpitch;
    p.plane = in.plane;
    p.tau = in.tau;
    p.inv_tau = in.inv_tau;
    p.G = in.G;
    p.rho0 = in.rho0;
    p.inv_rho0 = in.inv_rho0;
    p.rho_ref = in.rho_ref;
    uint32_t worst = 0;
    bool ok;
    if (TAU_ONE && it.width == kBX2)  // full strips take the compile-time-width march
      ok = march2<S, MASKED, TAU_ONE, NSTAGE, TAU_ONE>(p, sm, it.x0, it.width, it.y0, it.y1, gstage, worst);
    else if (!TAU_ONE && in.tau_one)  // a tau = 1 box among others: the collision it takes alone
      ok = march2<S, MASKED, true, NSTAGE, false>(p, sm, it.x0, it.width, it.y0, it.y1, gstage, worst);
    else  // (with tau != 1 a third copy would spill at this kernel's register budget)
      ok = march2<S, MASKED, TAU_ONE, NSTAGE, false>(p, sm, it.x0, it.width, it.y0, it.y1, gstage, worst);
    if (!ok) return;
    report_faults(worst, p.flags);
  }
}

// Stage ring depth and CTAs per SM, from measured sweeps at 8192^2: with
// four CTAs per SM, prefetching two rows ahead (FP32) gave more DRAM
// throughput than deeper rings (more reads in flight lowered it).
template <int S>
constexpr int tma_stages() { return S == LBM_F32 ? 3 : 6; }
constexpr int kTmaMinBlocks = 4;

template <int S>
bool tma_ok(int nx) {
  return nx % 16 == 0 && nx >= TmaGeom<S>::WIN;
}
inline bool tma2_ok(int nx) { return nx >= 16; }

int sm_count() { return device_sm_count(); }

// Rows per chunk so that all CTAs are resident at once (one wave).
void tma_geometry(int nx, int ny, int resident_per_sm, int* gx, int* gy, int* rows) {
  *gx = (nx + kBX - 1) / kBX;
  const int resident = resident_per_sm * sm_count();
  int g = resident / *gx;
  if (g < 1) g = 1;
  if (g > ny) g = ny;
  *rows = (ny + g - 1) / g;
  *gy = (ny + *rows - 1) / *rows;
}

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_tma(const StepParams& p, cudaStream_t s) {
  constexpr int NS = tma_stages<S>();
  auto kern = k_step_tma<S, MASKED, TAU_ONE, NS, kTmaMinBlocks>;
  constexpr size_t smem = tma_smem_bytes_c<S, MASKED, NS>();
  static PerDevice per_sm;  // per instantiation
  int resident = 0;
  LBM_TRY(per_sm.get([&](int* n) { return ctas_per_sm(kern, kTmaThreads, smem, n); }, &resident));
  int gx, gy, rows;
  tma_geometry(p.nx, p.ny, resident, &gx, &gy, &rows);
  StepParams q = p;
  q.rows_per_chunk = rows;
  return launch_chain(kern, dim3(gx, gy), dim3(kTmaThreads), smem, s, q);
}

// Measured at 8192^2 (FP16): 4 stages at 4 CTAs per SM (56 registers, no
// spills) beat deeper rings and 3 or 5 CTAs per SM.
template <int S>
constexpr int tma2_stages() { return S == LBM_F32 ? 3 : 4; }
// FP32 stages allow 3 CTAs per SM: its register budget follows
template <int S, bool TAU_ONE>
constexpr int tma2_min_blocks() { return TAU_ONE ? (S == LBM_F32 ? 3 : 4) : 2; }
constexpr int kDynRows = 48;  // row chunk of the dynamically scheduled step

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_tma2(const StepParams& p, cudaStream_t s) {
  constexpr int NS = tma2_stages<S>();
  // the relaxation blend (tau != 1) keeps both population sets live: fewer CTAs
  auto kern = k_step_tma2<S, MASKED, TAU_ONE, NS, tma2_min_blocks<S, TAU_ONE>()>;
  constexpr size_t smem = tma2_smem_bytes_c<S, MASKED, NS>();
  static PerDevice per_sm;  // per instantiation
  int resident = 0;
  LBM_TRY(per_sm.get([&](int* n) { return ctas_per_sm(kern, kTmaThreads, smem, n); }, &resident));
  const int gx = (p.nx + kBX2 - 1) / kBX2;
  int g = resident * sm_count() / gx;
  if (g < 1) g = 1;
  if (g > p.ny) g = p.ny;
  StepParams q = p;
  q.rows_per_chunk = (p.ny + g - 1) / g;
  const int gy = (p.ny + q.rows_per_chunk - 1) / q.rows_per_chunk;
  return launch_chain(kern, dim3(gx, gy), dim3(kTmaThreads), smem, s, q);
}

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_dyn(const StepParams& p, cudaStream_t s) {
  constexpr int NS = tma2_stages<S>();
  auto kern = k_step_dyn<S, MASKED, TAU_ONE, NS, tma2_min_blocks<S, TAU_ONE>()>;
  constexpr size_t smem = tma2_smem_bytes_c<S, MASKED, NS>();
  static PerDevice per_sm;  // per instantiation
  int resident = 0;         // CTAs that fit the GPU at once
  LBM_TRY(per_sm.get([&](int* n) { return ctas_per_sm(kern, kTmaThreads, smem, n); }, &resident));
  resident *= sm_count();
  const int gx = (p.nx + kBX2 - 1) / kBX2;
  // 48-row chunks (best at 8192^2: 4.5 waves of 608 CTAs for 16-bit
  // storage, 6 of 456 for FP32) unless they make fewer than four waves;
  // then whole waves: the fewest for 16-bit storage, at least four for FP32
  // (4096^2: FP16 0.170 -> 0.135 ms, FP32 0.214 -> 0.205 ms;
  // 5120^2: 0.224 -> 0.207, 0.320 -> 0.309; 6144^2: 0.305 -> 0.287,
  // 0.442 -> 0.437). A box of at most one wave gets one chunk per CTA.
  const int rows = dyn_chunk_rows(gx, p.ny, resident, kDynRows, 4, S == LBM_F32 ? 4 : 1);
  const long long items = (long long)gx * ((p.ny + rows - 1) / rows);
  if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int nitems = (int)items;
  // automatic choice: with no more chunks than resident CTAs there is nothing
  // to balance, and the static split saves the counter's round trips (a
  // few microseconds, a large part of a small box's step)
  if (p.force_generic == 0 && nitems <= resident) return launch_tma2<S, MASKED, TAU_ONE>(p, s);
  const int grid = nitems < resident ? nitems : resident;
  return launch_chain(kern, dim3(grid), dim3(kTmaThreads), smem, s, p, rows, gx, nitems);
}

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_strip(const StepParams& p, cudaStream_t s) {
  int gx, gy, rows, block;
  step_geometry(p.nx, p.ny, &gx, &gy, &rows, &block);
  StepParams q = p;
  q.rows_per_chunk = rows;
  return launch_chain(k_step_strip<S, MASKED, TAU_ONE>, dim3(gx, gy), dim3(block), 0, s, q);
}

// Variant 0 (automatic): the tile kernel in its range (step_tiles; the two
// times are in tile.cu), beyond it the two-cell staged march over dynamically
// scheduled row chunks (8192^2 FP16 434 us against 485 in tiles; boxes with no
// more chunks than resident CTAs take the static split of variant 3). 1: plain
// loads; 2: one-cell staged; 3: two-cell staged, one chunk per CTA; 4: two-cell
// staged, dynamic chunks; plain loads where the box does not allow these.
template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_variant(const StepParams& p, cudaStream_t s) {
  const int v = p.force_generic;
  if (step_tiles(S, p)) return launch_tile(S, p, s);
  if ((v == 4 || v == 0) && tma2_ok(p.nx)) return launch_dyn<S, MASKED, TAU_ONE>(p, s);
  if (v == 3 && tma2_ok(p.nx)) return launch_tma2<S, MASKED, TAU_ONE>(p, s);
  if (v == 2 && tma_ok<S>(p.nx)) return launch_tma<S, MASKED, TAU_ONE>(p, s);
  return launch_strip<S, MASKED, TAU_ONE>(p, s);
}

template <int S>
cudaError_t launch_typed(const StepParams& p, cudaStream_t s) {
  const bool tau_one = p.tau == 1.0f;
  if (p.mask) return tau_one ? launch_variant<S, true, true>(p, s) : launch_variant<S, true, false>(p, s);
  return tau_one ? launch_variant<S, false, true>(p, s) : launch_variant<S, false, false>(p, s);
}

}  // namespace

int device_sm_count() {
  static PerDevice sms;
  int n = 0;
  auto ask = [](int* out) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? cudaDeviceGetAttribute(out, cudaDevAttrMultiProcessorCount, dev) : e;
  };
  return sms.get(ask, &n) == cudaSuccess && n > 0 ? n : 152;
}

void step_geometry(int nx, int ny, int* grid_x, int* grid_y, int* rows_per_chunk, int* block) {
  const int gx = (nx + kBX - 1) / kBX;
  const int target = device_sm_count() * 6;  // CTAs: a few per SM
  int gy = (target + gx - 1) / gx;
  if (gy > ny) gy = ny;
  if (gy < 1) gy = 1;
  int rows = (ny + gy - 1) / gy;
  gy = (ny + rows - 1) / rows;
  *grid_x = gx;
  *grid_y = gy;
  *rows_per_chunk = rows;
  *block = kBX;
}

// ---------------------------------------------------------------- batched launch
namespace {

template <int S, bool MASKED, bool TAU_ONE>
struct BatchKernel {
  static constexpr int NS = tma2_stages<S>();
  static constexpr int MINB = tma2_min_blocks<S, TAU_ONE>();
  static constexpr size_t SMEM = tma2_smem_bytes_c<S, MASKED, NS>();
  static int resident() {  // CTAs that fit the GPU at once
    static PerDevice per_sm;
    int n = 0;
    auto ask = [](int* out) { return ctas_per_sm(k_step_batch<S, MASKED, TAU_ONE, NS, MINB>, kTmaThreads, SMEM, out); };
    return per_sm.get(ask, &n) == cudaSuccess ? n * sm_count() : 0;
  }
  static cudaError_t launch(const BatchInst* insts, const BatchItem* items, int nitems, int* counters, int parity,
                            cudaStream_t s) {
    const int res = resident();
    if (res == 0) return cudaErrorInvalidConfiguration;
    const int grid = nitems < res ? nitems : res;
    if (grid <= 0) return cudaMemsetAsync(counters, 0, 2 * sizeof(int), s);  // no launch resets them
    return launch_chain(k_step_batch<S, MASKED, TAU_ONE, NS, MINB>, dim3(grid), dim3(kTmaThreads), SMEM, s, insts, items,
                        nitems, counters, parity);
  }
};

template <int S>
cudaError_t launch_batch_s(bool masked, bool tau_one, const BatchInst* insts, const BatchItem* items, int nitems,
                           int* counter, int parity, cudaStream_t s) {
  if (masked)
    return tau_one ? BatchKernel<S, true, true>::launch(insts, items, nitems, counter, parity, s)
                   : BatchKernel<S, true, false>::launch(insts, items, nitems, counter, parity, s);
  return tau_one ? BatchKernel<S, false, true>::launch(insts, items, nitems, counter, parity, s)
                 : BatchKernel<S, false, false>::launch(insts, items, nitems, counter, parity, s);
}

template <int S>
int batch_resident_s(bool masked, bool tau_one) {
  if (masked)
    return tau_one ? BatchKernel<S, true, true>::resident() : BatchKernel<S, true, false>::resident();
  return tau_one ? BatchKernel<S, false, true>::resident() : BatchKernel<S, false, false>::resident();
}

}  // namespace

cudaError_t launch_step_batch(int storage, bool masked, bool tau_one, const BatchInst* insts, const BatchItem* items,
                              int nitems, int* counter, int parity, cudaStream_t s) {
  switch (storage) {
    case LBM_F32: return launch_batch_s<LBM_F32>(masked, tau_one, insts, items, nitems, counter, parity, s);
    case LBM_F16_DEV: return launch_batch_s<LBM_F16_DEV>(masked, tau_one, insts, items, nitems, counter, parity, s);
    case LBM_BF16_DEV: return launch_batch_s<LBM_BF16_DEV>(masked, tau_one, insts, items, nitems, counter, parity, s);
    default: return cudaErrorInvalidValue;
  }
}

int batch_resident_ctas(int storage, bool masked, bool tau_one) {
  switch (storage) {
    case LBM_F32: return batch_resident_s<LBM_F32>(masked, tau_one);
    case LBM_F16_DEV: return batch_resident_s<LBM_F16_DEV>(masked, tau_one);
    case LBM_BF16_DEV: return batch_resident_s<LBM_BF16_DEV>(masked, tau_one);
    default: return 0;
  }
}

bool step_tma_allowed(int storage, int nx) {
  return storage == LBM_F32 ? tma_ok<LBM_F32>(nx)
                            : (storage == LBM_F16_DEV ? tma_ok<LBM_F16_DEV>(nx) : tma_ok<LBM_BF16_DEV>(nx));
}

bool step_tma2_allowed(int nx) { return tma2_ok(nx); }

cudaError_t launch_step(int storage, const StepParams& p, cudaStream_t s) {
  switch (storage) {
    case LBM_F32: return launch_typed<LBM_F32>(p, s);
    case LBM_F16_DEV: return launch_typed<LBM_F16_DEV>(p, s);
    case LBM_BF16_DEV: return launch_typed<LBM_BF16_DEV>(p, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbm
