// Fused time step over tiles of a few rows: k_step_tile (one box) and
// k_step_tile_batch (many). It serves every box but those that the staged march
// of step.cu steps faster: above 30 M cells for 16-bit storage at tau = 1, above
// 1.5 M for FP32 at tau != 1 (Tiles).
//
// A CTA takes a few rows of a strip of columns, one warp per row and one for
// the halo row on either side. Each lane owns 2 P neighbouring cells;
// lanes 0 and 31 own the halo columns that a pull and a force need. A warp
// issues all its loads at once (one vector load per lane and plane); the
// planes the pull shifts by a column and the neighbours' psi come by shuffles;
// psi of the rows passes through shared memory, and one barrier later each
// warp collides and stores its row from registers. A step is one load latency,
// one barrier and one store, every box of any width gives as many CTAs as the
// GPU holds; what it repeats is the moments of the two halo rows and two lanes in
// 32. (The staged march of step.cu reads every row once and
// keeps HBM busiest, but pays a bulk copy's latency and a barrier per row.)
#include "cellmath.cuh"
#include "launch.cuh"

namespace lbm {
namespace {

constexpr unsigned kAll = 0xffffffffu;

// One box as the kernel takes it: planes and mask as byte pointers to their
// rows' starts, so that a lane's address is a uniform base and a 32-bit offset.
struct TileBox {
  const char* src[Q];
  char* dst[Q];
  const char* mask;  // nullptr: plain Shan-Chen
  int* flags;
  int nx, ny;
  uint32_t row_bytes, mask_row;  // strides
  int reverse;                   // tiles from the last to the first
  int pull_bounce;               // src holds populations that have not bounced back yet
  StepParams s;                  // constants of the arithmetic
};

// Stored words of a lane's 2 P cells.
template <int S, int P>
struct Words;
template <>
struct Words<LBM_F32, 1> {
  using V = float2;
};
template <>
struct Words<LBM_F32, 2> {
  using V = float4;
};
template <>
struct Words<LBM_F16_DEV, 1> {
  using V = uint32_t;
};
template <>
struct Words<LBM_F16_DEV, 2> {
  using V = uint2;
};
template <>
struct Words<LBM_BF16_DEV, 1> {
  using V = uint32_t;
};
template <>
struct Words<LBM_BF16_DEV, 2> {
  using V = uint2;
};

template <int S>
__device__ __forceinline__ float2 decode(uint32_t b) {
  if constexpr (S == LBM_F16_DEV) {
    const __half2 h = *reinterpret_cast<const __half2*>(&b);
    return make_float2(__low2float(h), __high2float(h));
  } else {
    return make_float2(__uint_as_float(b << 16), __uint_as_float(b & 0xffff0000u));
  }
}

template <int S>
__device__ __forceinline__ uint32_t encode(float2 v) {
  if constexpr (S == LBM_F16_DEV) {
    const __half2 h = __halves2half2(__float2half_rn(v.x), __float2half_rn(v.y));
    return *reinterpret_cast<const uint32_t*>(&h);
  } else {
    const __nv_bfloat162 h = __halves2bfloat162(__float2bfloat16_rn(v.x), __float2bfloat16_rn(v.y));
    return *reinterpret_cast<const uint32_t*>(&h);
  }
}

// The pairs of values a pull by CX takes for the lane's cells, f(x) = raw(x - CX).
template <int S, int P, int CX>
__device__ __forceinline__ void pulled(typename Words<S, P>::V w, float2 (&f)[P]) {
  if constexpr (S == LBM_F32) {
    if constexpr (P == 1) {
      if constexpr (CX > 0) f[0] = make_float2(__shfl_up_sync(kAll, w.y, 1), w.x);
      else if constexpr (CX < 0) f[0] = make_float2(w.y, __shfl_down_sync(kAll, w.x, 1));
      else f[0] = w;
    } else {
      if constexpr (CX > 0) {
        f[0] = make_float2(__shfl_up_sync(kAll, w.w, 1), w.x);
        f[1] = make_float2(w.y, w.z);
      } else if constexpr (CX < 0) {
        f[0] = make_float2(w.y, w.z);
        f[1] = make_float2(w.w, __shfl_down_sync(kAll, w.x, 1));
      } else {
        f[0] = make_float2(w.x, w.y);
        f[1] = make_float2(w.z, w.w);
      }
    }
  } else if constexpr (P == 1) {
    if constexpr (CX > 0) f[0] = decode<S>(__byte_perm(__shfl_up_sync(kAll, w, 1), w, 0x5432));
    else if constexpr (CX < 0) f[0] = decode<S>(__byte_perm(w, __shfl_down_sync(kAll, w, 1), 0x5432));
    else f[0] = decode<S>(w);
  } else {
    if constexpr (CX > 0) {
      f[0] = decode<S>(__byte_perm(__shfl_up_sync(kAll, w.y, 1), w.x, 0x5432));
      f[1] = decode<S>(__byte_perm(w.x, w.y, 0x5432));
    } else if constexpr (CX < 0) {
      f[0] = decode<S>(__byte_perm(w.x, w.y, 0x5432));
      f[1] = decode<S>(__byte_perm(w.y, __shfl_down_sync(kAll, w.x, 1), 0x5432));
    } else {
      f[0] = decode<S>(w.x);
      f[1] = decode<S>(w.y);
    }
  }
}

template <int S, int P>
__device__ __forceinline__ typename Words<S, P>::V words(const float2 (&v)[P]) {
  if constexpr (S == LBM_F32) {
    if constexpr (P == 1) return v[0];
    else return make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  } else {
    if constexpr (P == 1) return encode<S>(v[0]);
    else return make_uint2(encode<S>(v[0]), encode<S>(v[1]));
  }
}

// psi of a row's cells and of their left and right neighbours.
template <int P>
struct PsiRow {
  float2 l[P], c[P], r[P];
  __device__ __forceinline__ void set(const float2 (&v)[P]) {
    const float left = __shfl_up_sync(kAll, v[P - 1].y, 1), right = __shfl_down_sync(kAll, v[0].x, 1);
#pragma unroll
    for (int q = 0; q < P; ++q) {
      l[q] = make_float2(q ? v[q ? q - 1 : 0].y : left, v[q].x);
      c[q] = v[q];
      r[q] = make_float2(v[q].y, q + 1 < P ? v[q + 1 < P ? q + 1 : q].x : right);
    }
  }
};

// A tile: P pairs of cells per lane, 30 lanes with cells of their own, ROWS
// rows; CTAS per SM is what the register budget is set for.
template <int P_, int ROWS_, int CTAS_>
struct Tile {
  static constexpr int P = P_, ROWS = ROWS_, CTAS = CTAS_, COLS = 60 * P_, THREADS = 32 * (ROWS_ + 2);
};

// Columns xo .. xo + COLS (xo a multiple of it) and rows y0 .. y1 (at most
// ROWS) of box b; all threads of the CTA.
template <int S, bool MASKED, bool TAU_ONE, typename G>
__device__ __forceinline__ void tile_step(const TileBox& b, int xo, int y0, int y1) {
  constexpr int P = G::P;
  using T = typename Store<S>::T;
  using V = typename Words<S, P>::V;
  constexpr int E = sizeof(T), C = 2 * P;
  // before the addresses: formed ahead of the wait they cost registers (FP32
  // 8192^2 740 us against 696)
  grid_begin();
  __shared__ float2 ring[G::ROWS + 2][P][32];
  const int lane = threadIdx.x & 31, w = __shfl_sync(kAll, (int)(threadIdx.x >> 5), 0);
  const int nx = b.nx, ny = b.ny;
  const int r = y0 - 1 + w;           // this warp's row
  const int x = xo - C + C * lane;    // the lane's first column
  const int xl = min(x, (nx + 1) / C * C);  // lanes beyond the right ghosts read the last cells again
  const uint32_t xb = (uint32_t)(kRowPad + xl * E);
  const int r0 = r < 0 ? r + ny : (r >= ny ? r - ny : r);
  const int rm = r0 == 0 ? ny - 1 : r0 - 1, rp = r0 == ny - 1 ? 0 : r0 + 1;
  const uint32_t o0 = (uint32_t)r0 * b.row_bytes + xb, om = (uint32_t)rm * b.row_bytes + xb,
                 op = (uint32_t)rp * b.row_bytes + xb;
  float2 rho[P], jx[P], jy[P], psi[P], g[Q][P];
  PsiRow<P> B;
  unsigned mask = 0;  // a byte per cell
  if (r <= y1) {
    V raw[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i)
      raw[i] = __ldcg(reinterpret_cast<const V*>(b.src[i] + (cy(i) > 0 ? om : (cy(i) < 0 ? op : o0))));
    if (MASKED) {
      const char* m = b.mask + ((uint32_t)r0 * b.mask_row + (uint32_t)(kMaskPad + xl));
      mask = P == 1 ? __ldcg(reinterpret_cast<const unsigned short*>(m)) : __ldcg(reinterpret_cast<const unsigned*>(m));
    }
    pulled<S, P, cx(0)>(raw[0], g[0]);
    pulled<S, P, cx(1)>(raw[1], g[1]);
    pulled<S, P, cx(2)>(raw[2], g[2]);
    pulled<S, P, cx(3)>(raw[3], g[3]);
    pulled<S, P, cx(4)>(raw[4], g[4]);
    pulled<S, P, cx(5)>(raw[5], g[5]);
    pulled<S, P, cx(6)>(raw[6], g[6]);
    pulled<S, P, cx(7)>(raw[7], g[7]);
    pulled<S, P, cx(8)>(raw[8], g[8]);
    if (MASKED && b.pull_bounce && mask) {
      // the step before left its bounce-back to this pull: what would have
      // come across a blocked edge (x, x + e_i) is the cell's own outgoing
      // population i, returning as opp(i) (film cells only)
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const T* own = reinterpret_cast<const T*>(b.src[i] + o0);
#pragma unroll
        for (int q = 0; q < P; ++q) {
          if ((mask >> (16 * q + i - 1)) & 1u) g[opp(i)][q].x = Store<S>::raw(own, 2 * q);
          if ((mask >> (16 * q + i + 7)) & 1u) g[opp(i)][q].y = Store<S>::raw(own, 2 * q + 1);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < P; ++q) {
      float2 f[Q];
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] = g[i][q];
      moments9(f, rho[q], jx[q], jy[q]);
      psi[q] = psi_of(full_rho<S != LBM_F32>(rho[q], b.s), b.s);
      ring[w][q][lane] = psi[q];
    }
    B.set(psi);
  }
  __syncthreads();
  if (w == 0 || r >= y1) return;  // halo rows
  float2 above[P], below[P];
#pragma unroll
  for (int q = 0; q < P; ++q) {
    above[q] = ring[w - 1][q][lane];
    below[q] = ring[w + 1][q][lane];
  }
  PsiRow<P> A, N;
  A.set(above);
  N.set(below);
  const bool out = lane >= 1 && lane <= 30 && x < nx;
  const bool full = out && x + C <= nx;
  const bool edge = out && (x < 2 || x + C > nx - 2);
  uint32_t worst = 0;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    float2 Fx, Fy, f[Q];
    const float2 s[Q] = {B.c[q], B.r[q], N.c[q], B.l[q], A.c[q], N.r[q], N.l[q], A.l[q], A.r[q]};
    if (MASKED && mask) {  // a path of its own keeps the other free of copies
      float2 v[Q];
      const unsigned ma = (mask >> (16 * q)) & 0xffu, mb = (mask >> (16 * q + 8)) & 0xffu;
#pragma unroll
      for (int i = 1; i < Q; ++i)
        v[i] = make_float2((ma >> (i - 1)) & 1u ? B.c[q].x : s[i].x, (mb >> (i - 1)) & 1u ? B.c[q].y : s[i].y);
      force_of(v, B.c[q], b.s.G, Fx, Fy);
    } else {
      force_of(s, B.c[q], b.s.G, Fx, Fy);
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = g[i][q];
    uint32_t pair_worst = 0;  // a pair that starts in the box pulls valid columns only
    collide<TAU_ONE, S != LBM_F32>(f, rho[q], jx[q], jy[q], Fx, Fy, b.s, pair_worst);
    if (x + 2 * q < nx) worst = max(worst, pair_worst);
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i][q] = f[i];
  }
  const uint32_t at = (uint32_t)r * b.row_bytes + xb;
  if (full && !edge) {
#pragma unroll
    for (int i = 0; i < Q; ++i) *reinterpret_cast<V*>(b.dst[i] + at) = words<S, P>(g[i]);
  }
  if (edge) {  // a ragged end, or the outer columns with their ghosts
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      T* row = reinterpret_cast<T*>(b.dst[i] + at) - x;
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (x + c < nx) put_cell(row, x + c, nx, Store<S>::enc(c & 1 ? g[i][c / 2].y : g[i][c / 2].x));
    }
  }
  if (out) report_faults(worst, b.flags);
}

// Tiles by storage and relaxation (us per step, swept over rows x CTAs per SM
// x pairs per lane; "staged" is step.cu's march). A small box wants many small
// tiles: one pair per lane, six rows (128^2 2.7 us; two pairs and ten rows
// 4.1). A large one wants few instructions per cell and many loads in flight:
//  - FP32, tau = 1: two pairs, six rows, four CTAs per SM. 8192^2 696
//    (staged 760; eight rows and three CTAs 704, ten and three 736, one pair
//    and ten rows 728), 4096^2 181 (206), 2048^2 49.0 (60), 1024^2 12.9 (15.8).
//  - 16-bit, tau = 1: two pairs, ten rows, three CTAs. 4096^2 122 (staged 136;
//    six rows and four CTAs 132), 2048^2 36.0 (36.6), 1531^2 19.5 (24.9).
//  - tau != 1 keeps a row's populations in registers: six rows, three CTAs.
//    2000 x 1504 BF16 30.0 (staged 34.8), FP32 40.1 (38.7).
template <int S, bool TAU_ONE>
struct Tiles {
  using Small = Tile<1, 6, 3>;
  using Large = Tile<2, TAU_ONE && S != LBM_F32 ? 10 : 6, TAU_ONE && S == LBM_F32 ? 4 : 3>;
  // cells up to which Small is taken (the two cross there), and up to which
  // the tile kernel is (beyond, the staged march is faster)
  static constexpr long long kSmall = !TAU_ONE && S == LBM_F32 ? 1500000 : (S == LBM_F32 ? 500000 : 1200000);
  static constexpr long long most() {
    return TAU_ONE ? (S == LBM_F32 ? 1ll << 40 : 30000000) : (S == LBM_F32 ? kSmall : 1ll << 40);
  }
};

// Planes as the kernel wants them.
__host__ __device__ __forceinline__ void tile_planes(TileBox& b, const void* src, void* dst, long long plane, int E) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    b.src[i] = static_cast<const char*>(src) - kRowPad + (long long)i * plane * E;
    b.dst[i] = static_cast<char*>(dst) - kRowPad + (long long)i * plane * E;
  }
}

template <int S, bool MASKED, bool TAU_ONE, typename G>
__global__ void __launch_bounds__(G::THREADS, G::CTAS) k_step_tile(const TileBox b, int gx) {
  const int t = b.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  const int y0 = t / gx * G::ROWS;
  tile_step<S, MASKED, TAU_ONE, G>(b, t % gx * G::COLS, y0, min(y0 + G::ROWS, b.ny));
}

__device__ __forceinline__ void batch_box(TileBox& b, const BatchInst& in, int parity, int pull_bounce, bool masked, int E) {
  const int c = in.cur ^ parity;
  tile_planes(b, c ? in.pops1 : in.pops0, c ? in.pops0 : in.pops1, in.plane, E);
  b.mask = masked ? reinterpret_cast<const char*>(in.mask) - kMaskPad : nullptr;
  b.flags = in.flags;
  b.nx = in.nx;
  b.ny = in.ny;
  b.row_bytes = (uint32_t)in.pitch * E;
  b.mask_row = (uint32_t)in.mpitch;
  b.pull_bounce = pull_bounce;
  b.s.tau = in.tau;
  b.s.inv_tau = in.inv_tau;
  b.s.G = in.G;
  b.s.rho0 = in.rho0;
  b.s.inv_rho0 = in.inv_rho0;
  b.s.rho_ref = in.rho_ref;
}

// A batch holds boxes of any tau. One with a tau other than 1 in it runs the
// kernels for TAU_ONE = false, where a tau = 1 box still takes the collision it
// takes alone (f = feq; the blend f + (feq - f) rounds feq - f first).
template <int S, bool MASKED, bool TAU_ONE, typename G>
__device__ __forceinline__ void batch_tile(const TileBox& b, int one, int xo, int y0, int y1) {
  if (!TAU_ONE && one) tile_step<S, MASKED, true, G>(b, xo, y0, y1);  // uniform over the CTA
  else tile_step<S, MASKED, TAU_ONE, G>(b, xo, y0, y1);
}

// One item per CTA. The item and its box's descriptor are constant while the
// launches that use them run, so they are read before the wait for the kernel
// before.
template <int S, bool MASKED, bool TAU_ONE, typename G>
__global__ void __launch_bounds__(G::THREADS, G::CTAS)
    k_step_tile_batch(const BatchInst* __restrict__ insts, const BatchItem* __restrict__ items, int parity,
                      int pull_bounce, int reverse) {
  const BatchItem it = items[reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x];
  TileBox b;
  batch_box(b, insts[it.inst], parity, pull_bounce, MASKED, sizeof(typename Store<S>::T));
  batch_tile<S, MASKED, TAU_ONE, G>(b, insts[it.inst].tau_one, it.x0, it.y0, it.y1);
}

// The same with the boxes as a kernel argument: a CTA finds its tile from its
// index and reads no table (two dependent loads: 16 boxes of 11 M cells, FP16,
// 101.8 us per step with them, 94.2 without).
template <int S, bool MASKED, bool TAU_ONE, typename G>
__global__ void __launch_bounds__(G::THREADS, G::CTAS)
    k_step_tile_boxes(const __grid_constant__ BatchBoxes boxes, int parity, int pull_bounce, int reverse) {
  const int t = reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  int lo = 0, hi = boxes.n - 1;
  while (lo < hi) {  // the last box with first <= t
    const int mid = (lo + hi + 1) >> 1;
    if (boxes.first[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  const BatchInst& in = boxes.in[lo];
  const int gx = (in.nx + G::COLS - 1) / G::COLS, k = t - boxes.first[lo], y0 = k / gx * G::ROWS;
  TileBox b;
  batch_box(b, in, parity, pull_bounce, MASKED, sizeof(typename Store<S>::T));
  batch_tile<S, MASKED, TAU_ONE, G>(b, in.tau_one, k % gx * G::COLS, y0, min(y0 + G::ROWS, in.ny));
}

// Every second step takes the tiles from the last to the first while the two
// buffers (`bytes`) are of the order of the L2: its reads then start with what
// the step before wrote last, which is still there. 2000 x 1504 BF16 29.9 ->
// 26.9 us, 2048^2 FP16 35.4 -> 33.6 and FP32 48.7 -> 47.3, 3000^2 FP16 67.0 ->
// 66.1. Below (all of it stays in L2) and above (4096^2 FP16, 600 MB) it gives
// nothing, or costs 1 %.
bool tile_turns(size_t bytes) { return bytes >= 64u << 20 && bytes <= 512u << 20; }

template <int S, bool MASKED, bool TAU_ONE, typename G>
cudaError_t launch_tile_g(const TileBox& b, cudaStream_t s) {
  const int gx = (b.nx + G::COLS - 1) / G::COLS;
  const unsigned grid = (unsigned)gx * (unsigned)((b.ny + G::ROWS - 1) / G::ROWS);
  return launch_chain(k_step_tile<S, MASKED, TAU_ONE, G>, dim3(grid), dim3(G::THREADS), 0, s, b, gx);
}

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_tile_t(const StepParams& p, cudaStream_t s) {
  TileBox b{};
  const int E = storage_bytes(S);
  tile_planes(b, p.src, p.dst, p.plane, E);
  b.mask = p.mask ? reinterpret_cast<const char*>(p.mask) - kMaskPad : nullptr;
  b.flags = p.flags;
  b.nx = p.nx;
  b.ny = p.ny;
  b.row_bytes = (uint32_t)p.pitch * E;
  b.mask_row = (uint32_t)p.mpitch;
  b.pull_bounce = p.pull_bounce;
  b.reverse = p.odd && tile_turns(2 * Q * (size_t)p.plane * E);
  b.s = p;
  using Small = typename Tiles<S, TAU_ONE>::Small;
  using Large = typename Tiles<S, TAU_ONE>::Large;
  if ((long long)p.nx * p.ny <= Tiles<S, TAU_ONE>::kSmall)
    return launch_tile_g<S, MASKED, TAU_ONE, Small>(b, s);
  return launch_tile_g<S, MASKED, TAU_ONE, Large>(b, s);
}

template <int S>
cudaError_t launch_tile_s(const StepParams& p, cudaStream_t s) {
  const bool one = p.tau == 1.0f;
  if (p.mask) return one ? launch_tile_t<S, true, true>(p, s) : launch_tile_t<S, true, false>(p, s);
  return one ? launch_tile_t<S, false, true>(p, s) : launch_tile_t<S, false, false>(p, s);
}

template <int S, bool MASKED, bool TAU_ONE>
cudaError_t launch_tile_batch_t(const TileBatch& t, int reverse, cudaStream_t s) {
  using G = typename Tiles<S, TAU_ONE>::Large;
  if (t.boxes)
    return launch_chain(k_step_tile_boxes<S, MASKED, TAU_ONE, G>, dim3(t.nitems), dim3(G::THREADS), 0, s, *t.boxes,
                        t.parity, t.pull_bounce, reverse);
  return launch_chain(k_step_tile_batch<S, MASKED, TAU_ONE, G>, dim3(t.nitems), dim3(G::THREADS), 0, s, t.insts, t.items,
                      t.parity, t.pull_bounce, reverse);
}

template <int S>
cudaError_t launch_tile_batch_s(const TileBatch& t, int reverse, cudaStream_t s) {
  if (t.masked)
    return t.tau_one ? launch_tile_batch_t<S, true, true>(t, reverse, s)
                     : launch_tile_batch_t<S, true, false>(t, reverse, s);
  return t.tau_one ? launch_tile_batch_t<S, false, true>(t, reverse, s)
                   : launch_tile_batch_t<S, false, false>(t, reverse, s);
}

// f(Tiles<S, TAU_ONE>) for a storage and relaxation known at run time.
template <typename F>
auto by_tiles(int storage, bool tau_one, F f) {
  if (storage == LBM_F32) return tau_one ? f(Tiles<LBM_F32, true>{}) : f(Tiles<LBM_F32, false>{});
  return tau_one ? f(Tiles<LBM_F16_DEV, true>{}) : f(Tiles<LBM_F16_DEV, false>{});
}

}  // namespace

bool tile_fits(int storage, long long plane) {
  // a plane's bytes are addressed with 32 bits
  return plane * storage_bytes(storage) < (1ll << 32) - 4096;
}

void tile_item_size(int storage, bool tau_one, int* cols, int* rows) {
  by_tiles(storage, tau_one, [&](auto t) {
    *cols = decltype(t)::Large::COLS;
    *rows = decltype(t)::Large::ROWS;
    return 0;
  });
}

long long tile_cells(int storage, bool tau_one) {
  return by_tiles(storage, tau_one, [](auto t) { return decltype(t)::most(); });
}

bool step_tiles(int storage, const StepParams& p) {
  return p.force_generic == 0 && (long long)p.nx * p.ny <= tile_cells(storage, p.tau == 1.0f) &&
         tile_fits(storage, p.plane);
}

cudaError_t launch_tile(int storage, const StepParams& p, cudaStream_t s) {
  switch (storage) {
    case LBM_F32: return launch_tile_s<LBM_F32>(p, s);
    case LBM_F16_DEV: return launch_tile_s<LBM_F16_DEV>(p, s);
    case LBM_BF16_DEV: return launch_tile_s<LBM_BF16_DEV>(p, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_tile_batch(int storage, const TileBatch& t, cudaStream_t s) {
  if (t.nitems <= 0) return cudaSuccess;
  int cols, rows;
  tile_item_size(storage, t.tau_one, &cols, &rows);
  const int reverse = t.parity && tile_turns((size_t)t.nitems * cols * rows * 2 * Q * storage_bytes(storage));
  switch (storage) {
    case LBM_F32: return launch_tile_batch_s<LBM_F32>(t, reverse, s);
    case LBM_F16_DEV: return launch_tile_batch_s<LBM_F16_DEV>(t, reverse, s);
    case LBM_BF16_DEV: return launch_tile_batch_s<LBM_BF16_DEV>(t, reverse, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbm
