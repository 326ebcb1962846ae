// Internal declarations shared by the CUDA translation units of liblbm.
// Lattice: D2Q9 (arXiv 1708.01613, Sec. 2.1.1, Eqs. 15-16), directions
// 0:(0,0) 1:(1,0) 2:(0,1) 3:(-1,0) 4:(0,-1) 5:(1,1) 6:(-1,1) 7:(-1,-1) 8:(1,-1).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm.h"

namespace lbm {

constexpr int Q = 9;

__host__ __device__ constexpr int cx(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__host__ __device__ constexpr int cy(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
// Opposite direction: e_opp(i) = -e_i.
__host__ __device__ constexpr int opp(int i) { return i == 0 ? 0 : (i <= 4 ? (i + 1) % 4 + 1 : (i - 3) % 4 + 5); }
__host__ __device__ constexpr double wq(int i) {
  return i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
}
__host__ __device__ constexpr float wqf(int i) {
  return i == 0 ? 4.0f / 9.0f : (i < 5 ? 1.0f / 9.0f : 1.0f / 36.0f);
}

// Device flag slots (int32 each) in the workspace.
enum Flag : int {
  FLAG_NUMERIC = 0,   // NaN/Inf or rho <= 0 seen by the step kernel
  FLAG_TIMEOUT = 1,   // a bounded device loop gave up
  FLAG_OPENED = 2,    // cells opened by the latest rupture test
  FLAG_TILES = 3,     // tiles in the relabel work list
  FLAG_GAS = 4,       // gas points in the growth list
  FLAG_ITEM = 5,      // work-item counter of the dynamically scheduled step (0 between launches)
  FLAG_DONE = 6,      // CTAs of that launch that have finished (0 between launches)
  FLAG_FILM = 7,      // tiles in the list of film tiles
  FLAG_MERGES = 8,    // coalescence events counted by the relabels since the last init
  FLAG_SUMS = 16,     // four FP64 sums of the statistics
  FLAG_HIST = 64,     // 64 histogram counters
  FLAG_COUNT = 128
};

// Population storage: FP32 value, or a 16-bit deviation from w_i rho_ref.
// Decode and encode are explicitly rounded single operations so that every
// kernel (scalar or packed) turns a stored value into the same float.
template <int S>
struct Store;

template <>
struct Store<LBM_F32> {
  using T = float;
  static constexpr int bytes = 4;
  __device__ static __forceinline__ float load(const T* p, size_t i, float) { return __ldcg(p + i); }
  __device__ static __forceinline__ T of(float v, float) { return v; }
  // raw stored value (FP32: the population itself)
  __device__ static __forceinline__ float raw(const T* p, size_t i) { return __ldcg(p + i); }
  __device__ static __forceinline__ float raw_smem(const T* p, int i) { return p[i]; }
  __device__ static __forceinline__ T enc(float v) { return v; }
};

template <>
struct Store<LBM_F16_DEV> {
  using T = __half;
  static constexpr int bytes = 2;
  __device__ static __forceinline__ float load(const T* p, size_t i, float base) {
    return __fadd_rn(base, __half2float(__ldcg(p + i)));
  }
  // the stored word of a full population value
  __device__ static __forceinline__ T of(float v, float base) { return __float2half_rn(__fsub_rn(v, base)); }
  // raw stored value: the deviation g = f - w_i rho_ref
  __device__ static __forceinline__ float raw(const T* p, size_t i) { return __half2float(__ldcg(p + i)); }
  __device__ static __forceinline__ float raw_smem(const T* p, int i) { return __half2float(p[i]); }
  __device__ static __forceinline__ T enc(float g) { return __float2half_rn(g); }
};

template <>
struct Store<LBM_BF16_DEV> {
  using T = __nv_bfloat16;
  static constexpr int bytes = 2;
  __device__ static __forceinline__ float load(const T* p, size_t i, float base) {
    return __fadd_rn(base, __bfloat162float(__ldcg(p + i)));
  }
  __device__ static __forceinline__ T of(float v, float base) { return __float2bfloat16_rn(__fsub_rn(v, base)); }
  __device__ static __forceinline__ float raw(const T* p, size_t i) { return __bfloat162float(__ldcg(p + i)); }
  __device__ static __forceinline__ float raw_smem(const T* p, int i) { return __bfloat162float(p[i]); }
  __device__ static __forceinline__ T enc(float g) { return __float2bfloat16_rn(g); }
};

inline int storage_bytes(int s) { return s == LBM_F32 ? 4 : 2; }

// Population planes in HBM. A plane is ny rows of `pitch` values; a row's
// column 0 starts on a 128-byte boundary, kRowPad bytes into the row, and two
// ghost columns on either side repeat the other end of the periodic row
// (columns -2, -1 hold nx - 2, nx - 1; columns nx, nx + 1 hold 0, 1), so a
// kernel that reads up to two columns beyond its own never wraps, and every
// row of every width takes aligned vector loads and bulk copies. Each kernel
// that writes a slot of the outer two columns writes its ghost too. What lies
// beyond the ghosts is never used, but may be read (vector loads, bulk copies).
// The mask has rows of `mask_pitch` bytes with the same ghosts.
constexpr int kRowPad = 128, kMaskPad = 16;

struct PopShape {
  int pitch;        // values between rows
  long long plane;  // values between planes
};

inline PopShape pop_shape(int storage, int nx, int ny) {
  const int e = storage_bytes(storage);
  // 16 bytes at least after the last column
  const long long row = ((long long)kRowPad + (long long)nx * e + 16 + 127) / 128 * 128;
  PopShape s;
  s.pitch = (int)(row / e);
  s.plane = (long long)s.pitch * ny;
  return s;
}
inline int mask_pitch(int nx) { return (2 * kMaskPad + nx + 15) / 16 * 16; }

// One value in its slot and, in the outer two columns, in its ghost. `row`
// points at column 0.
template <typename T>
__device__ __forceinline__ void put_cell(T* row, int x, int nx, T v) {
  row[x] = v;
  if (x < 2) row[nx + x] = v;
  if (x >= nx - 2) row[x - nx] = v;
}

// The indices at, at + stride, ... below n of one thread of a grid; the last step
// stops at n, because at + stride may be beyond 2^31 for a list of nearly 2^31
// entries.
struct StridedIndex {
  int at, stride, n;
  __host__ __device__ __forceinline__ bool in() const { return at < n; }
  __host__ __device__ __forceinline__ void next() { at = at < n - stride ? at + stride : n; }
};

// Row-chunk height of a launch whose `resident` CTAs draw chunks (gx strips
// by ny rows) from a counter. Chunks of max_rows rows give `items48` chunks;
// if those make at least keep_waves waves (chunks / resident CTAs), the last
// wave's tail is small beside the whole and max_rows stays. Otherwise the
// height is the one that fills a whole number of waves: the fewest that
// max_rows allows, but at least min_waves once the chunks overflow one wave
// (more, shorter chunks let the fast CTAs take more). A last wave that
// fills only part of the GPU leaves the rest idle for a whole chunk time.
inline int dyn_chunk_rows(long long gx, long long ny, long long resident, int max_rows, int keep_waves,
                          int min_waves) {
  if (gx < 1 || ny < 1 || resident < 1 || max_rows < 1) return 1;
  const long long items = gx * ((ny + max_rows - 1) / max_rows);
  if (items >= (long long)keep_waves * resident) return max_rows;
  long long waves = (items + resident - 1) / resident;
  if (items > resident && waves < min_waves) waves = min_waves;
  long long per = waves * resident / gx;  // chunks per strip
  if (per < 1) per = 1;
  const long long rows = (ny + per - 1) / per;
  return (int)(rows < 1 ? 1 : (rows > max_rows ? max_rows : rows));
}

// Arguments of the fused step kernel.
struct StepParams {
  const void* src;       // populations after collision of the previous step
  void* dst;             // populations after collision of this step
  const uint8_t* mask;   // blocked-edge mask (nullptr: plain Shan-Chen)
  int* flags;            // device flag slots
  int nx, ny;
  int pitch, mpitch;     // row strides: population values, mask bytes (src, dst and mask point at column 0)
  long long plane;       // plane stride
  int rows_per_chunk;    // rows marched by one CTA
  int odd;               // tile kernel: every second step (tiles in reverse)
  int pull_bounce;       // tile kernel: src holds populations that have not bounced back yet
  int force_generic;     // kernel variant: 0 automatic, 1 plain loads, 2 one-cell staged, 3 two-cell staged,
                         // 4 two-cell staged with dynamically scheduled row chunks
  float tau, inv_tau, G, rho0, inv_rho0;
  float rho_ref;         // reference density of 16-bit deviations
};

// Two-component step (step2.cu): 18 FP32 planes per buffer, melt then gas.
struct Step2Params {
  const void* src;
  void* dst;
  const uint8_t* mask;  // nullptr: no barrier
  int* flags;
  int nx, ny;
  int pitch, mpitch;    // as in StepParams
  long long plane;
  int rows_per_chunk;
  float tau_m, tau_g, inv_tau_m, inv_tau_g;
  float G_mm, G_mg, G_gg, rho0, inv_rho0;
};
cudaError_t launch_step2(const Step2Params& p, cudaStream_t s);
// Melt/gas densities, mixture velocity (j + F/2)/rho and pressure of the
// state in p.src; any output may be nullptr.
cudaError_t launch_fields2(const Step2Params& p, float* rho_m, float* rho_g, float* ux, float* uy, float* pr,
                           cudaStream_t s);

// One box of a batched launch (device array).
struct BatchInst {
  void* pops0;
  void* pops1;
  const uint8_t* mask;  // nullptr: plain Shan-Chen
  int* flags;
  int nx, ny;
  int pitch, mpitch;
  long long plane;
  float tau, inv_tau, G, rho0, inv_rho0, rho_ref;
  int cur;              // buffer holding the state when parity == 0
  int tau_one;          // tau == 1 (not asked of tau in a kernel: the compiler then
                        // folds tau F + j into an add and contracts it with F's product)
};

// One work item of a batched launch: columns x0 .. x0+width, rows y0 .. y1.
struct BatchItem {
  int inst, x0, width, y0, y1;
};

// Streaming multiprocessors of the current device (queried once per device;
// 152 on a GB300 if the query fails). Grids that are sized per SM use it.
int device_sm_count();

// Launch of the fused step (step.cu). Returns a cudaError_t.
cudaError_t launch_step(int storage, const StepParams& p, cudaStream_t s);
// Whether launch_step takes the tile kernel (tile.cu) for this box (automatic
// variant): then the bounce-back of the step before may be left to the pull
// (pull_bounce).
// Many steps in one launch, src to dst, for a box that fits a cluster's shared
// memory (resident.cu); src has bounced back already, dst has not.
bool steps_resident(const StepParams& p, long long steps);
cudaError_t launch_resident(int storage, const StepParams& p, int steps, cudaStream_t s);
bool step_tiles(int storage, const StepParams& p);
cudaError_t launch_tile(int storage, const StepParams& p, cudaStream_t s);
// The same over many boxes, items of at most cols x rows cells (x0 a multiple
// of cols). Boxes need tile_fits.
bool tile_fits(int storage, long long plane);
void tile_item_size(int storage, bool tau_one, int* cols, int* rows);
// Cells up to which the tile kernel beats the staged ones.
long long tile_cells(int storage, bool tau_one);
// The boxes of a batch as a kernel argument, with the tiles of the boxes
// before each (rows of tiles, top to bottom).
struct BatchBoxes {
  static constexpr int kMost = 40;  // 4 KB; larger batches read the tables (32 KB of arguments would go)
  int n;
  int first[kMost];
  BatchInst in[kMost];
};
struct TileBatch {
  bool masked, tau_one, pull_bounce;
  int parity, nitems;
  const BatchBoxes* boxes;  // host; nullptr: the tables below (device)
  const BatchInst* insts;
  const BatchItem* items;
};
cudaError_t launch_tile_batch(int storage, const TileBatch& t, cudaStream_t s);
// Launch geometry the fused step uses for a box (for tests/benchmarks).
void step_geometry(int nx, int ny, int* grid_x, int* grid_y, int* rows_per_chunk, int* block);
// Widths the staged variants accept (lbm_set_step_variant): 2 takes widths
// that are multiples of 16 and of at least one strip and its halo, 3 and 4
// any width of 16 or more.
bool step_tma_allowed(int storage, int nx);
bool step_tma2_allowed(int nx);
// Batched fused step (two-cell staged march over a list of work items of
// many boxes); one persistent grid drawing items from counters[parity] and
// zeroing counters[parity ^ 1]. Both counters must be zero before the
// first launch and consecutive launches must alternate parity.
cudaError_t launch_step_batch(int storage, bool masked, bool tau_one, const BatchInst* insts, const BatchItem* items,
                              int nitems, int* counters, int parity, cudaStream_t s);
// CTAs of the batched kernel that fit the GPU at once.
int batch_resident_ctas(int storage, bool masked, bool tau_one);

// Barrier / field / reduction kernels (barrier.cu).
struct FieldParams {
  const void* pops;    // column 0 of the current populations (post-collision of the last step)
  int storage;
  int nx, ny;
  int pitch, mpitch;
  long long plane;
  long long N;         // cells
  float G, rho0, inv_rho0, tau;
  float wref[Q];
};

cudaError_t launch_density(const FieldParams& fp, float* rho, cudaStream_t s);
// Relabel of a box that does not use the tiled pipeline: gas labels
// (4-connected, smallest index) of rho into label. Each new gas cell first
// parks its label of the previous relabel in keep (the owner array) and the
// coalescence events are added to flags[FLAG_MERGES].
cudaError_t launch_labels(const FieldParams& fp, const float* rho, float threshold, int32_t* label,
                          int* flags, cudaStream_t s, int32_t* keep);
cudaError_t launch_owner(int nx, int ny, int R, const int32_t* label, int32_t* owner, cudaStream_t s);
cudaError_t launch_rupture(int nx, int ny, float G, float rho0, float eps, const float* rho,
                           const int32_t* owner, int8_t* sgn, uint8_t* open, int* flags,
                           cudaStream_t s);
cudaError_t launch_mask(int nx, int ny, int mpitch, const int32_t* owner, const uint8_t* open, uint8_t* mask,
                        cudaStream_t s);
// Diagnostics (fields.cu). Any of rho, u and p in one pass (nullptr: not asked for).
struct FieldOuts {
  float *rho, *ux, *uy, *p;
};
cudaError_t launch_fields(const FieldParams& fp, const uint8_t* mask, const FieldOuts& out, cudaStream_t s);
// The mask in dense rows.
cudaError_t launch_mask_out(const FieldParams& fp, const uint8_t* mask, uint8_t* out, cudaStream_t s);
// Planes plane0 .. plane0 + planes of the incoming state, back to back.
cudaError_t launch_pops_out(const FieldParams& fp, int plane0, int planes, float* out, cudaStream_t s);
// Scratch the three label passes need beside their arrays (8-byte aligned).
size_t diag_scratch_bytes(int nx, int ny);
// Gas labels of the current state.
cudaError_t launch_diag_labels(const FieldParams& fp, float threshold, int32_t* label, void* scratch, int* flags,
                               cudaStream_t s);
// Labels, areas (at their roots), then [0] bubbles [1] gas cells [2] sum of
// equivalent diameters [3] mass into out_dev and the histogram into hist.
cudaError_t launch_diag_stats(const FieldParams& fp, float threshold, int32_t* label, int32_t* area, void* scratch,
                              int* flags, double* partials, int nparts, double* out_dev, int* hist, int nbins,
                              double dmin, double dmax, cudaStream_t s);
// Labels, areas, and the (root, area) pairs in any order with their count.
cudaError_t launch_diag_areas(const FieldParams& fp, float threshold, int32_t* label, int32_t* area, int32_t* list,
                              int* count, void* scratch, int* flags, cudaStream_t s);
// Initialisation of the buffer fp.pops: rest equilibrium at rho (nine planes),
// or the incoming plane `plane` from f (dense rows).
cudaError_t launch_init_from_rho(const FieldParams& fp, const double* rho, cudaStream_t s);
cudaError_t launch_load_plane(const FieldParams& fp, const float* f, int plane, cudaStream_t s);
cudaError_t launch_bubbles_rho(const lbm_bubble* d_bubbles, int n, double rho_l, double rho_g,
                               double width, int nx, int ny, double* rho, cudaStream_t s);
cudaError_t launch_mass(const FieldParams& fp, double* partials, int nparts, double* out_dev,
                        cudaStream_t s);
constexpr int kMaxHistBins = 64;
// Tiled barrier pipeline (relabel.cu). One launch per phase serves one box or
// any number of boxes.
bool relabel_tiled_ok(int nx, int ny, int R);
int relabel_tile_count(int nx, int ny);
constexpr int kRelabelTileX = 32, kRelabelTileY = 8;  // tile of the pipeline
constexpr int kRelabelLaunches = 4;
// Launches of an untiled relabel: density, label init, union, flatten,
// coalescence count, owner, rupture, mask.
constexpr int kUntiledLaunches = 8;

// A box as the pipeline sees it (a kernel argument, or device memory).
// Populations are read from pops[cur ^ parity], parity being the launch
// argument.
struct RelabelBox {
  const void* pops[2];  // column 0, like mask
  int32_t* label;
  int32_t* old;  // scratch: labels of the previous relabel at gas cells
  int32_t* owner;
  int8_t* sgn;
  uint8_t* open;
  uint8_t* mask;
  uint8_t* tile_gas;
  uint8_t* tile_active;
  uint8_t* tile_prev;
  int* tile_list;     // tiles to visit
  int* film_list;     // tiles of it where owners meet (mask, bounce-back)
  int32_t* gas_list;  // gas cells for the growth source (nullptr: no source)
  int* flags;
  int nx, ny, ntx, nty, R, cur;
  int pitch, mpitch;
  long long plane;
  float threshold, G, rho0, eps;
  float G_mg, G_gg;  // two components: melt-gas and gas-gas couplings
  float wref[Q];
};

// Box `box` in a launch's entry list, with the CTAs of the entries before it
// in each kind of phase (per-tile, tile-scan, tile-list, film-list). An entry
// list of m boxes has m + 1 entries: the last holds the totals.
struct RelabelEntry {
  int box, off_tiles, off_scan, off_list, off_film;
};

// CTAs a box takes in each kind of phase.
RelabelEntry relabel_entry_sizes(int nx, int ny);
// The phases over a box (state: pops[cur]), or over the first m entries;
// totals = entries[m]. two: two components (FP32).
cudaError_t launch_relabel_lone(int storage, const RelabelBox& box, bool two, cudaStream_t s);
cudaError_t launch_relabel_boxes(int storage, const RelabelBox* boxes, const RelabelEntry* entries, int m,
                                 const RelabelEntry& totals, int parity, cudaStream_t s);

// Halfway bounce-back across the blocked edges of the mask (the barrier of
// Sec. 2.1.5), run on the buffer a step has just written (after the growth
// source, if any): the two slots of each blocked edge trade values, so the
// next step's pull returns every population that would cross the wall to
// its own cell in the opposite direction. `two`: 18 planes (two lattices).
// launch_bounce scans every cell; the others visit the tiles that the latest
// tiled relabel found holding a blocked edge, on buffer pops[cur ^ q] (q = 0
// for a lone box; ctas = the entries' film-CTA total).
cudaError_t launch_bounce(const FieldParams& fp, bool two, void* pops, const uint8_t* mask, cudaStream_t s);
cudaError_t launch_bounce_lone(int storage, const RelabelBox& box, bool two, cudaStream_t s);
cudaError_t launch_bounce_boxes(int storage, const RelabelBox* boxes, const RelabelEntry* entries, int m, int ctas,
                                int q, cudaStream_t s);
int mass_partials_needed();

// Nucleation and growth (growth.cu). The gas census appends every cell with
// rho < threshold to `list` (order irrelevant) and sets *count (the tiled
// relabel takes its census itself). The growth
// kernel adds w_i drho to the post-collision populations of the listed
// cells, drho = min(rate, budget - released) / count, reading the released
// total from released[parity] and writing the new total to
// released[parity ^ 1] (consecutive steps alternate parity).
cudaError_t launch_gas_census(const float* rho, long long N, float threshold, int32_t* list, int* count,
                              cudaStream_t s);
cudaError_t launch_growth(const FieldParams& fp, void* pops, const int32_t* list, const int* count, double rate,
                          double budget, double* released, int parity, cudaStream_t s);
cudaError_t launch_nucleate(const FieldParams& fp, void* pops, const lbm_bubble* nuclei, int n, double rho_g,
                            cudaStream_t s);

}  // namespace lbm
