// internal.h -- declarations shared by the C-ABI layer (api.cpp) and the
// CUDA translation units of the stencil library.  Not installed, not part of
// the ABI; nothing here is visible outside libstencil_gb300.so.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <vector>

namespace gbst {

// Largest tap set: a radius-2 box in 3D.
constexpr int kMaxTaps = 125;

// Stencil classes the plan recognises from the non-zero pattern of the
// weights.  The class fixes the compile-time tap list of the kernels.
enum class Shape : int {
  kStar = 0,  // taps only on the axes through the centre (2*d*r + 1 taps)
  kBox = 1,   // every offset in [-r, r]^d ((2r+1)^d taps)
};

// Boundary rule (same values as stencil_boundary).
enum Boundary : int { kDirichlet = 0, kPeriodic = 1 };

// Kernel variants selectable through stencil_set_tuning.  Ids are ABI-stable.
enum Variant : int {
  kVariantAuto = 0,
  kVariantDirect = 1,     // one cell per thread per plane, taps from L1
  kVariantStream = 2,     // slowest-axis streaming through a TMA-fed SMEM ring
  kVariantTemporal = 3,   // Tb fused steps per HBM round trip (overlapped tiles)
  kVariantPersistent = 4, // one launch for all steps: barrier per step (Tb 1) or tile flags (Tb > 1)
  kVariantExchange = 5,   // Tb fused steps per launch, 3D, no recompute: tiles hand over levels through L2
  kVariantCount = 6
};

// Tap list for a launch, passed by value (kernel parameter space lives in the
// constant bank, so the weights are constant-bank operands of the FMAs).
template <int NT>
struct TapList {
  double w[NT];
  int8_t dz[NT], dy[NT], dx[NT];
};

// Grid geometry padded to three axes (leading axes of length 1).
struct Geom {
  int nz, ny, nx;
  int64_t cells() const { return (int64_t)nz * ny * nx; }
};

// Host-side description of the taps (any count up to kMaxTaps).
struct HostTaps {
  int n = 0;
  double w[kMaxTaps];
  int8_t dz[kMaxTaps], dy[kMaxTaps], dx[kMaxTaps];
};

// The weights split for the integer form of the weighted sum (wide.cuh); n = 0
// when that form does not cover them.
constexpr int kWideMaxTaps = 27;
template <int N>
struct WideTapsOf {
  int n = 0;
  int hi[N], lo[N];                        // limbs of the significand: hi * 2^26 + lo
  int hi2[N];                              // 2 * hi
  int ex[N];                               // exponent below the largest weight's (<= 0)
  int heat;                                // one weight at the centre tap (n / 2), one at all others
  int bias;                                // exponent of the result: E - bias above R's
  int e_min;                               // E in [e_min, e_min + e_span], else the FMA chain
  unsigned int e_span;
  int equal;                               // a box whose weights are all equal
};
using WideTaps = WideTapsOf<kWideMaxTaps>;

// Launchers implemented in the .cu files.  Each returns a cudaError_t from
// the launch (cudaSuccess when nothing failed) and enqueues on `stream`.
// wdev: the plan's weights on the device (taps.n weights in tap order, then
// zero and one slots; see taps.cuh).  wide: the same weights split for the
// integer form of the sum; n = 0 selects the FMA chain.
cudaError_t launch_direct(int ndim, int radius, Shape shape, int boundary, const Geom& g,
                          const HostTaps& taps, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                          cudaStream_t stream);

// FP32 twin of the direct sweep (accuracy studies only; up to 27 taps).
cudaError_t launch_direct_f32(int ndim, int radius, int boundary, const Geom& g, const HostTaps& taps,
                              const float* src, float* dst, cudaStream_t stream);

// 3D radius-1 streaming sweep (TMA-fed shared-memory plane ring) over tiles
// of 64 columns by tile_y rows (8, 16 or 32; 0 = the default: 32 for the
// star, 16 for the box).  Eligible when nx is even, both buffers are 16-byte
// aligned and, for periodic grids, nx % 64 == 0 and ny % tile_y == 0.
bool stream3d_eligible(int ndim, int radius, Shape shape, int boundary, const Geom& g, const void* a,
                       const void* b, int tile_y = 0);
// The shape part of that rule (no buffers, no driver query).
bool stream3d_shape_ok(int ndim, int radius, Shape shape, int boundary, const Geom& g, int tile_y = 0);
// The tile height a tile_y request resolves to (-1: not a supported height).
int stream3d_tile_y(Shape shape, int tile_y);
// wait_ns bounds every mbarrier wait (kSpinLimitNs in normal runs); skip_plane
// >= 0 is the self-test's starved plane (the producer posts no copy for it).
cudaError_t launch_stream3d(Shape shape, int boundary, const Geom& g, const HostTaps& taps,
                            const double* wdev, const double* src, double* dst, int* status,
                            int sms, cudaStream_t stream, unsigned long long wait_ns = 2000000000ull,
                            long long skip_plane = -1, int tile_y = 0);

// 3D radius-1 sweep with the weighted sum in the integer form (wide.n != 0):
// tiles of 64 columns by 16 rows (tile_y = 8: 8, and with tma 32: 32).  tma: the grid is one that
// stream3d_eligible takes; false: any shape, alignment and boundary.  chained: the
// stream's last launch is a step of the same run by this kernel or launch_wide2d's
// (launch_step in widestream.cuh).
cudaError_t launch_wide3d(Shape shape, int boundary, const Geom& g, const WideTaps& wide, const double* wdev,
                          const double* src, double* dst, int* status, int sms, cudaStream_t stream, int tile_y,
                          bool tma, bool chained = false);

// 2D radius-1 or radius-2 streaming sweep (TMA-fed ring of 16-row blocks).  Same
// eligibility rules with ny % 16 == 0 for periodic grids.  `equal` selects
// the shared-partial-sum form for a box whose weights are all equal.
bool stream2d_eligible(int ndim, int radius, int boundary, const Geom& g, const void* a,
                       const void* b);
bool stream2d_shape_ok(int ndim, int radius, int boundary, const Geom& g);
bool taps_all_equal(const HostTaps& t);
cudaError_t launch_stream2d(Shape shape, int radius, int boundary, bool equal, const Geom& g,
                            const HostTaps& taps, const double* wdev, const double* src, double* dst,
                            int* status, int sms, cudaStream_t stream);

// 2D sweep (radius 1 or 2, star or box) with the weighted sum in the integer
// form (wide.n != 0), tiles of 64 columns by 16 rows.  tma: the grid is one that
// stream2d_eligible takes; false: any shape, alignment and boundary.  chained: as
// in launch_wide3d.
cudaError_t launch_wide2d(Shape shape, int radius, int boundary, const Geom& g, const WideTaps& wide,
                          const double* wdev, const double* src, double* dst, int* status, int sms,
                          cudaStream_t stream, bool tma, bool chained = false);

// Self-tests of those kernels' bounded waits (a star with wide.heat on a periodic grid that TMA takes):
// the producers leave copies out, so that waits run out after wait_ns.
cudaError_t launch_wide3d_starved(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                                  int* status, int sms, cudaStream_t stream, unsigned long long wait_ns);
cudaError_t launch_wide2d_starved(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                                  int* status, int sms, cudaStream_t stream, unsigned long long wait_ns);

// 1D sweep (radius 1 or 2) with the weighted sum in the integer form (wide.n != 0),
// `steps` fused steps (at most kWide1dSteps).
constexpr int kWide1dSteps = 8;
cudaError_t launch_wide1d(int radius, int boundary, int steps, const Geom& g, const WideTapsOf<5>& wide,
                          const double* wdev, const double* src, double* dst, int sms, cudaStream_t stream);

// All steps of a small 3D 7-point grid in one cooperative launch, one brick per SM (wide.n == 7).
struct Steps3dLaunch {
  double* a;        // the caller's grid
  double* b;        // partner buffer
  int nz, ny, nx;
  int periodic;
  int T;
  int bricks[3];    // along x, y, z
  const double* wdev;
  WideTapsOf<7> wide;
  unsigned int* progress;  // kFlagWords words for each brick, zero before the launch
  int* status;
  long long spin_limit;    // ns
  int mute = -1;           // self-test: the brick that does not publish its steps
};
// Cuts a grid into at most `sms` bricks; returns their cells per thread (launch_steps3d's
// z), 0 when the grid is too large.
int steps3d_cut(const Geom& g, int sms, int (&bricks)[3]);
cudaError_t launch_steps3d(const Steps3dLaunch& L, int z, cudaStream_t stream);

// Temporal blocking: Tb fused steps per launch (2D and 3D: radius 1, any
// shape and boundary; 1D: radius 1 or 2; Tb in {2, 4, 8}).
bool temporal_supported(int ndim, int radius, int Tb);
// equal: a 2D box whose weights are all equal takes the shared-partial-sum
// form (within rounding of the tap-order kernels, not bitwise equal).
cudaError_t launch_temporal(int ndim, int radius, Shape shape, int boundary, int Tb, const Geom& g,
                            const WideTaps& wide, const double* wdev, const double* src, double* dst, int sms,
                            cudaStream_t stream, bool equal = false);

// Temporal blocking without recomputation (3D radius 1, star or box, Tb >= 2):
// one co-resident CTA per 64-column tile of a band of rows of the (y, x)
// plane, intermediate time levels handed between tiles through a ring of
// Tb-1 x K band planes (K = 9 / 10, 7 / 8 and 5 / 6 for the star / box at Tb = 2, 4 and 8).  A
// plane taller than the co-resident tiles cover (32 rows each) is cut into
// bands, one launch each, every band with a margin of Tb-1 rows toward each
// neighbouring band: the rows its last stage may get wrong at an edge whose
// neighbour rows it does not compute.
struct ExchangeBand {
  int y_base;          // grid row of the band's first row (periodic: may be negative)
  int rows;            // rows of the band, margins included
  int own_lo, own_hi;  // grid rows the band writes to the output
  int tiles_y;         // tile rows (tiles of at most 32 rows)
  bool whole;          // the band is the whole plane (periodic rows wrap within it)
};
struct ExchangeLaunch {
  Geom g;
  const double* src;       // time t (16-byte aligned)
  double* dst;             // time t + Tb (16-byte aligned, not src)
  double* ring;            // exchange_ring_cells(g, Tb, band.rows) doubles
  unsigned int* counters;  // exchange_counter_words(tiles) words, zero before the launch
  int* status;
  const double* wdev;
  WideTaps wide;
  int Tb;
  int tiles_x;             // exchange_tiles_x(g): ceil(nx / 64)
  ExchangeBand band;
  long long spin_limit;    // ns
};
// True when the kernel takes the shape: 3D radius 1, nx even (a multiple of
// 64 on a periodic grid), at most `sms` tile columns of 64.
bool exchange_fits(int ndim, int radius, const Geom& g, bool periodic, int sms);
int exchange_tiles_x(const Geom& g);
// The bands of a shape that fits, for `sms` co-resident CTAs and Tb steps.
std::vector<ExchangeBand> exchange_bands(const Geom& g, bool periodic, int Tb, int sms);
size_t exchange_ring_cells(const Geom& g, int Tb, int band_rows);
int exchange_counter_words(int tiles);
cudaError_t launch_exchange(Shape shape, int boundary, const ExchangeLaunch& L, cudaStream_t stream);

// Variable-coefficient diffusion: coefficient preparation, one forward step,
// one fused adjoint step, gradient finalisation and the loss reduction.
struct VarcoefBufs {
  // per-cell coefficients: centre c0 = 1 - sum of face coefficients, and the
  // coefficient of the +x, +y, +z face of each cell (dt * face diffusivity)
  double* c0;
  double* cx;
  double* cy;
  double* cz;
};
cudaError_t launch_varcoef_prepare(int ndim, int boundary, const Geom& g, const double* kappa,
                                   double dt, VarcoefBufs b, cudaStream_t stream);
cudaError_t launch_varcoef_step(int ndim, int boundary, const Geom& g, VarcoefBufs b,
                                const double* src, double* dst, const double* zero,
                                cudaStream_t stream);
// lam_out = A^T lam_in, and for every +face f=(i,n): G_f += (u_n - u_i)(lam_i - lam_n)
// (lam = lam_in = lambda^{t+1}, u = u^t); ghost faces: Gg_i -= k_i * u_i * lam_i
// where k_i is the number of ghost faces of cell i (Dirichlet only).
cudaError_t launch_adjoint_step(int ndim, int boundary, const Geom& g, VarcoefBufs b,
                                const double* lam_in, const double* u, double* lam_out,
                                double* gx, double* gy, double* gz, double* gg, const double* zero,
                                cudaStream_t stream);
// grad_kappa_i = (dt/2) * sum_{faces f of i} G_f + dt * Gg_i
cudaError_t launch_adjoint_finalize(int ndim, int boundary, const Geom& g, double dt,
                                    const double* gx, const double* gy, const double* gz,
                                    const double* gg, double* grad_kappa, cudaStream_t stream);
// lam = u - target, and block partial sums of 0.5*(u - target)^2 into partials
// (nblocks entries); then a single-block pass sums the partials in order.
cudaError_t launch_loss_residual(int64_t n, const double* u, const double* target, double* lam,
                                 double* partials, int nblocks, double* loss_out,
                                 cudaStream_t stream);

// Batched persistent sweep over many 2D heat grids.
struct BatchTile {
  int item;     // index into the item table
  int k0;       // first cell of the tile (row-major index within the item)
  int n;        // cells in the tile (batched_tile_cells(), fewer at an item's end)
};
struct BatchItemDev {
  double* a;     // the caller's grid (time level parity 0)
  double* b;     // library-owned partner buffer (parity 1)
  int ny, nx;
  int T;
  // 5-point star weights in lexicographic tap order: north (y-1), west (x-1),
  // centre, east (x+1), south (y+1); Eq. 3 gives alpha, alpha, 1-4 alpha, alpha, alpha
  double w[5];
  double zero[2];  // 0.0: the addends of the first FMA of each row's chain
  WideTapsOf<5> wide;  // the weights split for the integer form (n = 0: the FMA chain)
};
struct BatchLaunch {
  const BatchItemDev* items;
  const BatchTile* tiles;
  int ntiles;
  int max_T;
  int boundary;
  unsigned int* barrier;  // two words: arrival count, generation
  int* status;            // 0 ok, else a stencil_status
  long long spin_limit;   // bounded waits: wall-time limit in ns
  int barrier_blocks;     // arrivals a device-wide barrier waits for (0: the grid size)
  int wide = 0;           // some item takes the integer form (wide.n != 0)
};
// The same sweep over tiles of 64 x 16 cells with the weighted sum in the integer
// form (every item's wide.n != 0): widesteps.cu.
struct WideStepItem {
  double* a;      // the caller's grid (time level parity 0)
  double* b;      // library-owned partner buffer (parity 1)
  int ny, nx, T;
  int tiles_y;        // tiles per column of tiles
  int tile0, ntiles;  // the item's tiles in the launch's list
  int vec;            // rows of both buffers start on 16 bytes
  double w[5];
  WideTapsOf<5> wide;
};
struct WideStepsLaunch {
  const WideStepItem* items = nullptr;  // device, largest T first; nullptr: the one item below
  WideStepItem one;
  int nitems;
  int max_T;
  int any_odd;            // some item's T is odd
  int heat;               // every item's wide.heat
  unsigned int* progress;  // kProgressWords words, zero before the launch: steps done by every CTA
  int* status;
  long long spin_limit;    // ns
  int mute = -1;           // self-test: the CTA that does not publish its steps
};
constexpr int kWideStepCtas = 512;  // most CTAs of a launch
constexpr int kProgressWords = 16 * kWideStepCtas;  // half a line for each
void wide_step_item(WideStepItem& d, const BatchItemDev& it, int tile0);
// Whether a grid fills its tiles of 64 x 16 cells well enough, and the SMs with them
// (one step per device-wide barrier by cells instead: 256^2 17 against 13 GStencil/s,
// 512^2 43.6 against 46).
inline bool wide_steps_worth(int64_t ny, int64_t nx) {
  const int64_t tiles = ((ny + 15) / 16) * ((nx + 63) / 64);
  return tiles >= 200 && 10 * ny * nx >= 8 * tiles * 1024;
}
cudaError_t launch_wide_steps(const WideStepsLaunch& L, int tiles, int boundary, int sms, cudaStream_t stream);

// Words from one flag (progress word) that other CTAs poll to the next: a line.
constexpr int kFlagWords = 32;

// Threads per block of the batched kernel; a tile is cpt * kBatchThreads
// consecutive cells, so the smallest tile (cpt = 1) holds kBatchThreads cells.
constexpr int kBatchThreads = 256;
constexpr int kBatchMinTileCells = kBatchThreads;
// cpt: cells per thread of the kernel (1, 2 or 4); a tile holds cpt * 256 cells.
cudaError_t launch_batched(const BatchLaunch& L, int grid_blocks, int cpt, cudaStream_t stream);
int batched_block_size();
int batched_default_cpt();
int batched_tile_cells(int cpt);
int batched_blocks_per_sm(int cpt, bool wide);

// Persistent temporal blocking for one small 2D grid (radius 1, star or box):
// Tb in {2, 4, 8} steps per exchange, tiles synchronised by per-tile flags.
struct PersistTbLaunch {
  double* a;             // the caller's grid
  double* b;             // partner buffer
  int ny, nx;
  long long T;
  const double* wdev;    // weights, then the zero and one slots
  WideTapsOf<9> wide;    // the weights split for the integer form (n = 0: the FMA chain)
  int tiles_y, tiles_x;  // near-equal cut of the grid (from persist_tiling)
  int reach_y, reach_x;  // tiles a Tb-cell halo can reach on each side
  unsigned int* flags;   // tiles_y * tiles_x * kFlagWords words, zero before the launch
  int* status;
  long long spin_limit;  // ns
};
// Batched temporal blocking: many 2D 5-point heat grids advanced Tb steps in
// shared memory per exchange, one launch, tiles synchronised by per-tile
// flags (each item cut into tiles of at most 16 x 32 cells).
struct BatchTbItemDev {
  double* a;              // the caller's grid
  double* b;              // partner buffer
  int ny, nx, T;
  int tiles_y, tiles_x;   // near-equal cut of the item
  int reach_y, reach_x;   // tiles a Tb-cell halo can reach on each side
  int tile_base;          // the item's first tile (its flag words start there)
  double w[5];            // north, west, centre, east, south (lexicographic taps)
  double zero;            // 0.0, the addend of each chain's first FMA
  WideTapsOf<5> wide;     // the weights split for the integer form (n = 0: the FMA chain)
};
struct BatchTbTile {
  int item, ty, tx;       // tile (ty, tx) of item `item`
};
struct BatchTbLaunch {
  const BatchTbItemDev* items;
  const BatchTbTile* tiles;
  int ntiles;
  int max_blocks;         // the largest ceil(T / Tb) over the items
  unsigned int* flags;    // ntiles * kFlagWords words, zero before the launch
  int* status;
  long long spin_limit;   // ns
};
cudaError_t launch_batched_tb(const BatchTbLaunch& L, int grid_blocks, int Tb, int boundary,
                              cudaStream_t stream);
int batched_tb_blocks_per_sm(int Tb, int boundary);
// Largest tile of the batched temporal kernel.
constexpr int kBatchTbTileH = 16, kBatchTbTileW = 32;

// Picks the cut of an ny x nx grid into tiles of at most 16 x 32 cells that
// minimises the FP64 work of the busiest SM for Tb steps per block, and the
// reach of a Tb-cell halo in tiles.
void persist_tiling(int ny, int nx, int Tb, int sms, int* tiles_y, int* tiles_x, int* reach_y, int* reach_x);
cudaError_t launch_persist_tb(Shape shape, int boundary, int Tb, const PersistTbLaunch& L, int sms,
                              cudaStream_t stream);

// FP64 peak microbenchmark: `iters` rounds of 8 independent DFMA chains in
// blocks x 256 threads; out receives one double per thread.
cudaError_t launch_fp64_peak(int blocks, int iters, double* out, cudaStream_t stream);

// Wall-time limit of every bounded device-side wait the host configures
// (barriers of the persistent kernels): 2 s.
constexpr long long kSpinLimitNs = 2000000000LL;

// Launch accounting (every kernel launch of the library adds one).
extern std::atomic<int64_t> g_launches;

// Ordinal of the current device, clamped to [0, kMaxDeviceOrdinals).
constexpr int kMaxDeviceOrdinals = 64;
int device_ordinal();

// Per-device cache of a kernel's launch property (occupancy after its
// attributes are set): `compute` runs on the first call for each device and
// must be idempotent (concurrent first calls may both run it).  `cache` is a
// zero-initialised static array owned by the call site.
template <typename F>
int cached_per_device(std::atomic<int> (&cache)[kMaxDeviceOrdinals], F&& compute) {
  const int dev = device_ordinal();
  int v = cache[dev].load(std::memory_order_acquire);
  if (v == 0) {
    v = compute() + 1;
    cache[dev].store(v, std::memory_order_release);
  }
  return v - 1;
}

}  // namespace gbst
