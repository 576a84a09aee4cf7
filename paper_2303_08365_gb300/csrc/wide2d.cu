// wide2d.cu -- 2D sweep (radius 1 or 2, star or box) with the weighted sum in the
// integer form (wide.cuh).
//
// One step of u'(x) = sum_o w_o u~(x+o) (paper Sec. 2.1, Listing 1).  The grid is
// cut into tiles of 64 columns by 16 rows, taken down each column of tiles.  As in
// wide3d.cu a tile's values are unpacked once, into shared memory:
//   - the raw tile (its columns, RAD rows more above and below) arrives up to
//     three tiles ahead: by TMA where the grid allows it (out-of-range parts read
//     zeros, the Dirichlet ghosts), else row by row by bulk copies, which take any
//     size, alignment and wrap;
//   - iteration g: every consumer warp unpacks its own two rows of tile g into ring
//     slot g % 3 (the producer warp the rows and columns around the tile), arrives
//     on conv[g % 3], and computes its rows of tile g-1, which is complete
//     (waited for before tile g is unpacked; every warp has then also finished
//     tile g-3, whose slot tile g takes).
// The rows between two tiles are unpacked twice (18 or 20 rows for 16).
//
// Measured at 8192^2, periodic, general weights (FMA chain before): 25-point box
// 52 GStencil/s (23.6), radius-2 star 113 (67).  Boxes whose weights are all equal
// share alignments and partial sums among a lane's four cells (WideSum), with the bits that each
// cell has alone: 9-point box at 16384^2 210 GStencil/s (140 with shared sums on the FP64 pipe; 225
// with values cut to 58 bits at the four cells' common exponent, which made the bits depend on
// where a tile begins), 25-point box at 8192^2 147 (24; 139 cut), 512^2 49 (14).  Zero-mean noise,
// whose cells differ in exponent and lie further apart than 2^9, takes own_cells: 146, 91, 39.
//
// Work split: the tiles are cut into equal contiguous ranges, one per CTA.
#include <cudaTypedefs.h>

#include "internal.h"
#include "ptx.cuh"
#include "taps.cuh"
#include "wide.cuh"
#include "widestream.cuh"

namespace gbst {

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();  // stream.cu

namespace {

constexpr int kTX = kWTX, kRaw = kWRaw, kWarps = kWWarps, kThreads = kWThreads;
constexpr int kTC = 16;                // tile rows
constexpr int kR = kTC / kWarps;       // rows of a consumer warp
constexpr int kU = 3;

template <int RAD>
using Plane = WidePlane<kTC + 2 * RAD>;

template <int RAD, bool TMA>
struct __align__(128) Smem {
  double raw[kRaw][kTC + 2 * RAD][raw_col<TMA>()];
  int shift[kRaw][kTC + 2 * RAD];  // bulk copies: position of column x0 in the row (0 or 1)
  Plane<RAD> u[kU];
  uint64_t full[kRaw];   // raw tile has landed
  uint64_t empty[kRaw];  // raw tile is unpacked: 8 consumer warps, the producer
  uint64_t conv[kU];     // tile is unpacked: the same 9 arrivals
};
static_assert(kU == kRaw, "one ring position serves both");

struct Params {
  CUtensorMap map_row;   // box {64, 1} over src
  CUtensorMap map_tile;  // box {64, 16 + 2 RAD} over src
  const double* src;
  double* dst;
  int ny, nx;
  int tiles_y;
  int work;  // tiles
  int vec;   // rows start on 16 bytes
  int* status;
  const double* wdev;
  WideTaps wide;
  WideEqualTaps equal;         // of a box with wide.equal
  unsigned long long wait_ns;  // of STARVED
};

// First column and row of a tile, advanced tile by tile (a division per warp and tile
// would be 6 of a cell's 125 instructions).
struct TilePos {
  int x0, y0;
  __device__ __forceinline__ TilePos(int t, int tiles_y) : x0(t / tiles_y * kTX), y0(t % tiles_y * kTC) {}
  __device__ __forceinline__ void next(int ny) {
    y0 += kTC;
    if (y0 >= ny) {
      y0 = 0;
      x0 += kTX;
    }
  }
};

// -n <= c, wrapped; what lies further than n beyond the end (rows of a ragged tile
// that nobody uses): any of them.
__device__ __forceinline__ int wrap_near(int c, int n) { return c < 0 ? c + n : c >= n ? min(c - n, n - 1) : c; }

// Position of offset (dy, dx) in the lexicographic tap list of the class.
template <bool BOX, int RAD>
__device__ __forceinline__ constexpr int tap_at(int dy, int dx) {
  if (BOX) return (dy + RAD) * (2 * RAD + 1) + (dx + RAD);
  return dy < 0 ? dy + RAD : dy > 0 ? 3 * RAD + dy : 2 * RAD + dx;
}

// Columns c-RAD .. c+1+RAD of a row.
template <int RAD>
__device__ __forceinline__ void get_row(const Plane<RAD>& u, int row, int c, WideVal (&v)[2 * RAD + 2]) {
  get_pair(&u.m[row][c], &u.e[row][c], v[RAD], v[RAD + 1]);
  if constexpr (RAD == 1) {
    v[0] = get(&u.m[row][c - 1], &u.e[row][c - 1]);
    v[3] = get(&u.m[row][c + 2], &u.e[row][c + 2]);
  } else {
    get_pair(&u.m[row][c - 2], &u.e[row][c - 2], v[0], v[1]);
    get_pair(&u.m[row][c + 2], &u.e[row][c + 2], v[4], v[5]);
  }
}

// A lane's cells where all that they read are zeros (false: they are not).  Out of line,
// and apart from chain_cells, whose frame would cost more than this does.
template <bool BOX, int RAD>
__device__ __noinline__ bool zero_cells(const Plane<RAD>& u, int row0, int rows, int cols, int c0, double* out, int nx) {
  constexpr int RX = BOX ? RAD : 0;  // (nobody writes a star's corner columns)
  if (!zero_rows<kR, RAD>(u, row0, c0, cols) || !zero_rows<RAD, RX>(u, row0 - RAD, c0, cols) ||
      !zero_rows<RAD, RX>(u, row0 + kR, c0, cols))
    return false;
  put_zeros(out, rows, cols, nx);
  return true;
}

// One cell by the FMA chain.
template <bool BOX, int RAD, bool TWOS = false>
__device__ __noinline__ double chain_cell(const Plane<RAD>& u, int row, int c, const double* wdev) {
  constexpr int NT = BOX ? (2 * RAD + 1) * (2 * RAD + 1) : 4 * RAD + 1;
  double v[NT];
  for (int dy = -RAD; dy <= RAD; ++dy)
    for (int dx = -RAD; dx <= RAD; ++dx) {
      if (!BOX && dy != 0 && dx != 0) continue;
      const WideVal x = get(&u.m[row + dy][c + dx], &u.e[row + dy][c + dx]);
      v[tap_at<BOX, RAD>(dy, dx)] = wide_repack(TWOS ? wide_ones(x) : x);
    }
  return wide_chain(v, wdev, NT);
}

// The cells of a lane that the integer form does not take: zeros, or by the FMA chain:
// `cols` columns from c0 on of rows row0 .. row0+rows-1.  Out of line: rarely run.
template <bool BOX, int RAD>
__device__ __noinline__ void chain_cells(const Plane<RAD>& u, int row0, int rows, int cols, int c0, const WideTaps& T,
                                         const double* wdev, double* out, int nx) {
  for (int r = 0; r < rows; ++r)
    for (int i = 0; i < cols; ++i) {
      const int row = row0 + r, c = c0 + i;
      unsigned int any = 0;
      int E = -0x7fffffff;
#pragma unroll
      for (int dy = -RAD; dy <= RAD; ++dy)
#pragma unroll
        for (int dx = -RAD; dx <= RAD; ++dx) {
          if (!BOX && dy != 0 && dx != 0) continue;
          const WideVal x = get(&u.m[row + dy][c + dx], &u.e[row + dy][c + dx]);
          any |= wide_nonzero(x);
          E = max(E, x.e + T.ex[tap_at<BOX, RAD>(dy, dx)]);
        }
      if (any == 0) out[(int64_t)r * nx + i] = 0.0;
      else if (!wide_covers(E, T)) out[(int64_t)r * nx + i] = chain_cell<BOX, RAD>(u, row, c, wdev);
    }
}

// An equal-weight box's cells of a lane, each aligned to its own exponent E (or by the FMA
// chain).  Out of line: where they differ in E and are not within 2^9 of each other.
template <int RAD>
__device__ __noinline__ void own_cells(const Plane<RAD>& u, int row0, int rows, int cols, int c, const WideTaps& T,
                                       const double* wdev, double* out, int nx) {
#pragma unroll 1
  for (int r = 0; r < rows; ++r) {
    const int row = row0 + r;
    int E[2] = {0, 0};
#pragma unroll
    for (int dy = -RAD; dy <= RAD; ++dy)
#pragma unroll
      for (int dx = -RAD; dx <= RAD + 1; ++dx) {
        const int e = u.e[row + dy][c + dx];
        if (dx <= RAD) E[0] = max(E[0], e);
        if (dx > -RAD) E[1] = max(E[1], e);
      }
    E[0] |= 3;
    E[1] |= 3;
    WideSum S[2];
#pragma unroll
    for (int dy = -RAD; dy <= RAD; ++dy) {
      WideVal v[2 * RAD + 2];
      get_row<RAD>(u, row + dy, c, v);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int k = 0; k < 2 * RAD + 1; ++k) S[i] += wide_part(v[i + k], E[i]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (i < cols)
        out[(int64_t)r * nx + i] =
            wide_covers(E[i], T) ? wide_equal_double(S[i], E[i], T) : chain_cell<true, RAD, true>(u, row, c + i, wdev);
  }
}

// The smallest exponent of the values that an equal-weight box's lane reads.
template <int RAD>
__device__ __forceinline__ int least_exponent(const Plane<RAD>& u, int row0, int c) {
  int e = 0x7fffffff;
#pragma unroll
  for (int r = -RAD; r < kR + RAD; ++r)
#pragma unroll
    for (int x = -RAD; x < 2 + RAD; ++x) e = min(e, u.e[row0 + r][c + x]);
  return e;
}

template <bool BOX, int RAD, bool HEAT>
constexpr int wide2d_ctas() { return RAD == 1 && (!BOX || HEAT) ? 3 : 2; }

// HEAT: a star whose weights wide_sum_heat takes; a box whose weights are all equal.
// STARVED: the self-test of the bounded waits: no copy (and no arrival that announces one) for a
// CTA's tiles, and waits of P.wait_ns.
template <bool BOX, int RAD, bool HEAT, bool PERIODIC, bool TMA, bool STARVED = false>
__global__ void __launch_bounds__(kThreads, (wide2d_ctas<BOX, RAD, HEAT>())) k_wide2d(const __grid_constant__ Params P) {
  constexpr int kRows = kTC + 2 * RAD;
  const unsigned long long kWaitNs = STARVED ? P.wait_ns : (unsigned long long)kSpinLimitNs;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Smem<RAD, TMA>& S = *reinterpret_cast<Smem<RAD, TMA>*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRaw; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], kWarps + 1);
      mbar_init(&S.conv[s], kWarps + 1);
    }
    fence_mbar_init();
    if (TMA) {
      prefetch_tmap(&P.map_row);
      prefetch_tmap(&P.map_tile);
    }
  }
  __syncthreads();
  step_begins();
  // a bounded wait; false: it gave up (the other warps' waits on this one then do the same)
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (mbar_wait_bounded(bar, parity, kWaitNs)) return true;
    atomicCAS(P.status, 0, -5 /* STENCIL_ERR_TIMEOUT */);
    return false;
  };
  const int64_t pitch = P.nx;
  const int t0 = (int)((long long)P.work * blockIdx.x / gridDim.x);
  const int t1 = (int)((long long)P.work * (blockIdx.x + 1) / gridDim.x);
  RingPos<kU> pos;       // of tile g
  int u1 = kU - 1;       // slot of tile g-1
  uint32_t ph1 = 1;      // its phase (a fresh barrier lets a wait for phase 1 pass)
  auto next = [&] {
    u1 = pos.s;
    ph1 = pos.ph;
    pos.next();
  };
  if (warp == kWarps) {
    // ------------------------------------------------------------ producer
    RingPos<kU> post;  // of the next tile to post
    int posted = t0;
    TilePos ptile(t0, P.tiles_y), tile = ptile, htile = ptile;  // of the next tile to post, of tile g, of the halo's
    // copies the next tile into its raw slot, once the slot's earlier tile is unpacked
    auto post_tile = [&] {
      if (!wait(&S.empty[post.s], post.ph ^ 1)) return false;
      const int x0 = ptile.x0, y0 = ptile.y0;
      const int r = lane;
      int y = y0 - RAD + r;
      if (TMA) {
        const bool whole = !PERIODIC || (y0 >= RAD && y0 + kTC + RAD <= P.ny);
        fence_proxy_async_smem();
        if (lane == 0 && !STARVED) {
          mbar_arrive_expect_tx(&S.full[post.s], (uint32_t)sizeof(S.raw[0]));
          if (whole) tma_load_2d(&S.raw[post.s][0][0], &P.map_tile, x0, y0 - RAD, &S.full[post.s]);
        }
        __syncwarp();
        if (!whole && r < kRows && !STARVED)
          tma_load_2d(&S.raw[post.s][r][0], &P.map_row, x0, wrap_near(y, P.ny), &S.full[post.s]);
      } else {
        bool in = r < kRows;
        if (PERIODIC) {
          in = in && y < P.ny + RAD;  // rows past the ghosts of a ragged tile are not read
          y = wrap_near(y, P.ny);
        } else {
          in = in && y >= 0 && y < P.ny;
        }
        RowCopy cp;
        if (in) {
          cp.plan(S.raw[post.s][r], P.src + (y * pitch + x0), min(kTX, P.nx - x0), P.src, P.src + P.ny * pitch);
          fence_proxy_async_smem();
        }
        if (r < kRows) S.shift[post.s][r] = cp.shift;
        // rows outside the grid are zeros
        unsigned int out = __ballot_sync(0xffffffffu, r < kRows && !in);
        while (out) {
          const int q = __ffs((int)out) - 1;
          out &= out - 1;
          S.raw[post.s][q][lane] = 0.0;
          S.raw[post.s][q][lane + 32] = 0.0;
        }
        const uint32_t total = __reduce_add_sync(0xffffffffu, cp.bytes);
        __syncwarp();  // the lanes' own writes come before lane 0's arrival
        if (lane == 0) mbar_arrive_expect_tx(&S.full[post.s], total);
        __syncwarp();
        if (cp.bytes) bulk_load(&S.raw[post.s][r][cp.to], cp.from, cp.bytes, &S.full[post.s]);
      }
      post.next();
      ptile.next(P.ny);
      ++posted;
      return true;
    };
    // the columns beside a tile: RAD on either side of every row that has
    // them (star: the tile's own rows), HN values per lane
    constexpr int HR = BOX ? kRows : kTC, H0 = BOX ? 0 : RAD, HALL = 2 * RAD * HR, HN = (HALL + 31) / 32;
    auto halo = [&](double (&h)[HN]) {
      const int x0 = htile.x0, y0 = htile.y0;
      const int cols = TMA ? kTX : min(kTX, P.nx - x0);
#pragma unroll
      for (int q = 0; q < HN; ++q) {
        const int k = lane + 32 * q, j = k / HR;  // j: the column, west to east
        int x = j < RAD ? x0 - RAD + j : x0 + cols + (j - RAD), y = y0 - RAD + H0 + k % HR;
        bool in = k < HALL;
        if (PERIODIC) {
          x = wrap_near(x, P.nx);
          y = wrap_near(y, P.ny);
        } else {
          in = in && x >= 0 && x < P.nx && y >= 0 && y < P.ny;
        }
        h[q] = in ? __ldcg(P.src + (y * pitch + x)) : 0.0;
      }
      htile.next(P.ny);
    };
    // a wait that gave up: the copies already posted land (bounded) before the warp leaves
    auto leave = [&](int t) {
      RingPos<kU> q = pos;
      for (int k = t; k < posted; ++k, q.next()) mbar_wait_bounded(&S.full[q.s], q.ph, kWaitNs);
    };
    double h[HN], hn[HN];
    if (t0 < t1) halo(h);
    while (posted < t1 && posted < t0 + kRaw)
      if (!post_tile()) return leave(t0);
    for (int t = t0; t < t1; ++t) {
      if (t + 1 < t1) halo(hn);
      if (!wait(&S.conv[u1], ph1)) return leave(t);
      Plane<RAD>& u = S.u[pos.s];
      const int cols = TMA ? kTX : min(kTX, P.nx - tile.x0);
#pragma unroll
      for (int q = 0; q < HN; ++q) {
        const int k = lane + 32 * q, j = k / HR, row = H0 + k % HR;
        const int c = 2 + (j < RAD ? j - RAD : cols + (j - RAD));
        if (k < HALL) put(&u.m[row][c], &u.e[row][c], BOX && HEAT ? wide_twos(wide_unpack(h[q])) : wide_unpack(h[q]));
      }
      if (!wait(&S.full[pos.s], pos.ph)) return leave(t);
      WideVal v[2];
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        unpack_row<TMA, kRows, BOX && HEAT>(S.raw[pos.s], S.shift[pos.s], u, r, lane, cols, v);
        unpack_row<TMA, kRows, BOX && HEAT>(S.raw[pos.s], S.shift[pos.s], u, kTC + RAD + r, lane, cols, v);
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&S.empty[pos.s]);
        mbar_arrive(&S.conv[pos.s]);
      }
#pragma unroll
      for (int q = 0; q < HN; ++q) h[q] = hn[q];
      next();
      tile.next(P.ny);
      // (after this tile's share of the unpacking, which the consumers wait for)
      if (posted < t1 && !post_tile()) return leave(t + 1);
    }
    return;
  }
  // -------------------------------------------------------------- consumers
  const int row0 = RAD + warp * kR;  // the warp's first row in the planes
  const int c = 2 + 2 * lane;
  TilePos tile(t0, P.tiles_y), before = tile;  // of tiles g and g-1
  for (int t = t0; t <= t1 && t0 < t1; ++t) {  // (the last iteration unpacks nothing)
    if (!wait(&S.conv[u1], ph1)) return;
    if (t < t1) {
      if (!wait(&S.full[pos.s], pos.ph)) return;
      const int cols = TMA ? kTX : min(kTX, P.nx - tile.x0);
      WideVal v[2];
#pragma unroll
      for (int r = 0; r < kR; ++r)
        unpack_row<TMA, kRows, BOX && HEAT>(S.raw[pos.s], S.shift[pos.s], S.u[pos.s], row0 + r, lane, cols, v);
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&S.empty[pos.s]);
        mbar_arrive(&S.conv[pos.s]);
      }
    }
    if (t > t0) {
      const Plane<RAD>& u = S.u[u1];
      const int xa = before.x0 + 2 * lane, ya = before.y0 + warp * kR;
      const int rows = xa < P.nx ? min(kR, P.ny - ya) : 0;  // rows that the lane stores
      double* out = P.dst + ya * pitch + xa;
      auto store = [&](int r, double v0, double v1) {
        if (r >= rows) return;
        double* o = out + r * pitch;
        if (TMA || (P.vec && xa + 1 < P.nx)) {  // (TMA grids: nx even, rows on 16 bytes)
          st_global_v2(o, v0, v1);
        } else {
          o[0] = v0;
          if (xa + 1 < P.nx) o[1] = v1;
        }
      };
      // the integer form takes every cell that is stored (the others may hold anything)
      bool all = true, zeros = true;  // (zeros: there may be nothing else)
      auto covers = [&](bool ok, int r, int i) { return ok || r >= rows || (!TMA && i == 1 && xa + 1 >= P.nx); };
      if constexpr (!BOX) {
#pragma unroll
        for (int r = 0; r < kR; ++r) {
          const int row = row0 + r;
          WideVal y[2 * RAD][2], x[2 * RAD + 2];
#pragma unroll
          for (int k = 0; k < 2 * RAD; ++k) {
            const int rr = row + (k < RAD ? k - RAD : k - RAD + 1);
            get_pair(&u.m[rr][c], &u.e[rr][c], y[k][0], y[k][1]);
          }
          get_row<RAD>(u, row, c, x);
          double v[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            WideVal w[4 * RAD + 1];
#pragma unroll
            for (int k = 0; k < RAD; ++k) {
              w[k] = y[k][i];
              w[3 * RAD + 1 + k] = y[RAD + k][i];
            }
#pragma unroll
            for (int k = 0; k <= 2 * RAD; ++k) w[RAD + k] = x[i + k];
            bool ok;
            if constexpr (HEAT) v[i] = wide_sum_heat<4 * RAD + 1>(w, P.wide, ok);
            else v[i] = wide_sum<4 * RAD + 1>(w, P.wide, ok);
            all = all && covers(ok, r, i);
          }
          store(r, v[0], v[1]);
        }
      } else if constexpr (HEAT) {
        // equal weights, the lane's two rows and columns as one block: each value is
        // aligned once for the four cells, and rows (mid: their common columns) and
        // columns share their partial sums
        constexpr int N = 2 * RAD + 2;
        static_assert(kR == 2, "the block");
        int own[2][2], e[N][N];  // the cells' largest exponents
#pragma unroll
        for (int r = 0; r < N; ++r) {
          const int* er = &u.e[row0 - RAD + r][c];
#pragma unroll
          for (int k = 0; k < RAD + 1; ++k) {
            if (RAD == 1 && k != 0) continue;
            const int2 m = *reinterpret_cast<const int2*>(er + (RAD == 1 ? 0 : 2 * k - 2));
            e[r][RAD == 1 ? 1 : 2 * k] = m.x;
            e[r][RAD == 1 ? 2 : 2 * k + 1] = m.y;
          }
          if (RAD == 1) {
            e[r][0] = er[-1];
            e[r][3] = er[2];
          }
          int mid = e[r][1];
#pragma unroll
          for (int k = 2; k < N - 1; ++k) mid = max(mid, e[r][k]);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int h = max(mid, e[r][i * (N - 1)]);
            if (r < N - 1) own[0][i] = r == 0 ? h : max(own[0][i], h);
            if (r > 0) own[1][i] = r == 1 ? h : max(own[1][i], h);
          }
        }
        // (what is not stored may hold anything)
        if (!TMA && xa + 1 >= P.nx) {
          own[0][1] = own[0][0];
          own[1][1] = own[1][0];
        }
        if (rows < 2) {
          own[1][0] = own[0][0];
          own[1][1] = own[0][1];
        }
        int E = max(max(own[0][0], own[0][1]), max(own[1][0], own[1][1])) | 3;
        const int least = min(min(own[0][0], own[0][1]), min(own[1][0], own[1][1])) | 3;
        zeros = E == 3;
        // Where cells differ in E (a field passes a power of 16), no bit is cut as long as all
        // values are within the 2^9 that the integers have room for: the sums are exact then,
        // and those of each cell's own alignment follow.  Else the warp takes own_cells.
        all = wide_covers(E, P.equal) && (E == least || (wide_covers(least, P.equal) && least_exponent<RAD>(u, row0, c) + 9 >= E));
        const bool fits = __all_sync(0xffffffffu, all || rows <= 0);
        all = rows <= 0 || fits;
        if (fits) {
          WideSum S[2][2], both[2];  // both: of the rows that both read
          if (RAD > 1) asm volatile("" ::: "memory");  // 36 exponents would not fit the registers: read again
          // (two values fit 64 bits: by pairs, side by side or one below the other)
          auto part = [&](const WideVal& x, const WideVal& y) {
            return WideSum(wide_align(x, E - x.e) + wide_align(y, E - y.e));
          };
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            WideVal v[N];
            get_row<RAD>(u, row0 - RAD + q * (N - 1), c, v);
            WideSum mid = part(v[1], v[2]);
#pragma unroll
            for (int k = 3; k < N - 1; k += 2) mid += part(v[k], v[k + 1]);
#pragma unroll
            for (int i = 0; i < 2; ++i) S[q][i] = mid + wide_part(v[i * (N - 1)], E);
          }
#pragma unroll
          for (int r = 1; r < N - 1; r += 2) {
            WideVal v[N], w[N];
            get_row<RAD>(u, row0 - RAD + r, c, v);
            get_row<RAD>(u, row0 - RAD + r + 1, c, w);
            WideSum mid = part(v[1], w[1]);
#pragma unroll
            for (int k = 2; k < N - 1; ++k) mid += part(v[k], w[k]);
#pragma unroll
            for (int i = 0; i < 2; ++i) both[i] += mid + part(v[i * (N - 1)], w[i * (N - 1)]);
          }
          int Ec[2][2] = {{E, E}, {E, E}};
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              S[r][i] += both[i];
              if (E != least) {
                Ec[r][i] = own[r][i] | 3;
                S[r][i].shift(E - Ec[r][i]);
              }
            }
#pragma unroll
          for (int r = 0; r < 2; ++r)
            store(r, wide_equal_double(S[r][0], Ec[r][0], P.equal), wide_equal_double(S[r][1], Ec[r][1], P.equal));
        }
      } else {
        // row by row; the largest exponents first, then the sums: a pair's values would
        // not fit the registers, so their rows are read twice
#pragma unroll 1
        for (int r = 0; r < kR; ++r) {
          int E[2] = {-0x7fffffff, -0x7fffffff};
#pragma unroll
          for (int dy = -RAD; dy <= RAD; ++dy) {
            const int* er = &u.e[row0 + r + dy][c];
            int e[2 * RAD + 2];
#pragma unroll
            for (int k = 0; k < RAD + 1; ++k) {
              if (RAD == 1 && k != 0) continue;
              const int2 m = *reinterpret_cast<const int2*>(er + (RAD == 1 ? 0 : 2 * k - 2));
              e[RAD == 1 ? 1 : 2 * k] = m.x;
              e[RAD == 1 ? 2 : 2 * k + 1] = m.y;
            }
            if (RAD == 1) {
              e[0] = er[-1];
              e[3] = er[2];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
              for (int dx = -RAD; dx <= RAD; ++dx)
                E[i] = max(E[i], e[RAD + i + dx] + P.wide.ex[tap_at<true, RAD>(dy, dx)]);
          }
          WideAcc acc[2];
#pragma unroll
          for (int dy = -RAD; dy <= RAD; ++dy) {
            WideVal v[2 * RAD + 2];
            get_row<RAD>(u, row0 + r + dy, c, v);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
              for (int dx = -RAD; dx <= RAD; ++dx) {
                const int k = tap_at<true, RAD>(dy, dx);
                acc[i].add(v[RAD + i + dx], k, E[i] - v[RAD + i + dx].e - P.wide.ex[k], P.wide);
              }
          }
          all = all && covers(wide_covers(E[0], P.wide), r, 0) && covers(wide_covers(E[1], P.wide), r, 1);
          store(r, acc[0].get(E[0], P.wide), acc[1].get(E[1], P.wide));
        }
      }
      if (!all && (!zeros || !zero_cells<BOX, RAD>(u, row0, rows, min(2, P.nx - xa), c, out, P.nx))) {
        if constexpr (BOX && HEAT) own_cells<RAD>(u, row0, rows, min(2, P.nx - xa), c, P.wide, P.wdev, out, P.nx);
        else chain_cells<BOX, RAD>(u, row0, rows, min(2, P.nx - xa), c, P.wide, P.wdev, out, P.nx);
      }
      __syncwarp();
    }
    if (t < t1) next();
    before = tile;
    tile.next(P.ny);
  }
}

bool encode_2d(CUtensorMap* map, const double* base, const Geom& g, int rows) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny};
  cuuint64_t strides[1] = {(cuuint64_t)g.nx * sizeof(double)};
  cuuint32_t box[2] = {(cuuint32_t)kTX, (cuuint32_t)rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<double*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool BOX, int RAD, bool HEAT, bool PERIODIC, bool TMA, bool STARVED = false>
cudaError_t launch_t(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                     int* status, int sms, cudaStream_t stream, bool chained, unsigned long long wait_ns = 0) {
  auto kern = k_wide2d<BOX, RAD, HEAT, PERIODIC, TMA, STARVED>;
  constexpr size_t bytes = sizeof(Smem<RAD, TMA>);
  static std::atomic<int> cache[kMaxDeviceOrdinals];
  const int occ = cached_per_device(cache, [kern] {
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kThreads, bytes) != cudaSuccess)
      n = 0;
    return n;
  });
  if (occ < 1) return cudaErrorInvalidConfiguration;
  Params P;
  if (TMA && (!encode_2d(&P.map_row, src, g, 1) || !encode_2d(&P.map_tile, src, g, kTC + 2 * RAD)))
    return cudaErrorInvalidValue;
  P.src = src;
  P.dst = dst;
  P.ny = g.ny;
  P.nx = g.nx;
  P.tiles_y = (g.ny + kTC - 1) / kTC;
  const int64_t work = (int64_t)((g.nx + kTX - 1) / kTX) * P.tiles_y;
  if (work > INT32_MAX) return cudaErrorInvalidValue;
  P.work = (int)work;
  P.vec = g.nx % 2 == 0 && ((uintptr_t)dst & 15) == 0;
  P.status = status;
  P.wait_ns = wait_ns;
  P.wdev = wdev;
  P.wide = wide;
  P.equal = wide;
  int64_t grid = (int64_t)sms * occ;
  if (grid > work) grid = work;
  if (const cudaError_t e = launch_step(kern, (unsigned)grid, kThreads, bytes, stream, chained, P)) return e;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <bool BOX, int RAD, bool HEAT>
cudaError_t launch_p(bool per, bool tma, const Geom& g, const WideTaps& wide, const double* wdev, const double* src,
                     double* dst, int* status, int sms, cudaStream_t stream, bool chained) {
  if (tma)
    return per ? launch_t<BOX, RAD, HEAT, true, true>(g, wide, wdev, src, dst, status, sms, stream, chained)
               : launch_t<BOX, RAD, HEAT, false, true>(g, wide, wdev, src, dst, status, sms, stream, chained);
  return per ? launch_t<BOX, RAD, HEAT, true, false>(g, wide, wdev, src, dst, status, sms, stream, chained)
             : launch_t<BOX, RAD, HEAT, false, false>(g, wide, wdev, src, dst, status, sms, stream, chained);
}

}  // namespace

cudaError_t launch_wide2d(Shape shape, int radius, int boundary, const Geom& g, const WideTaps& wide,
                          const double* wdev, const double* src, double* dst, int* status, int sms,
                          cudaStream_t stream, bool tma, bool chained) {
  const bool per = boundary == kPeriodic, box = shape == Shape::kBox;
  const int side = 2 * radius + 1;
  if (wide.n != (box ? side * side : 4 * radius + 1)) return cudaErrorInvalidValue;
  if (box && wide.equal)
    return radius == 2 ? launch_p<true, 2, true>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained)
                       : launch_p<true, 1, true>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained);
  if (radius == 2)
    return box ? launch_p<true, 2, false>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained)
               : launch_p<false, 2, false>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained);
  if (box) return launch_p<true, 1, false>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained);
  return wide.heat ? launch_p<false, 1, true>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained)
                   : launch_p<false, 1, false>(per, tma, g, wide, wdev, src, dst, status, sms, stream, chained);
}

cudaError_t launch_wide2d_starved(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                                  int* status, int sms, cudaStream_t stream, unsigned long long wait_ns) {
  return launch_t<false, 1, true, true, true, true>(g, wide, wdev, src, dst, status, sms, stream, false, wait_ns);
}

}  // namespace gbst
