// wide3d.cu -- 3D radius-1 sweep (7-point star or 27-point box) with the
// weighted sum in the integer form (wide.cuh), streaming along z.
//
// One step of u'(x) = sum_o w_o u~(x+o) (paper Sec. 2.1, Listing 1).  The tile
// is 64 columns by TC rows, advanced plane by plane.  The integer issue rate is
// the bound, and unpacking a value costs about thirteen instructions, so every
// plane is unpacked once, into shared memory, and all its readers take it from
// there:
//   - raw planes (the tile's columns, one row more above and below) arrive up to
//     three ahead: by TMA boxes where the grid allows it (out-of-range boxes read
//     zeros, the Dirichlet ghosts), else row by row by bulk copies from the
//     16-byte boundary at or before the row's start, which take any size,
//     alignment and wrap;
//   - iteration g: every consumer warp unpacks its own TC/8 rows of plane g into
//     ring slot g % kU (the producer warp the rows and columns around the tile),
//     arrives on conv[g % kU], and computes its rows of the middle plane: g-1
//     for the star, which reads only its own rows of plane g, and g-2 for the box;
//   - it waits for conv(g-1) before it unpacks plane g: plane g-1 is then
//     complete, and every warp has left iteration g-2, the last in which it reads
//     another warp's rows of the plane whose slot plane g takes.
// Each lane owns two adjacent columns.  Warps meet only at mbarriers; every wait is
// bounded.
//
// Measured at 512^3, star, periodic: 166 GStencil/s (87 for the FMA chain, whose
// bound is the FP64 pipe).  Registers instead of shared memory for the three
// planes (1.5 unpacks per cell, rows of 4) ran at 142 and spilled; a converter
// warp that loads and unpacks everything for the consumers at 94.
// Box, 384^3, zero outside: general weights 48 GStencil/s (22.7 for the FMA chain), equal
// ones (WideSum) 102, 64 where a warp takes own_cells (zero-mean noise).  Each plane's sums kept
// in registers for the next two planes spilled.
// Work split: the (tile, z) planes are cut into equal contiguous ranges, one per CTA.
#include <cudaTypedefs.h>

#include "internal.h"
#include "ptx.cuh"
#include "taps.cuh"
#include "wide.cuh"
#include "widestream.cuh"

namespace gbst {

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder();  // stream.cu

namespace {

constexpr int kTX = kWTX, kRaw = kWRaw;
// Consumer warps: two rows each of a tile of 16, one of 8; of 32 rows (a caller's or the tuner's
// choice) twice as many, one CTA to an SM.  GStencil/s at 8, 16 and 32 rows: heat 512^3 138, 170.5,
// 173.5, 128^3 96, 106, 118, general box 384^3 46, 48.7, 50.5, equal box 77, 108, 110.
template <int TC>
constexpr int warps() { return TC == 32 ? 2 * kWWarps : kWWarps; }
template <int TC>
constexpr int threads() { return 32 * (warps<TC>() + 1); }
template <int TC>
using Plane = WidePlane<TC + 2>;

// Unpacked planes.  Star: the three that are read.  Box: a warp reads other
// warps' rows of all three, the oldest (g-4 in iteration g-1) while another warp
// may already be unpacking plane g: five.
template <bool BOX>
constexpr int ring() { return BOX ? 5 : 3; }

template <bool BOX, bool TMA, int TC>
struct __align__(128) Smem {
  double raw[kRaw][TC + 2][raw_col<TMA>()];
  int shift[kRaw][TC + 2];      // bulk copies: position of column x0 in the row (0 or 1)
  Plane<TC> u[ring<BOX>()];
  uint64_t full[kRaw];          // raw plane has landed
  uint64_t empty[kRaw];         // raw plane is unpacked: 8 consumer warps, the producer
  uint64_t conv[ring<BOX>()];   // plane is unpacked: the same 9 arrivals
};

struct Params {
  CUtensorMap map_row;   // box {64, 1, 1} over src
  CUtensorMap map_main;  // box {64, TC, 1} over src
  const double* src;
  double* dst;
  int nz, ny, nx;
  int tiles_x, tiles_y;
  long long work;  // tiles * nz
  int vec;         // rows start on 16 bytes
  int* status;
  const double* wdev;
  WideTaps wide;
  WideEqualTaps equal;         // of a box with wide.equal
  unsigned long long wait_ns;  // of STARVED
};

// Columns c-1 .. c+2 of a row.
template <int TC>
__device__ __forceinline__ void get_row(const Plane<TC>& u, int row, int c, WideVal (&v)[4]) {
  v[0] = get(&u.m[row][c - 1], &u.e[row][c - 1]);
  get_pair(&u.m[row][c], &u.e[row][c], v[1], v[2]);
  v[3] = get(&u.m[row][c + 2], &u.e[row][c + 2]);
}

// Tap index of offset (dz, dy, dx) in the class's lexicographic tap list.
template <bool BOX>
__device__ __forceinline__ constexpr int tap_at(int dz, int dy, int dx) {
  if (BOX) return ((dz + 1) * 3 + (dy + 1)) * 3 + (dx + 1);
  return dz < 0 ? 0 : dz > 0 ? 6 : dy < 0 ? 1 : dy > 0 ? 5 : 3 + dx;
}

// A lane's cells where all that they read are zeros (false: they are not).  Out of line,
// and apart from chain_cells, whose frame would cost more than this does.
template <bool BOX, int TC>
__device__ __noinline__ bool zero_cells(const Plane<TC>& um, const Plane<TC>& u0, const Plane<TC>& up, int row0,
                                        int rows, int cols, int c0, double* out, int nx) {
  constexpr int R = TC / warps<TC>();
  if (!zero_rows<R, 1>(u0, row0, c0, cols)) return false;
  if (BOX ? !zero_rows<1, 1>(u0, row0 - 1, c0, cols) || !zero_rows<1, 1>(u0, row0 + R, c0, cols) ||
                !zero_rows<R + 2, 1>(um, row0 - 1, c0, cols) || !zero_rows<R + 2, 1>(up, row0 - 1, c0, cols)
          // (nobody writes a star's corner columns)
          : !zero_rows<1, 0>(u0, row0 - 1, c0, cols) || !zero_rows<1, 0>(u0, row0 + R, c0, cols) ||
                !zero_rows<R, 0>(um, row0, c0, cols) || !zero_rows<R, 0>(up, row0, c0, cols))
    return false;
  put_zeros(out, rows, cols, nx);
  return true;
}

// One cell by the FMA chain.
template <bool BOX, int TC, bool TWOS = false>
__device__ __noinline__ double chain_cell(const Plane<TC>& um, const Plane<TC>& u0, const Plane<TC>& up, int row, int c,
                                          const double* wdev) {
  constexpr int NT = BOX ? 27 : 7;
  const Plane<TC>* const pl[3] = {&um, &u0, &up};
  double v[NT];
  for (int k = 0; k < 27; ++k) {
    const int dz = k / 9 - 1, dy = k / 3 % 3 - 1, dx = k % 3 - 1;
    if (!BOX && (dz != 0) + (dy != 0) + (dx != 0) > 1) continue;
    const WideVal x = get(&pl[dz + 1]->m[row + dy][c + dx], &pl[dz + 1]->e[row + dy][c + dx]);
    v[tap_at<BOX>(dz, dy, dx)] = wide_repack(TWOS ? wide_ones(x) : x);
  }
  return wide_chain(v, wdev, NT);
}

// The cells of a lane that the integer form does not take: zeros, or by the FMA chain:
// `cols` columns from c0 on of rows row0 .. row0+rows-1.  Out of line, one call for
// a lane's cells: rarely run, and a call within the sum's code costs every cell
// 19 instructions.
template <bool BOX, int TC>
__device__ __noinline__ void chain_cells(const Plane<TC>& um, const Plane<TC>& u0, const Plane<TC>& up, int row0,
                                         int rows, int cols, int c0, const WideTaps& T, const double* wdev,
                                         double* out, int nx) {
  for (int r = 0; r < rows; ++r)
    for (int i = 0; i < cols; ++i) {
      const int row = row0 + r, c = c0 + i;
      unsigned int any = 0;
      int E = -0x7fffffff;
#pragma unroll
      for (int k = 0; k < 27; ++k) {
        const int dz = k / 9 - 1, dy = k / 3 % 3 - 1, dx = k % 3 - 1;
        if (!BOX && (dz != 0) + (dy != 0) + (dx != 0) > 1) continue;
        const Plane<TC>& p = dz < 0 ? um : dz > 0 ? up : u0;
        const WideVal u = get(&p.m[row + dy][c + dx], &p.e[row + dy][c + dx]);
        any |= wide_nonzero(u);
        E = max(E, u.e + T.ex[tap_at<BOX>(dz, dy, dx)]);
      }
      if (any == 0) out[(int64_t)r * nx + i] = 0.0;
      else if (!wide_covers(E, T)) out[(int64_t)r * nx + i] = chain_cell<BOX, TC>(um, u0, up, row, c, wdev);
    }
}

// An equal-weight box's cells of a lane, each aligned to its own exponent E (or by the FMA
// chain).  Out of line: where they differ in E and are not within 2^9 of each other.
template <int TC>
__device__ __noinline__ void own_cells(const Plane<TC>& um, const Plane<TC>& u0, const Plane<TC>& up, int row0, int rows,
                                       int cols, int c, const WideTaps& T, const double* wdev, double* out, int nx) {
  const Plane<TC>* const pl[3] = {&um, &u0, &up};
#pragma unroll 1
  for (int r = 0; r < rows; ++r) {
    const int row = row0 + r;
    int E[2] = {0, 0};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int* er = &pl[k / 3]->e[row + k % 3 - 1][c];
      const int2 m = *reinterpret_cast<const int2*>(er);
      const int mid = max(m.x, m.y);
      E[0] = max(E[0], max(mid, er[-1]));
      E[1] = max(E[1], max(mid, er[2]));
    }
    E[0] |= 3;
    E[1] |= 3;
    WideSum S[2];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      WideVal v[4];
      get_row<TC>(*pl[k / 3], row + k % 3 - 1, c, v);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int x = 0; x < 3; ++x) S[i] += wide_part(v[i + x], E[i]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (i < cols)
        out[(int64_t)r * nx + i] =
            wide_covers(E[i], T) ? wide_equal_double(S[i], E[i], T) : chain_cell<true, TC, true>(um, u0, up, row, c + i, wdev);
  }
}

// HEAT: a star whose weights wide_sum_heat takes; a box whose weights are all equal.
// Three CTAs of nine warps per SM where 72 registers are enough (199 x 251 x 301 by bulk
// copies, us a step, three against two: heat 124 / 137; general weights, which spill,
// 167 / 148).
// STARVED: the self-test of the bounded waits: no copy (and no arrival that announces one) for a
// CTA's second plane, and waits of P.wait_ns.
template <bool BOX, bool HEAT, bool PERIODIC, bool TMA, int TC, bool STARVED = false>
__global__ void __launch_bounds__(threads<TC>(), TC == 32 ? 1 : BOX || !(TMA || HEAT) ? 2 : 3)
    k_wide3d(const __grid_constant__ Params P) {
  constexpr int kWarps = warps<TC>(), R = TC / kWarps;  // R: rows of a consumer warp
  static_assert(TMA || TC < 32, "by bulk copies, a lane copies a row");
  constexpr int kU = ring<BOX>();
  constexpr int kLag = BOX ? 2 : 1;  // the middle plane is kLag planes behind the one being unpacked
  const unsigned long long kWaitNs = STARVED ? P.wait_ns : (unsigned long long)kSpinLimitNs;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Smem<BOX, TMA, TC>& S = *reinterpret_cast<Smem<BOX, TMA, TC>*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRaw; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], kWarps + 1);
    }
    for (int s = 0; s < kU; ++s) mbar_init(&S.conv[s], kWarps + 1);
    fence_mbar_init();
    if (TMA) {
      prefetch_tmap(&P.map_row);
      prefetch_tmap(&P.map_main);
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
  const int64_t pitch = P.nx, plane = (int64_t)P.ny * P.nx;
  RingPos<kRaw> raw;  // of plane g
  RingPos<kU> ring;   // of plane g
  auto con = [&]() -> const auto& {  // (the same numbers when the rings are of one length)
    if constexpr (kU == kRaw) return raw;
    else return ring;
  };
  int u1 = kU - 1, u2 = kU - 2, u3 = kU - 3;  // slots of planes g-1, g-2, g-3
  uint32_t ph1 = 1;   // phase of plane g-1 (a fresh barrier lets a wait for phase 1 pass)
  auto next = [&] {
    u3 = u2;
    u2 = u1;
    u1 = con().s;
    ph1 = con().ph;
    raw.next();
    if constexpr (kU != kRaw) ring.next();
  };
  // the CTA's range of the (tile, z) planes; its ends are worked out again for
  // every tile rather than kept in registers
  auto range = [&](unsigned int b) { return P.work * b / gridDim.x; };
  for (int tile = (int)(range(blockIdx.x) / P.nz);; ++tile) {
    const long long first = (long long)tile * P.nz;
    if (first >= range(blockIdx.x + 1)) return;
    const int za = (int)max(0ll, range(blockIdx.x) - first);
    const int zb = (int)min((long long)P.nz, range(blockIdx.x + 1) - first);
    const int x0 = (tile % P.tiles_x) * kTX;
    const int y0 = (tile / P.tiles_x) * TC;
    const int nplanes = zb - za + 2;            // planes za-1 .. zb
    const int cols = min(kTX, P.nx - x0);       // columns of the tile in the grid
    const int niter = nplanes + (kLag - 1);     // the box's last iteration unpacks nothing
    if (warp == kWarps) {
      // ---------------------------------------------------------- producer
      RingPos<kRaw> post;  // of the next plane to post
      post = raw;
      int posted = 0;
      // copies plane j into its raw slot, once the slot's earlier plane is unpacked
      auto post_plane = [&](int j) {
        if (!wait(&S.empty[post.s], post.ph ^ 1)) return false;
        const int z = wrap1(za - 1 + j, P.nz, PERIODIC);
        if (TMA) {
          if (lane == 0 && !(STARVED && j == 1)) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(&S.full[post.s], (uint32_t)sizeof(S.raw[0]));
            tma_load_3d(&S.raw[post.s][0][0], &P.map_row, x0, wrap1(y0 - 1, P.ny, PERIODIC), z, &S.full[post.s]);
            tma_load_3d(&S.raw[post.s][1][0], &P.map_main, x0, y0, z, &S.full[post.s]);
            tma_load_3d(&S.raw[post.s][TC + 1][0], &P.map_row, x0, wrap1(y0 + TC, P.ny, PERIODIC), z,
                        &S.full[post.s]);
          }
        } else {
          const int r = lane;  // lane r copies row r
          int y = y0 - 1 + r;
          bool in = r < TC + 2 && y <= P.ny && z >= 0 && z < P.nz;
          if (PERIODIC) y = y < 0 ? P.ny - 1 : y >= P.ny ? 0 : y;
          else in = in && y >= 0 && y < P.ny;
          RowCopy cp;
          if (in) {
            cp.plan(S.raw[post.s][r], P.src + (z * plane + y * pitch + x0), cols, P.src, P.src + P.nz * plane);
            fence_proxy_async_smem();
          }
          if (r < TC + 2) S.shift[post.s][r] = cp.shift;
          // rows outside the grid are zeros (those below a ragged tile are not read)
          unsigned int out = __ballot_sync(0xffffffffu, r < TC + 2 && !in);
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
        ++posted;
        return true;
      };
      // the columns beside the tile: one value per lane (the box's corner
      // rows, TC + 2 per side: a second one on the first lanes)
      constexpr int HR = BOX ? TC + 2 : TC, HN = (2 * HR + 31) / 32, H0 = BOX ? 0 : 1;
      int hrow[HN], hcol[HN];
      int64_t hoff[HN];
      bool hin[HN];
#pragma unroll
      for (int q = 0; q < HN; ++q) {
        const int k = lane + 32 * q, side = k / HR;
        hrow[q] = k < 2 * HR ? H0 + k % HR : -1;
        // (right of the last column: column 64 of the tile, or of a ragged one its first beyond the grid)
        hcol[q] = side ? (TMA ? kTX : cols) + 2 : 1;
        int hx = side ? x0 + (TMA ? kTX : cols) : x0 - 1, hy = y0 - 1 + hrow[q];
        hin[q] = hrow[q] >= 0;
        if (PERIODIC) {
          hx = wrapn(hx, P.nx);
          hy = wrapn(hy, P.ny);
        } else {
          hin[q] = hin[q] && hx >= 0 && hx < P.nx && hy >= 0 && hy < P.ny;
        }
        hoff[q] = hy * pitch + hx;
      }
      auto halo = [&](int j, double (&h)[HN]) {
        const int z = wrap1(za - 1 + j, P.nz, PERIODIC);
        const bool zin = z >= 0 && z < P.nz;
#pragma unroll
        for (int q = 0; q < HN; ++q) h[q] = zin && hin[q] ? __ldcg(P.src + z * plane + hoff[q]) : 0.0;
      };
      // a wait that gave up: the copies already posted land (bounded) before the warp leaves
      auto leave = [&](int j) {
        RingPos<kRaw> q = raw;
        for (int k = j; k < posted; ++k, q.next()) mbar_wait_bounded(&S.full[q.s], q.ph, kWaitNs);
      };
      double h[HN], hn[HN];
      halo(0, h);
      while (posted < nplanes && posted < kRaw)
        if (!post_plane(posted)) return leave(0);
      for (int j = 0; j < nplanes; ++j) {
        if (j + 1 < nplanes) halo(j + 1, hn);
        if (!wait(&S.conv[u1], ph1)) return leave(j);
        Plane<TC>& u = S.u[con().s];
#pragma unroll
        for (int q = 0; q < HN; ++q)
          if (hrow[q] >= 0) put(&u.m[hrow[q]][hcol[q]], &u.e[hrow[q]][hcol[q]], BOX && HEAT ? wide_twos(wide_unpack(h[q])) : wide_unpack(h[q]));
        if (!wait(&S.full[raw.s], raw.ph)) return leave(j);
        WideVal v[2];
        unpack_row<TMA, TC + 2, BOX && HEAT>(S.raw[raw.s], S.shift[raw.s], u, 0, lane, cols, v);
        unpack_row<TMA, TC + 2, BOX && HEAT>(S.raw[raw.s], S.shift[raw.s], u, TC + 1, lane, cols, v);
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&S.empty[raw.s]);
          mbar_arrive(&S.conv[con().s]);
        }
#pragma unroll
        for (int q = 0; q < HN; ++q) h[q] = hn[q];
        next();
        // (after this plane's share of the unpacking, which the consumers wait for)
        if (posted < nplanes && !post_plane(posted)) return leave(j + 1);
      }
      continue;
    }
    // ------------------------------------------------------------ consumers
    const int row0 = 1 + warp * R;  // the warp's first row in the planes
    const int xa = x0 + 2 * lane;
    const int rows = xa < P.nx ? min(R, P.ny - (y0 + warp * R)) : 0;  // rows that the lane stores
    double* out = P.dst + za * plane + (y0 + warp * R) * pitch + xa;
    const int c = 2 + 2 * lane;
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
    for (int j = 0; j < niter; ++j) {
      WideVal zp[R][2];  // the star's values of plane g
      if (!wait(&S.conv[u1], ph1)) return;
      if (j < nplanes) {
        if (!wait(&S.full[raw.s], raw.ph)) return;
#pragma unroll
        for (int r = 0; r < R; ++r) unpack_row<TMA, TC + 2, BOX && HEAT>(S.raw[raw.s], S.shift[raw.s], S.u[con().s], row0 + r, lane, cols, zp[r]);
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&S.empty[raw.s]);
          mbar_arrive(&S.conv[con().s]);
        }
      }
      if (j >= 1 + kLag) {
        const Plane<TC>& um = S.u[BOX ? u3 : u2];
        const Plane<TC>& u0 = S.u[BOX ? u2 : u1];
        const Plane<TC>& up = S.u[BOX ? u1 : con().s];
        // the integer form takes every cell that is stored (the others may hold
        // anything, and one CTA that calls chain_cells for them delays the rest)
        bool all = true, zeros = true;  // (zeros: there may be nothing else)
        auto covers = [&](bool ok, int r, int i) {
          return ok || r >= rows || (!TMA && i == 1 && xa + 1 >= P.nx);
        };
        if constexpr (!BOX) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int row = row0 + r;
            WideVal zm[2], n[2], s[2], x[4];
            get_pair(&um.m[row][c], &um.e[row][c], zm[0], zm[1]);
            get_pair(&u0.m[row - 1][c], &u0.e[row - 1][c], n[0], n[1]);
            get_row<TC>(u0, row, c, x);
            get_pair(&u0.m[row + 1][c], &u0.e[row + 1][c], s[0], s[1]);
            double v[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const WideVal u[7] = {zm[i], n[i], x[i], x[i + 1], x[i + 2], s[i], zp[r][i]};
              bool ok;
              if constexpr (HEAT) v[i] = wide_sum_heat<7>(u, P.wide, ok);
              else v[i] = wide_sum<7>(u, P.wide, ok);
              all = all && covers(ok, r, i);
            }
            store(r, v[0], v[1]);
          }
        } else if constexpr (HEAT) {
          // equal weights, the lane's rows and two columns as one block: each value is
          // aligned once for all cells, and rows (mid: their common columns) share their
          // partial sums.  Exponents first: a block's values would not fit the registers.
          int own[R][2];
#pragma unroll
          for (int r = 0; r < R; ++r) own[r][0] = own[r][1] = 0;
#pragma unroll 1
          for (int p = 0; p < 3; ++p) {
            const Plane<TC>& u = p == 0 ? um : p == 1 ? u0 : up;
#pragma unroll
            for (int q = 0; q < R + 2; ++q) {  // the block's row: read by cells q-2 .. q
              const int* er = &u.e[row0 - 1 + q][c];
              const int2 m = *reinterpret_cast<const int2*>(er);
              const int mid = max(m.x, m.y), h0 = max(mid, er[-1]), h1 = max(mid, er[2]);
#pragma unroll
              for (int r = 0; r < R; ++r)
                if (q - 2 <= r && r <= q) {
                  own[r][0] = max(own[r][0], h0);
                  own[r][1] = max(own[r][1], h1);
                }
            }
          }
          // (what is not stored may hold anything)
          int E = own[0][0], least = own[0][0];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (r > 0 && r >= rows) own[r][0] = own[0][0];
            if ((!TMA && xa + 1 >= P.nx) || (r > 0 && r >= rows)) own[r][1] = own[0][0];
            E = max(E, max(own[r][0], own[r][1]));
            least = min(least, min(own[r][0], own[r][1]));
          }
          E |= 3;
          least |= 3;
          zeros = E == 3;
          // Where cells differ in E (a field passes a power of 16), no bit is cut as long as all
          // values are within the 2^9 that the integers have room for: the sums are exact then,
          // and those of each cell's own alignment follow.  Else the warp takes own_cells.
          all = wide_covers(E, P.equal);
          if (all && E != least) {
            int low = 0x7fffffff;
#pragma unroll 1
            for (int p = 0; p < 3; ++p) {
              const Plane<TC>& u = p == 0 ? um : p == 1 ? u0 : up;
#pragma unroll
              for (int q = 0; q < R + 2; ++q)
#pragma unroll
                for (int x = -1; x < 3; ++x) low = min(low, u.e[row0 - 1 + q][c + x]);
            }
            all = wide_covers(least, P.equal) && low + 9 >= E;
          }
          const bool fits = __all_sync(0xffffffffu, all || rows <= 0);
          all = rows <= 0 || fits;
          if (fits) {
            WideSum sum[R][2], both[2];  // both: of the rows that all cells read
            // (two values fit 64 bits: by pairs, side by side or one below the other)
            auto part = [&](const WideVal& x, const WideVal& y) {
              return WideSum(wide_align(x, E - x.e) + wide_align(y, E - y.e));
            };
#pragma unroll 1
            for (int p = 0; p < 3; ++p) {
              const Plane<TC>& u = p == 0 ? um : p == 1 ? u0 : up;
              auto one = [&](int q, WideSum (&to)[2]) {
                WideVal v[4];
                get_row<TC>(u, row0 - 1 + q, c, v);
                const WideSum mid = part(v[1], v[2]);
                to[0] += mid + wide_part(v[0], E);
                to[1] += mid + wide_part(v[3], E);
              };
              one(R == 2 ? 0 : 2, R == 2 ? sum[0] : both);
              if constexpr (R == 2) one(3, sum[R - 1]);
              WideVal v[4], w[4];
              get_row<TC>(u, row0 + R - 2, c, v);
              get_row<TC>(u, row0 + R - 1, c, w);
              const WideSum mid = part(v[1], w[1]) + part(v[2], w[2]);
              both[0] += mid + part(v[0], w[0]);
              both[1] += mid + part(v[3], w[3]);
            }
            int Ec[R][2];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                sum[r][i] += both[i];
                Ec[r][i] = E;
                if (E != least) {
                  Ec[r][i] = own[r][i] | 3;
                  sum[r][i].shift(E - Ec[r][i]);
                }
              }
#pragma unroll
            for (int r = 0; r < R; ++r)
              store(r, wide_equal_double(sum[r][0], Ec[r][0], P.equal), wide_equal_double(sum[r][1], Ec[r][1], P.equal));
          }
        } else {
          // row by row; the largest exponents first, then the sums: the 36 values of
          // a pair would not fit the registers, so their rows are read twice
          const Plane<TC>* const pl[3] = {&um, &u0, &up};
#pragma unroll 1
          for (int r = 0; r < R; ++r) {
            int E[2] = {-0x7fffffff, -0x7fffffff};
#pragma unroll
            for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
              for (int dy = -1; dy <= 1; ++dy) {
                const int* er = &pl[dz + 1]->e[row0 + r + dy][c];
                const int2 m = *reinterpret_cast<const int2*>(er);
                const int e[4] = {er[-1], m.x, m.y, er[2]};
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                  for (int dx = -1; dx <= 1; ++dx)
                    E[i] = max(E[i], e[1 + i + dx] + P.wide.ex[tap_at<true>(dz, dy, dx)]);
              }
            WideAcc acc[2];
#pragma unroll
            for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
              for (int dy = -1; dy <= 1; ++dy) {
                WideVal v[4];
                get_row<TC>(*pl[dz + 1], row0 + r + dy, c, v);
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                  for (int dx = -1; dx <= 1; ++dx)
                    acc[i].add(v[1 + i + dx], tap_at<true>(dz, dy, dx),
                               E[i] - v[1 + i + dx].e - P.wide.ex[tap_at<true>(dz, dy, dx)], P.wide);
              }
            all = all && covers(wide_covers(E[0], P.wide), r, 0) && covers(wide_covers(E[1], P.wide), r, 1);
            store(r, acc[0].get(E[0], P.wide), acc[1].get(E[1], P.wide));
          }
        }
        if (!all && (!zeros || !zero_cells<BOX, TC>(um, u0, up, row0, rows, min(2, P.nx - xa), c, out, P.nx))) {
          if constexpr (BOX && HEAT) own_cells<TC>(um, u0, up, row0, rows, min(2, P.nx - xa), c, P.wide, P.wdev, out, P.nx);
          else chain_cells<BOX, TC>(um, u0, up, row0, rows, min(2, P.nx - xa), c, P.wide, P.wdev, out, P.nx);
        }
        __syncwarp();
        out += plane;
      }
      if (j < nplanes) next();  // (the box's last iteration takes no new plane)
    }
  }
}

bool encode_3d(CUtensorMap* map, const double* base, const Geom& g, int box_y) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
  cuuint64_t strides[2] = {(cuuint64_t)g.nx * sizeof(double), (cuuint64_t)g.nx * g.ny * sizeof(double)};
  cuuint32_t box[3] = {(cuuint32_t)kTX, (cuuint32_t)box_y, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, const_cast<double*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool BOX, bool HEAT, bool PERIODIC, bool TMA, int TC, bool STARVED = false>
cudaError_t launch_t(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                     int* status, int sms, cudaStream_t stream, bool chained, unsigned long long wait_ns = 0) {
  auto kern = k_wide3d<BOX, HEAT, PERIODIC, TMA, TC, STARVED>;
  constexpr size_t bytes = sizeof(Smem<BOX, TMA, TC>);
  static std::atomic<int> cache[kMaxDeviceOrdinals];
  const int occ = cached_per_device(cache, [kern] {
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads<TC>(), bytes) != cudaSuccess)
      n = 0;
    return n;
  });
  if (occ < 1) return cudaErrorInvalidConfiguration;
  Params P;
  if (TMA && (!encode_3d(&P.map_row, src, g, 1) || !encode_3d(&P.map_main, src, g, TC))) return cudaErrorInvalidValue;
  P.src = src;
  P.dst = dst;
  P.nz = g.nz;
  P.ny = g.ny;
  P.nx = g.nx;
  P.tiles_x = (g.nx + kTX - 1) / kTX;
  P.tiles_y = (g.ny + TC - 1) / TC;
  P.work = (long long)P.tiles_x * P.tiles_y * g.nz;
  P.vec = g.nx % 2 == 0 && ((uintptr_t)dst & 15) == 0;
  P.status = status;
  P.wait_ns = wait_ns;
  P.wdev = wdev;
  P.wide = wide;
  P.equal = wide;
  long long grid = (long long)sms * occ;
  if (grid > P.work) grid = P.work;
  if (const cudaError_t e = launch_step(kern, (unsigned)grid, threads<TC>(), bytes, stream, chained, P)) return e;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <bool BOX, bool HEAT, bool PERIODIC>
cudaError_t launch_p(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                     int* status, int sms, cudaStream_t stream, bool tma, int tile_y, bool chained) {
  const bool low = tile_y == 8;
  if (tma && tile_y == 32) return launch_t<BOX, HEAT, PERIODIC, true, 32>(g, wide, wdev, src, dst, status, sms, stream, chained);
  if (tma)
    return low ? launch_t<BOX, HEAT, PERIODIC, true, 8>(g, wide, wdev, src, dst, status, sms, stream, chained)
               : launch_t<BOX, HEAT, PERIODIC, true, 16>(g, wide, wdev, src, dst, status, sms, stream, chained);
  return low ? launch_t<BOX, HEAT, PERIODIC, false, 8>(g, wide, wdev, src, dst, status, sms, stream, chained)
             : launch_t<BOX, HEAT, PERIODIC, false, 16>(g, wide, wdev, src, dst, status, sms, stream, chained);
}

}  // namespace

cudaError_t launch_wide3d(Shape shape, int boundary, const Geom& g, const WideTaps& wide, const double* wdev,
                          const double* src, double* dst, int* status, int sms, cudaStream_t stream, int tile_y,
                          bool tma, bool chained) {
  const bool per = boundary == kPeriodic;
  if (shape == Shape::kBox) {
    if (wide.n != 27) return cudaErrorInvalidValue;
    if (wide.equal)
      return per ? launch_p<true, true, true>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained)
                 : launch_p<true, true, false>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained);
    return per ? launch_p<true, false, true>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained)
               : launch_p<true, false, false>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained);
  }
  if (wide.n != 7) return cudaErrorInvalidValue;
  if (wide.heat)
    return per ? launch_p<false, true, true>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained)
               : launch_p<false, true, false>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained);
  return per ? launch_p<false, false, true>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained)
             : launch_p<false, false, false>(g, wide, wdev, src, dst, status, sms, stream, tma, tile_y, chained);
}

cudaError_t launch_wide3d_starved(const Geom& g, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                                  int* status, int sms, cudaStream_t stream, unsigned long long wait_ns) {
  return launch_t<false, true, true, true, 16, true>(g, wide, wdev, src, dst, status, sms, stream, false, wait_ns);
}

}  // namespace gbst
