// widesteps.cu -- many steps of one or many 2D 5-point grids (each its own weights and
// step count T) in ONE persistent cooperative launch, with the weighted sum in the
// integer form (wide.cuh).
//
// Every grid is cut into tiles of 64 x 16 cells, listed grid by grid, largest T
// first, so the tiles still active at step t are a prefix of the list; step t gives
// every CTA an equal contiguous range of it.  A tile goes through a CTA as in
// wide2d.cu: its raw rows arrive by bulk copies (any size and alignment), eight
// consumer warps and the producer warp unpack them into a ring of three planes, and
// the consumers compute the tile before while the next one lands.  What a consumer
// needs to know of a tile the producer leaves beside it (Desc).
//
// Between two steps a CTA waits only for those that own its tiles' neighbours: the
// consumers arrive on `done` after the last tile of a step, the producer publishes the
// CTA's step count and reads the neighbours' before it copies the next step's first
// rows.  Its writers' fences order their stores with other CTAs' bulk copies (the
// async proxy).  Every wait is bounded by wall time.
//
// Grids with odd T have their result copied back from the partner buffer at the end.
#include <algorithm>

#include "internal.h"
#include "ptx.cuh"
#include "taps.cuh"
#include "wide.cuh"
#include "widestream.cuh"

namespace gbst {
namespace {

constexpr int kTX = kWTX, kRaw = kWRaw, kWarps = kWWarps, kThreads = kWThreads;
constexpr int kTC = 16, kRows = kTC + 2;
constexpr int kR = kTC / kWarps;  // rows of a consumer warp
using Plane = WidePlane<kRows>;
using Taps = WideTapsOf<5>;

// A tile as the consumers see it; last: of this CTA's tiles of the step; stop: no tile.
struct Desc {
  double* out;  // its first cell
  int pitch;    // nx
  int rows, cols;
  int vec, last, stop, item;
  Taps wide;
};
constexpr int kTapWords = sizeof(Taps) / 4;
static_assert(sizeof(Taps) % 4 == 0 && kTapWords <= 32, "a warp copies the taps at once");
// A tile's Desc is read until it is computed, an iteration after its raw slot is
// given back: two rounds of raw slots cover that.
constexpr int kDesc = 2 * kRaw;

// A walk over the tiles of a range, with what it needs of their item at hand.
struct Walk {
  const WideStepItem* it;
  int k, x0, y0, nx, ny, vec;  // k: tiles of the item left
  const double* src;
  double* dst;
  __device__ __forceinline__ void enter(const WideStepItem* p, int skip, int odd) {
    it = p;
    nx = p->nx;
    ny = p->ny;
    vec = p->vec;
    k = p->ntiles - skip;
    x0 = skip / p->tiles_y * kTX;
    y0 = skip % p->tiles_y * kTC;
    src = odd ? p->b : p->a;
    dst = odd ? p->a : p->b;
  }
  __device__ __forceinline__ void next(int odd) {
    if (--k == 0) return enter(it + 1, 0, odd);
    y0 += kTC;
    if (y0 >= ny) {
      y0 = 0;
      x0 += kTX;
    }
  }
};

// A CTA's range of the active tiles (the producer's; kept here while the active items
// stay the same): its ends, its first tile, the CTAs that it waits for.
struct Range {
  int first, end;
  int ca[3], cb[3];
  Walk start;
};

struct __align__(128) Smem {
  double raw[kRaw][kRows][raw_col<false>()];
  int shift[kRaw][kRows];
  Plane u[kRaw];
  Desc desc[kDesc];
  Range range;
  uint64_t full[kRaw];   // raw tile has landed
  uint64_t empty[kRaw];  // raw tile is unpacked: 8 consumer warps, the producer
  uint64_t conv[kRaw];   // tile is unpacked: the same 9 arrivals
  uint64_t done;         // the step's tiles are stored: 8 consumer warps
};

// A lane's cells where all that they read are zeros (false: they are not).
__device__ __noinline__ bool zero_cells(const Plane& u, int row0, int rows, int cols, int c0, double* out, int pitch) {
  if (!zero_rows<kR, 1>(u, row0, c0, cols) || !zero_rows<1, 0>(u, row0 - 1, c0, cols) ||
      !zero_rows<1, 0>(u, row0 + kR, c0, cols))
    return false;
  put_zeros(out, rows, cols, pitch);
  return true;
}

// The cells of a lane that the integer form does not take: zeros, or by the FMA chain.
// Out of line: rarely run.
__device__ __noinline__ void chain_cells(const Plane& u, int row0, int rows, int cols, int c0, const Taps& T,
                                         const double* w, double* out, int pitch) {
  for (int r = 0; r < rows; ++r)
    for (int i = 0; i < cols; ++i) {
      const int row = row0 + r, c = c0 + i;
      const WideVal x[5] = {get(&u.m[row - 1][c], &u.e[row - 1][c]), get(&u.m[row][c - 1], &u.e[row][c - 1]),
                            get(&u.m[row][c], &u.e[row][c]), get(&u.m[row][c + 1], &u.e[row][c + 1]),
                            get(&u.m[row + 1][c], &u.e[row + 1][c])};
      int E = -0x7fffffff;
      double v[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        E = max(E, x[k].e + T.ex[k]);
        v[k] = wide_repack(x[k]);
      }
      if (wide_zeros<5>(x)) out[(int64_t)r * pitch + i] = 0.0;
      else if (!wide_covers(E, T)) out[(int64_t)r * pitch + i] = wide_chain(v, w, 5);
    }
}

constexpr int kProgressStride = kProgressWords / kWideStepCtas;  // half a line for each CTA's word

// Whether all lanes' waits ended well; what each of them has acquired holds for all from
// here on (the vote alone orders no memory).
__device__ __forceinline__ bool joined(bool ok) {
  ok = __all_sync(0xffffffffu, ok);
  __syncwarp();
  return ok;
}

// Waits until CTAs first[k]..last[k] (k < 3) have done `steps` steps (false: gave up:
// the limit is on the time in which none of a lane's makes a step).  All 32 lanes; a
// lane's loads are in flight together.
__device__ bool wait_progress(const unsigned int* progress, const int (&first)[3], const int (&last)[3],
                              unsigned int steps, long long limit_ns, int* status) {
  constexpr int kLoads = 4;
  const int n0 = max(0, last[0] - first[0] + 1), n1 = max(0, last[1] - first[1] + 1), n2 = max(0, last[2] - first[2] + 1);
  const int n = n0 + n1 + n2;
  bool ok = true;
  // the few words of most CTAs by acquire loads; many by relaxed ones in flight
  // together, and a fence
  if (n <= 32) {
    const int k = (int)(threadIdx.x & 31);
    const int c = k < n0 ? first[0] + k : k < n0 + n1 ? first[1] + (k - n0) : first[2] + (k - n0 - n1);
    unsigned int was = 0;
    unsigned long long t0 = 0;
    for (unsigned int spin = 0; k < n; ++spin) {
      unsigned int seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(progress + c * kProgressStride) : "memory");
      if (seen >= steps) break;
      if ((spin & 63) == 63) {
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0 || seen != was) t0 = now;
        was = seen;
        if (*(volatile int*)status != 0) ok = false;
        else if ((long long)(now - t0) > limit_ns) {
          atomicCAS(status, 0, -5 /* STENCIL_ERR_TIMEOUT */);
          ok = false;
        }
        if (!ok) break;
      }
    }
    return joined(ok);
  }
  for (int k0 = (int)(threadIdx.x & 31); ok && k0 < n; k0 += 32 * kLoads) {
    const unsigned int* p[kLoads];
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const int k = k0 + 32 * q;
      const int c = k < n0 ? first[0] + k : k < n0 + n1 ? first[1] + (k - n0) : first[2] + (k - n0 - n1);
      p[q] = k < n ? progress + c * kProgressStride : nullptr;
    }
    unsigned int sum = 0;
    unsigned long long t0 = 0;
    for (unsigned int spin = 0;; ++spin) {
      unsigned int seen[kLoads];
#pragma unroll
      for (int q = 0; q < kLoads; ++q) {
        seen[q] = steps;
        if (p[q]) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen[q]) : "l"(p[q]) : "memory");
      }
      bool all = true;
      unsigned int now_sum = 0;
#pragma unroll
      for (int q = 0; q < kLoads; ++q) {
        all = all && seen[q] >= steps;
        now_sum += seen[q];
      }
      if (all) break;
      if ((spin & 63) == 63) {
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0 || now_sum != sum) t0 = now;
        sum = now_sum;
        if (*(volatile int*)status != 0) ok = false;
        else if ((long long)(now - t0) > limit_ns) {
          atomicCAS(status, 0, -5 /* STENCIL_ERR_TIMEOUT */);
          ok = false;
        }
        if (!ok) break;
      }
    }
  }
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  return joined(ok);
}

// The CTA whose range of `tiles` tiles over n CTAs holds tile j.
__device__ __forceinline__ int tile_owner(int j, int tiles, int n) { return (int)((((long long)j + 1) * n - 1) / tiles); }

template <bool HEAT, bool PERIODIC>
__global__ void __launch_bounds__(kThreads, 3) k_wide_steps(const __grid_constant__ WideStepsLaunch L) {
  constexpr unsigned long long kWaitNs = (unsigned long long)kSpinLimitNs;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Smem& S = *reinterpret_cast<Smem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const WideStepItem* const items = L.items ? L.items : &L.one;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRaw; ++s) {
      mbar_init(&S.full[s], 1);
      mbar_init(&S.empty[s], kWarps + 1);
      mbar_init(&S.conv[s], kWarps + 1);
    }
    mbar_init(&S.done, kWarps);
    fence_mbar_init();
  }
  __syncthreads();
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (mbar_wait_bounded(bar, parity, kWaitNs)) return true;
    atomicCAS(L.status, 0, -5 /* STENCIL_ERR_TIMEOUT */);
    return false;
  };
  RingPos<kRaw> pos;     // of tile g
  RingPos<kDesc> dpos;
  int u1 = kRaw - 1;     // slot of tile g-1
  uint32_t ph1 = 1;      // its phase (a fresh barrier lets a wait for phase 1 pass)
  auto next = [&] {
    u1 = pos.s;
    ph1 = pos.ph;
    pos.next();
    dpos.next();
  };
  if (warp == kWarps) {
    // ------------------------------------------------------------ producer
    RingPos<kRaw> post;  // of the next tile to post
    RingPos<kDesc> dpost;
    uint32_t done_ph = 0;
    int na = L.nitems;  // active items
    // a wait that gave up: the copies already posted land (bounded) before the warp leaves
    auto leave = [&](int n) {
      RingPos<kRaw> q = pos;
      for (int k = 0; k < n; ++k, q.next()) mbar_wait_bounded(&S.full[q.s], q.ph, kWaitNs);
    };
    int act = 0, since = 0, until = 0;  // tiles active in steps since .. until-1
    bool owed = false;  // it had tiles in the step before
    // the CTA's steps so far are stored: tells the others
    auto publish = [&](int steps) {
      if (owed) {
        if (!wait(&S.done, done_ph)) return false;
        done_ph ^= 1;
      }
      if (lane == 0 && (int)blockIdx.x != L.mute) {
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(L.progress + blockIdx.x * kProgressStride), "r"(steps)
                     : "memory");
      }
      return true;
    };
    for (int t = 0; t < L.max_T; ++t) {
      if (t >= until || t == since + 1) {  // (else as in the step before)
        const int tiles = act;  // active in the step before
        if (t >= until) {
          while (na > 0 && items[na - 1].T <= t) --na;
          since = t;
          until = items[na - 1].T;
          act = items[na - 1].tile0 + items[na - 1].ntiles;
        }
        const int first = (int)((long long)act * blockIdx.x / gridDim.x);
        const int end = (int)((long long)act * (blockIdx.x + 1) / gridDim.x);
        int pi = 0;  // the first tile's item: the last whose tiles begin at or before it
        for (int hi = na; hi - pi > 1;) {
          const int mid = (pi + hi) / 2;
          if (items[mid].tile0 <= first) pi = mid;
          else hi = mid;
        }
        Range& R = S.range;
        R.first = first;  // (the same words from every lane)
        R.end = end;
        if (first < end) R.start.enter(items + pi, first - items[pi].tile0, 0);
        // the tiles whose last step this one reads, and which read what it overwrites:
        // those beside the range in its first and last column of tiles, west of its first
        // item's and east of its last item's.  Periodic: from the column before to the
        // column after (a column's ends meet), where the range has the item's first or
        // last column all of the item.  A CTA that has no tile follows the one whose range
        // begins where its own would.
        if (t > 0) {
          int a[3] = {min(first, act - 1), 0, 0}, b[3] = {a[0], -1, -1};
          if (first < end) {
            int qi = pi;
            while (items[qi].tile0 + items[qi].ntiles < end) ++qi;
            const int l = items[pi].tile0, ly = items[pi].tiles_y, lh = l + items[pi].ntiles;
            const int hl = items[qi].tile0, hy = items[qi].tiles_y, h = hl + items[qi].ntiles - 1;
            if (PERIODIC) {
              const bool all = pi < qi || first - l < ly || h - (end - 1) < hy;
              a[0] = all ? l : first - ly;
              b[0] = all ? h : end - 1 + hy;
            } else {
              a[0] = max(l, first - 1);
              b[0] = min(h, end);
              a[1] = max(l, first - ly);
              b[1] = min(first, min(end, lh) - ly) - 1;
              a[2] = max(end, max(first, hl) + hy);
              b[2] = min(h, end - 1 + hy);
            }
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const bool some = a[k] <= b[k];
            R.ca[k] = some ? tile_owner(a[k], tiles, gridDim.x) : 0;
            R.cb[k] = some ? tile_owner(b[k], tiles, gridDim.x) : -1;
          }
        }
        __syncwarp();
      }
      if (t > 0) {
        if (!publish(t)) return;
        if (!wait_progress(L.progress, S.range.ca, S.range.cb, t, L.spin_limit, L.status)) return;
        fence_proxy_async_global();
      }
      const int odd = t & 1, first = S.range.first, end = S.range.end;
      Walk pw = S.range.start;  // of the next tile to post
      if (odd) {
        pw.src = S.range.start.dst;
        pw.dst = const_cast<double*>(S.range.start.src);
      }
      Walk hw = pw;  // of the next halo
      int posted = first;
      auto post_tile = [&] {
        if (!wait(&S.empty[post.s], post.ph ^ 1)) return false;
        const int nx = pw.nx, ny = pw.ny, x0 = pw.x0, y0 = pw.y0;
        const double* src = pw.src;
        const int r = lane;
        int y = y0 - 1 + r;
        bool in = r < kRows;
        if (PERIODIC) {
          in = in && y <= ny;
          y = y < 0 ? ny - 1 : y >= ny ? 0 : y;
        } else {
          in = in && y >= 0 && y < ny;
        }
        RowCopy cp;
        if (in) {
          cp.plan(S.raw[post.s][r], src + ((int64_t)y * nx + x0), min(kTX, nx - x0), src, src + (int64_t)ny * nx);
          fence_proxy_async_smem();
        }
        if (r < kRows) S.shift[post.s][r] = cp.shift;
        unsigned int out = __ballot_sync(0xffffffffu, r < kRows && !in);  // rows outside the grid are zeros
        while (out) {
          const int q = __ffs((int)out) - 1;
          out &= out - 1;
          S.raw[post.s][q][lane] = 0.0;
          S.raw[post.s][q][lane + 32] = 0.0;
        }
        Desc& d = S.desc[dpost.s];
        if (lane < kTapWords) reinterpret_cast<int*>(&d.wide)[lane] = reinterpret_cast<const int*>(&pw.it->wide)[lane];
        if (lane == 0) {
          d.out = pw.dst + ((int64_t)y0 * nx + x0);
          d.pitch = nx;
          d.rows = ny - y0;
          d.cols = nx - x0;
          d.vec = pw.vec;
          d.last = posted + 1 == end;
          d.stop = 0;
          d.item = (int)(pw.it - items);
        }
        const uint32_t total = __reduce_add_sync(0xffffffffu, cp.bytes);
        __syncwarp();  // the lanes' own writes come before lane 0's arrival
        if (lane == 0) mbar_arrive_expect_tx(&S.full[post.s], total);
        __syncwarp();
        if (cp.bytes) bulk_load(&S.raw[post.s][r][cp.to], cp.from, cp.bytes, &S.full[post.s]);
        post.next();
        dpost.next();
        if (++posted < end) pw.next(odd);
        return true;
      };
      // the columns beside the walk's tile: one value per lane (rows y0 .. y0+15, west and east)
      auto halo = [&] {
        const int nx = hw.nx, ny = hw.ny;
        int x = lane < kTC ? hw.x0 - 1 : min(hw.x0 + kTX, nx), y = hw.y0 + lane % kTC;
        bool in = true;
        if (PERIODIC) {
          x = x < 0 ? nx - 1 : x >= nx ? 0 : x;
          y = wrapn(y, ny);
        } else {
          in = x >= 0 && x < nx && y < ny;
        }
        return in ? __ldcg(hw.src + ((int64_t)y * nx + x)) : 0.0;
      };
      double h = first < end ? halo() : 0.0;
      while (posted < end && posted < first + kRaw)
        if (!post_tile()) return leave(posted - first);
      for (int tile = first; tile < end; ++tile) {
        double hn = 0.0;
        if (tile + 1 < end) {
          hw.next(odd);
          hn = halo();
        }
        if (!wait(&S.conv[u1], ph1)) return leave(posted - tile);
        Plane& u = S.u[pos.s];
        const int cols = min(kTX, S.desc[dpos.s].cols);
        const int hr = 1 + lane % kTC, hc = 2 + (lane < kTC ? -1 : cols);
        put(&u.m[hr][hc], &u.e[hr][hc], wide_unpack(h));
        if (!wait(&S.full[pos.s], pos.ph)) return leave(posted - tile);
        WideVal v[2];
        unpack_row<false, kRows>(S.raw[pos.s], S.shift[pos.s], u, 0, lane, cols, v);
        unpack_row<false, kRows>(S.raw[pos.s], S.shift[pos.s], u, kTC + 1, lane, cols, v);
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&S.empty[pos.s]);
          mbar_arrive(&S.conv[pos.s]);
        }
        h = hn;
        next();
        // (after this tile's share of the unpacking, which the consumers wait for)
        if (posted < end && !post_tile()) return leave(posted - tile - 1);
      }
      owed = first < end;
    }
    if (L.any_odd) {
      const int a[3] = {0, 0, 0}, b[3] = {(int)gridDim.x - 1, -1, -1};
      if (!publish(L.max_T) || !wait_progress(L.progress, a, b, L.max_T, L.spin_limit, L.status)) return;
    }
    if (!wait(&S.empty[post.s], post.ph ^ 1)) return;
    if (lane == 0) {
      S.desc[dpost.s].stop = 1;
      mbar_arrive(&S.full[post.s]);
    }
    return;
  }
  // -------------------------------------------------------------- consumers
  const int row0 = 1 + warp * kR;  // the warp's first row in the planes
  const int c = 2 + 2 * lane;
  // the warp's rows of the tile in plane u
  auto compute = [&](const Plane& u, const Desc& d) {
    const Taps T = d.wide;
    const int left = d.cols - 2 * lane;                                     // columns from the lane's first on
    const int rows = left > 0 ? min(kR, d.rows - warp * kR) : 0;  // rows that it stores
    const bool vec = d.vec && left > 1;
    const int64_t pitch = d.pitch;
    double* out = d.out + warp * kR * pitch + 2 * lane;
    auto store = [&](int r, double v0, double v1) {
      if (r >= rows) return;
      double* o = out + r * pitch;
      if (vec) {
        st_global_v2(o, v0, v1);
      } else {
        o[0] = v0;
        if (left > 1) o[1] = v1;
      }
    };
    bool all = true;  // the integer form takes every cell that is stored
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const int row = row0 + r;
      WideVal n[2], s[2], x[4];
      get_pair(&u.m[row - 1][c], &u.e[row - 1][c], n[0], n[1]);
      x[0] = get(&u.m[row][c - 1], &u.e[row][c - 1]);
      get_pair(&u.m[row][c], &u.e[row][c], x[1], x[2]);
      x[3] = get(&u.m[row][c + 2], &u.e[row][c + 2]);
      get_pair(&u.m[row + 1][c], &u.e[row + 1][c], s[0], s[1]);
      double v[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const WideVal w[5] = {n[i], x[i], x[i + 1], x[i + 2], s[i]};
        bool ok;
        if constexpr (HEAT) v[i] = wide_sum_heat<5>(w, T, ok);
        else v[i] = wide_sum<5>(w, T, ok);
        all = all && (ok || r >= rows || (i == 1 && left < 2));
      }
      store(r, v[0], v[1]);
    }
    if (!all && !zero_cells(u, row0, rows, min(2, left), c, out, d.pitch))
      chain_cells(u, row0, rows, min(2, left), c, d.wide, items[d.item].w, out, d.pitch);
    __syncwarp();
  };
  // the next tile, or the stop: a CTA that has no tile left waits for the other
  // grids' steps, each of which ends within the limit or sets the status word
  auto wait_tile = [&] {
    const unsigned long long t0 = globaltimer_ns(), most = (unsigned long long)L.max_T + 2;
    while (!mbar_wait_bounded(&S.full[pos.s], pos.ph, 1000000ull)) {
      if (*(volatile int*)L.status != 0) return false;
      if ((globaltimer_ns() - t0) / kWaitNs >= most) return wait(&S.full[pos.s], pos.ph);
    }
    return true;
  };
  bool pending = false;  // tile g-1 is unpacked and not computed
  const Desc* dp = nullptr;
  for (;;) {
    if (!wait(&S.conv[u1], ph1)) return;
    if (!wait_tile()) return;
    const Desc& d = S.desc[dpos.s];
    if (d.stop) break;
    WideVal v[2];
#pragma unroll
    for (int r = 0; r < kR; ++r)
      unpack_row<false, kRows>(S.raw[pos.s], S.shift[pos.s], S.u[pos.s], row0 + r, lane, min(kTX, d.cols), v);
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&S.empty[pos.s]);
      mbar_arrive(&S.conv[pos.s]);
    }
    if (pending) compute(S.u[u1], *dp);
    dp = &d;
    next();
    pending = !d.last;
    if (d.last) {
      if (!wait(&S.conv[u1], ph1)) return;
      compute(S.u[u1], d);
      fence_proxy_async_global();  // this thread's stores, before other CTAs' copies of them
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.done);
    }
  }
  if (L.any_odd) {
    for (int i = 0; i < L.nitems; ++i) {
      const WideStepItem& it = items[i];
      if ((it.T & 1) == 0) continue;
      const int64_t n = (int64_t)it.ny * it.nx;
      for (int64_t k = (int64_t)blockIdx.x * (kWarps * 32) + threadIdx.x; k < n; k += (int64_t)gridDim.x * (kWarps * 32))
        it.a[k] = __ldcg(it.b + k);
    }
  }
}

template <bool HEAT, bool PERIODIC>
cudaError_t launch_t(const WideStepsLaunch& L, int tiles, int sms, cudaStream_t stream) {
  auto kern = k_wide_steps<HEAT, PERIODIC>;
  static std::atomic<int> cache[kMaxDeviceOrdinals];
  const int occ = cached_per_device(cache, [kern] {
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kThreads, sizeof(Smem)) != cudaSuccess)
      n = 0;
    return n;
  });
  if (occ < 1) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min(tiles, std::min(sms * occ, kWideStepCtas)), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = sizeof(Smem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, L);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return e;
}

}  // namespace

void wide_step_item(WideStepItem& d, const BatchItemDev& it, int tile0) {
  d.a = it.a;
  d.b = it.b;
  d.ny = it.ny;
  d.nx = it.nx;
  d.T = it.T;
  d.tiles_y = (it.ny + kTC - 1) / kTC;
  d.tile0 = tile0;
  d.ntiles = d.tiles_y * ((it.nx + kTX - 1) / kTX);
  d.vec = it.nx % 2 == 0 && (((uintptr_t)it.a | (uintptr_t)it.b) & 15) == 0;
  for (int k = 0; k < 5; ++k) d.w[k] = it.w[k];
  d.wide = it.wide;
}

cudaError_t launch_wide_steps(const WideStepsLaunch& L, int tiles, int boundary, int sms, cudaStream_t stream) {
  const bool per = boundary == kPeriodic;
  if (tiles < 1 || L.max_T < 1) return cudaErrorInvalidValue;
  if (L.heat) return per ? launch_t<true, true>(L, tiles, sms, stream) : launch_t<true, false>(L, tiles, sms, stream);
  return per ? launch_t<false, true>(L, tiles, sms, stream) : launch_t<false, false>(L, tiles, sms, stream);
}

}  // namespace gbst
