// widestream.cuh -- what the streaming kernels of the integer form (wide3d.cu,
// wide2d.cu) share: unpacked values in shared memory, the bulk copy of a tile's
// row from any alignment, ring positions.
#pragma once

#include "internal.h"
#include "ptx.cuh"
#include "wide.cuh"

namespace gbst {

constexpr int kWTX = 64;            // tile columns: two per lane
constexpr int kWCol = kWTX + 4;     // unpacked row: columns x0-2 .. x0+65 (the pair (x0, x0+1) on 16 bytes)
constexpr int kWRaw = 3;            // raw planes (tiles) in flight
constexpr int kWWarps = 8;          // consumer warps; one producer warp more
constexpr int kWThreads = (kWWarps + 1) * 32;

// A raw row: the tile's 64 columns, or (bulk copies) up to one element more on
// either side.
template <bool TMA>
constexpr int raw_col() { return TMA ? kWTX : kWTX + 2; }

// ROWS rows of unpacked values.
template <int ROWS>
struct __align__(16) WidePlane {
  long long m[ROWS][kWCol];
  int e[ROWS][kWCol];
};

__device__ __forceinline__ int wrapn(int c, int n) {
  const int m = c % n;
  return m < 0 ? m + n : m;
}
__device__ __forceinline__ int wrap1(int c, int n, bool periodic) {  // -n <= c < 2 n
  return !periodic ? c : c < 0 ? c + n : c >= n ? c - n : c;
}

// Bulk copy global -> shared (both 16-byte aligned, bytes a multiple of 16).
__device__ __forceinline__ void bulk_load(double* dst, const double* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// One raw row of `n` columns whose first is at `row`, by a bulk copy from the
// 16-byte boundary at or before it to the one at or after its end, within the
// grid [src, end); the grid's first or last element, when it has no whole 16
// bytes, by itself.  The row's first column lands at dst[shift].
struct RowCopy {
  uint32_t bytes = 0;  // of the bulk copy (0: none)
  const double* from = nullptr;
  int to = 0;     // its first element in the raw row
  int shift = 0;  // 0 or 1
  __device__ __forceinline__ void plan(double* dst, const double* row, int n, const double* src, const double* end) {
    shift = (int)(((uintptr_t)row >> 3) & 1);
    from = row - shift;
    to = 0;
    if (from < src) {  // the grid starts half-way through 16 bytes
      from += 2;
      to = 2;
      dst[1] = __ldcg(row);
    }
    int k1 = (shift + n + 1) & ~1;   // one past the last element copied
    if (from + (k1 - to) > end) {  // the grid ends half-way through 16 bytes
      k1 -= 2;
      dst[shift + n - 1] = __ldcg(row + n - 1);
    }
    bytes = k1 > to ? (uint32_t)(k1 - to) * 8 : 0;
  }
};

__device__ __forceinline__ void put(long long* m, int* e, const WideVal& u) {
  *m = (long long)(((unsigned long long)(unsigned int)u.hi << 32) | u.lo);
  *e = u.e;
}
__device__ __forceinline__ WideVal get(const long long* m, const int* e) {
  const long long v = *m;
  return {(int)(v >> 32), (unsigned int)v, *e};
}
__device__ __forceinline__ void get_pair(const long long* m, const int* e, WideVal& a, WideVal& b) {
  const int4 v = *reinterpret_cast<const int4*>(m);
  const int2 x = *reinterpret_cast<const int2*>(e);
  a = {v.y, (unsigned int)v.x, x.x};
  b = {v.w, (unsigned int)v.z, x.y};
}

// Unpacks row `row` of a raw plane (two columns per lane; those at or beyond
// column `cols` of the tile are the producer's or nobody's; TWOS: in two's complement).
template <bool TMA, int ROWS, bool TWOS = false>
__device__ __forceinline__ void unpack_row(const double (&raw)[ROWS][raw_col<TMA>()], const int (&shift)[ROWS],
                                           WidePlane<ROWS>& u, int row, int lane, int cols, WideVal (&v)[2]) {
  double2 p;
  if (TMA) {
    p = *reinterpret_cast<const double2*>(&raw[row][2 * lane]);
  } else {
    const double* r = &raw[row][2 * lane + shift[row]];
    p = make_double2(r[0], r[1]);
  }
  v[0] = TWOS ? wide_twos(wide_unpack(p.x)) : wide_unpack(p.x);
  v[1] = TWOS ? wide_twos(wide_unpack(p.y)) : wide_unpack(p.y);
  if (TMA || 2 * lane + 1 < cols) {
    *reinterpret_cast<int4*>(&u.m[row][2 + 2 * lane]) = make_int4((int)v[0].lo, v[0].hi, (int)v[1].lo, v[1].hi);
    *reinterpret_cast<int2*>(&u.e[row][2 + 2 * lane]) = make_int2(v[0].e, v[1].e);
  } else if (2 * lane < cols) {
    put(&u.m[row][2 + 2 * lane], &u.e[row][2 + 2 * lane], v[0]);
  }
}

// Whether rows row0 .. row0+N-1 of a plane are zeros in column c (cols = 2: and c + 1)
// and RAD columns on either side.
template <int N, int RAD, int ROWS>
__device__ __forceinline__ bool zero_rows(const WidePlane<ROWS>& u, int row0, int c, int cols) {
  const unsigned int second = cols == 2 ? ~0u : 0u;
  unsigned int any = 0;
#pragma unroll
  for (int r = 0; r < N; ++r) {
    const int row = row0 + r;
    WideVal a, b;
    get_pair(&u.m[row][c], &u.e[row][c], a, b);
    any |= wide_nonzero(a) | (RAD == 0 ? wide_nonzero(b) & second : wide_nonzero(b));
    if constexpr (RAD == 1) {
      any |= wide_nonzero(get(&u.m[row][c - 1], &u.e[row][c - 1]));
      any |= wide_nonzero(get(&u.m[row][c + 2], &u.e[row][c + 2])) & second;
    }
    if constexpr (RAD == 2) {
      get_pair(&u.m[row][c - 2], &u.e[row][c - 2], a, b);
      any |= wide_nonzero(a) | wide_nonzero(b);
      get_pair(&u.m[row][c + 2], &u.e[row][c + 2], a, b);
      any |= wide_nonzero(a) | (wide_nonzero(b) & second);
    }
  }
  return any == 0;
}

// Zeros for the pair's first `cols` columns of `rows` rows.
__device__ __forceinline__ void put_zeros(double* out, int rows, int cols, int64_t pitch) {
  for (int r = 0; r < rows; ++r, out += pitch) {
    out[0] = 0.0;
    if (cols > 1) out[1] = 0.0;
  }
}

// A slot and phase that advance plane by plane.
template <int N>
struct RingPos {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next() {
    if (++s == N) {
      s = 0;
      ph ^= 1;
    }
  }
};

// Step after step of a run, each of a few microseconds: a step's CTAs are launched,
// and set up their barriers, while the step before still runs (programmatic
// dependent launch); step_begins then waits until that one is complete and its
// results are visible.  The next step's CTAs may come up from here on: not
// earlier, so that no more than two steps are ever in flight.  (The kernels read
// the grids past L1, which may hold lines from two steps ago.)
__device__ __forceinline__ void step_begins() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("fence.proxy.async;" ::: "memory");  // the copies are of the async proxy
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launches a step's kernel.  chained: what the stream holds last is the step
// before of the same run (any other launch takes the stream's plain order).
template <class Kernel, class P>
cudaError_t launch_step(Kernel kern, unsigned int grid, int threads, size_t smem, cudaStream_t stream, bool chained, const P& p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace gbst
