// direct.cu -- the plain one-step sweep: every thread owns one (y, x) column
// of a tile and walks a chunk of planes along z, summing its taps straight
// from global memory (the L1 cache serves the neighbour reuse).  It handles
// every shape, radius and boundary and is the reference point that the
// streaming and temporal-blocking kernels are measured against.
//
// Operation: one step of u'(x) = sum_o w_o u~(x+o) (paper Sec. 2.1, Listing 1).
//
// The taps are a compile-time list and the wraps of an axis are worked out once per
// thread: a tap is one address addition and a load.  Us a step, against a list of
// offsets in the parameters with a wrap test for each: 113 x 28 x 118 star 8.3 (12.4;
// FMA chain 10.3), 27 x 242 x 31 125-point box 61 (99), 101^3 336 (656), 97^3
// star 16.4 (22.9).  The 125-point box is bound by the FP64 pipe (62 clocks a cell and
// SM: 231 us of the 336 at 101^3), the others by the integer pipes and the launch.
#include "internal.h"
#include "taps.cuh"
#include "wide.cuh"

namespace gbst {
namespace {

// The lexicographic tap list of a stencil class, at compile time.
template <int NDIM, int RAD, bool BOX>
struct Taps {
  static constexpr int kSide = 2 * RAD + 1;
  static constexpr int kN = !BOX ? 2 * NDIM * RAD + 1 : NDIM == 3 ? kSide * kSide * kSide : kSide * kSide;
  // offset of tap k along x (axis 0), y (1) or z (2)
  static __host__ __device__ constexpr int off(int k, int axis) {
    if (BOX) return axis == 0 ? k % kSide - RAD : axis == 1 ? k / kSide % kSide - RAD : NDIM == 3 ? k / (kSide * kSide) - RAD : 0;
    // star: the slowest axis's lower half, ..., the fastest axis, ..., the slowest axis's upper half
    int d = NDIM - 1;
    while (d > 0) {
      const int lo = (NDIM - 1 - d) * RAD, hi = kN - 1 - lo;
      if (k < lo + RAD) return axis == d ? k - lo - RAD : 0;
      if (k > hi - RAD) return axis == d ? k - hi + RAD : 0;
      --d;
    }
    return axis == 0 ? k - (NDIM - 1) * RAD - RAD : 0;
  }
};

// The 2 RAD + 1 positions around coordinate c of an axis of length n, as distances from
// c in elements (step: the axis's stride), and whether they are in the grid.
template <int RAD, bool PERIODIC, class Int>
struct Axis {
  Int at[2 * RAD + 1];
  bool in[2 * RAD + 1];
  __device__ __forceinline__ Axis(int c, int n, Int step) {
#pragma unroll
    for (int k = 0; k < 2 * RAD + 1; ++k) {
      int d = k - RAD;
      in[k] = true;
      if (d != 0) {
        if (PERIODIC) {
          if (n < RAD) d = ((c + d) % n + n) % n - c;  // (uniform) an axis shorter than the radius
          else d = c + d < 0 ? d + n : c + d >= n ? d - n : d;
        } else {
          in[k] = (unsigned)(c + d) < (unsigned)n;
        }
      }
      at[k] = (Int)d * step;
    }
  }
};

// Weights as kernel parameters (the constant bank).
template <int NT>
struct Weights {
  double w[NT];
};

struct DirectParams {
  const double* src;
  double* dst;
  int nz, ny, nx;
  int zper;
  const double* wdev;
};

// The thread's cells, plane by plane: body(v, cell) with the cell's NT values.
template <int NDIM, int RAD, bool BOX, bool PERIODIC, class Body>
__device__ __forceinline__ void each_cell(const DirectParams& P, const Body& body) {
  using T = Taps<NDIM, RAD, BOX>;
  constexpr int RZ = NDIM >= 3 ? RAD : 0, RY = NDIM >= 2 ? RAD : 0;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= P.nx || y >= P.ny) return;
  const int64_t plane = (int64_t)P.ny * P.nx;
  const Axis<RAD, PERIODIC, int> X(x, P.nx, 1);
  const Axis<RY, PERIODIC, int64_t> Y(y, P.ny, P.nx);
  const int z0 = blockIdx.z * P.zper, z1 = min(P.nz, z0 + P.zper);
  for (int z = z0; z < z1; ++z) {
    const Axis<RZ, PERIODIC, int64_t> Z(z, P.nz, plane);
    const int64_t cell = z * plane + (int64_t)y * P.nx + x;
    double v[T::kN];
#pragma unroll
    for (int k = 0; k < T::kN; ++k) {
      const int kx = T::off(k, 0) + RAD, ky = T::off(k, 1) + RY, kz = T::off(k, 2) + RZ;
      const double* row = P.src + cell + (Z.at[kz] + Y.at[ky]);
      v[k] = Z.in[kz] && Y.in[ky] && X.in[kx] ? __ldg(row + X.at[kx]) : 0.0;
    }
    P.dst[cell] = body(v);
  }
}

template <int NDIM, int RAD, bool BOX, bool PERIODIC>
__global__ void __launch_bounds__(256) k_direct(const __grid_constant__ DirectParams P) {
  constexpr int NT = Taps<NDIM, RAD, BOX>::kN;
  RegWeights<NT> W;  // the weights live in registers (full FP64 rate)
  W.load(P.wdev);
  each_cell<NDIM, RAD, BOX, PERIODIC>(P, [&](const double (&v)[NT]) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < NT; ++k) W.tap(acc, k, v[k], 0);
    return acc;
  });
}

// The 125-tap box: plane by plane of its taps, so that neither 125 values nor as many
// weights (in the constant bank) have to be held at once.
template <bool PERIODIC>
__global__ void __launch_bounds__(256) k_direct_box125(const __grid_constant__ DirectParams P,
                                                       const __grid_constant__ Weights<125> W) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= P.nx || y >= P.ny) return;
  const int64_t plane = (int64_t)P.ny * P.nx;
  const Axis<2, PERIODIC, int> X(x, P.nx, 1);
  const Axis<2, PERIODIC, int64_t> Y(y, P.ny, P.nx);
  const int z0 = blockIdx.z * P.zper, z1 = min(P.nz, z0 + P.zper);
  for (int z = z0; z < z1; ++z) {
    double acc = 0.0;
#pragma unroll 1
    for (int kz = 0; kz < 5; ++kz) {
      int zz = z + kz - 2;
      if (PERIODIC) zz = P.nz < 2 ? 0 : zz < 0 ? zz + P.nz : zz >= P.nz ? zz - P.nz : zz;
      const bool zin = PERIODIC || (unsigned)zz < (unsigned)P.nz;
      const double* p = P.src + (zz * plane + (int64_t)y * P.nx + x);
      double v[25];
#pragma unroll
      for (int k = 0; k < 25; ++k)
        v[k] = zin && Y.in[k / 5] && X.in[k % 5] ? __ldg(p + Y.at[k / 5] + X.at[k % 5]) : 0.0;
#pragma unroll
      for (int k = 0; k < 25; ++k) acc = fma(W.w[25 * kz + k], v[k], acc);
    }
    P.dst[z * plane + (int64_t)y * P.nx + x] = acc;
  }
}

// The same sweep with the weighted sum in the integer form (wide.cuh; HEAT: a star whose
// weights wide_sum_heat takes, a box whose weights are all equal).
template <int NDIM, int RAD, bool BOX, bool PERIODIC, bool HEAT>
__global__ void __launch_bounds__(256) k_direct_wide(const __grid_constant__ DirectParams P,
                                                     const __grid_constant__ WideTaps wide) {
  constexpr int NT = Taps<NDIM, RAD, BOX>::kN;
  each_cell<NDIM, RAD, BOX, PERIODIC>(P, [&](const double (&v)[NT]) {
    WideVal u[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) u[k] = wide_unpack(v[k]);
    bool ok;
    double r;
    if constexpr (HEAT && BOX) r = wide_sum_equal<NT>(u, wide, ok);
    else if constexpr (HEAT) r = wide_sum_heat<NT>(u, wide, ok);
    else r = wide_sum<NT>(u, wide, ok);
    if (ok) return r;
    if (wide_zeros<NT>(u)) return 0.0;
    return wide_chain(v, P.wdev, NT);
  });
}

// Index of a neighbour along one axis under each boundary mode.
//   MODE 0: Dirichlet zero -- returns false when outside [0, n)
//   MODE 1: periodic, |offset| <= n -- one conditional add or subtract
//   MODE 2: periodic, any offset -- true modulo (axes shorter than the radius)
template <int MODE>
__device__ __forceinline__ bool axis_index(int c, int n, int& out) {
  if (MODE == 0) {
    out = c;
    return (unsigned)c < (unsigned)n;
  } else if (MODE == 1) {
    out = c < 0 ? c + n : (c >= n ? c - n : c);
    return true;
  } else {
    int m = c % n;
    out = m < 0 ? m + n : m;
    return true;
  }
}

// FP32 twin of the direct sweep, for accuracy studies only (the paper's
// Table 4 compares an FP32 run of its thermal case with FP64): the same tap
// order with the weights rounded to float and float FMAs.
template <int NT, int MODE>
__global__ void __launch_bounds__(256) k_direct_f32(const float* __restrict__ src, float* __restrict__ dst,
                                                    int nz, int ny, int nx, int zper,
                                                    const __grid_constant__ TapList<NT> tp) {
  float w[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) w[k] = (float)tp.w[k];
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= nx || y >= ny) return;
  const int z0 = blockIdx.z * zper;
  const int z1 = min(nz, z0 + zper);
  for (int z = z0; z < z1; ++z) {
    float acc = 0.0f;
#pragma unroll
    for (int k = 0; k < NT; ++k) {
      int zz, yy, xx;
      bool in = axis_index<MODE>(z + tp.dz[k], nz, zz);
      in &= axis_index<MODE>(y + tp.dy[k], ny, yy);
      in &= axis_index<MODE>(x + tp.dx[k], nx, xx);
      float v = 0.0f;
      if (in) v = __ldg(src + ((int64_t)zz * ny + yy) * nx + xx);
      acc = (k == 0) ? w[0] * v : fmaf(w[k], v, acc);
    }
    dst[((int64_t)z * ny + y) * nx + x] = acc;
  }
}

// Enough blocks for every SM several times over; the rest of z is walked.
void direct_shape(const Geom& g, dim3& grid, dim3& block, int& zper) {
  zper = 1;
  if (g.ny == 1 && g.nz == 1) {
    block = dim3(256, 1, 1);
    grid = dim3((g.nx + 255) / 256, 1, 1);
  } else {
    block = dim3(32, 8, 1);
    unsigned gx = (g.nx + 31) / 32, gy = (g.ny + 7) / 8;
    int64_t tiles = (int64_t)gx * gy;
    int64_t want = 152 * 16;
    int64_t zchunks = (want + tiles - 1) / tiles;
    if (zchunks > g.nz) zchunks = g.nz;
    if (zchunks < 1) zchunks = 1;
    zper = (int)((g.nz + zchunks - 1) / zchunks);
    zchunks = (g.nz + zper - 1) / zper;
    grid = dim3(gx, gy, (unsigned)zchunks);
  }
}

template <int NT>
cudaError_t launch_nt_f32(int mode, const Geom& g, const HostTaps& ht, const float* src, float* dst,
                          cudaStream_t stream) {
  TapList<NT> tp;
  for (int k = 0; k < NT; ++k) {
    tp.w[k] = ht.w[k];
    tp.dz[k] = ht.dz[k];
    tp.dy[k] = ht.dy[k];
    tp.dx[k] = ht.dx[k];
  }
  dim3 block, grid;
  int zper;
  direct_shape(g, grid, block, zper);
  switch (mode) {
    case 0: k_direct_f32<NT, 0><<<grid, block, 0, stream>>>(src, dst, g.nz, g.ny, g.nx, zper, tp); break;
    case 1: k_direct_f32<NT, 1><<<grid, block, 0, stream>>>(src, dst, g.nz, g.ny, g.nx, zper, tp); break;
    default: k_direct_f32<NT, 2><<<grid, block, 0, stream>>>(src, dst, g.nz, g.ny, g.nx, zper, tp); break;
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <int NDIM, int RAD, bool BOX, bool PERIODIC>
cudaError_t launch_p(const Geom& g, const HostTaps& ht, const WideTaps& wide, const double* wdev, const double* src,
                     double* dst, cudaStream_t stream) {
  constexpr int NT = Taps<NDIM, RAD, BOX>::kN;
  dim3 block, grid;
  DirectParams P{src, dst, g.nz, g.ny, g.nx, 1, wdev};
  direct_shape(g, grid, block, P.zper);
  bool done = false;
  if constexpr (NDIM <= 2 || RAD == 1) {  // the classes that have the integer form
    if (wide.n) {
      done = true;
      if constexpr (BOX || RAD == 1) {
        if (BOX ? wide.equal : wide.heat) k_direct_wide<NDIM, RAD, BOX, PERIODIC, true><<<grid, block, 0, stream>>>(P, wide);
        else k_direct_wide<NDIM, RAD, BOX, PERIODIC, false><<<grid, block, 0, stream>>>(P, wide);
      } else {
        k_direct_wide<NDIM, RAD, BOX, PERIODIC, false><<<grid, block, 0, stream>>>(P, wide);
      }
    }
  }
  if (!done) {
    if constexpr (NT == 125) {
      Weights<NT> w;
      for (int k = 0; k < NT; ++k) w.w[k] = ht.w[k];
      k_direct_box125<PERIODIC><<<grid, block, 0, stream>>>(P, w);
    } else {
      k_direct<NDIM, RAD, BOX, PERIODIC><<<grid, block, 0, stream>>>(P);
    }
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

template <int NDIM, int RAD, bool BOX>
cudaError_t launch_c(int boundary, const Geom& g, const HostTaps& ht, const WideTaps& wide, const double* wdev,
                     const double* src, double* dst, cudaStream_t stream) {
  if (ht.n != Taps<NDIM, RAD, BOX>::kN) return cudaErrorInvalidValue;
  return boundary == kPeriodic ? launch_p<NDIM, RAD, BOX, true>(g, ht, wide, wdev, src, dst, stream)
                               : launch_p<NDIM, RAD, BOX, false>(g, ht, wide, wdev, src, dst, stream);
}

}  // namespace

cudaError_t launch_direct(int ndim, int radius, Shape shape, int boundary, const Geom& g,
                          const HostTaps& taps, const WideTaps& wide, const double* wdev, const double* src, double* dst,
                          cudaStream_t stream) {
  const bool box = shape == Shape::kBox;
  switch (ndim * 10 + radius) {
    case 11: return launch_c<1, 1, false>(boundary, g, taps, wide, wdev, src, dst, stream);
    case 12: return launch_c<1, 2, false>(boundary, g, taps, wide, wdev, src, dst, stream);
    case 21: return box ? launch_c<2, 1, true>(boundary, g, taps, wide, wdev, src, dst, stream)
                        : launch_c<2, 1, false>(boundary, g, taps, wide, wdev, src, dst, stream);
    case 22: return box ? launch_c<2, 2, true>(boundary, g, taps, wide, wdev, src, dst, stream)
                        : launch_c<2, 2, false>(boundary, g, taps, wide, wdev, src, dst, stream);
    case 31: return box ? launch_c<3, 1, true>(boundary, g, taps, wide, wdev, src, dst, stream)
                        : launch_c<3, 1, false>(boundary, g, taps, wide, wdev, src, dst, stream);
    case 32: return box ? launch_c<3, 2, true>(boundary, g, taps, wide, wdev, src, dst, stream)
                        : launch_c<3, 2, false>(boundary, g, taps, wide, wdev, src, dst, stream);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_direct_f32(int ndim, int radius, int boundary, const Geom& g, const HostTaps& taps,
                              const float* src, float* dst, cudaStream_t stream) {
  int mode = 0;
  if (boundary == kPeriodic) {
    bool small = g.nx < radius || (ndim >= 2 && g.ny < radius) || (ndim >= 3 && g.nz < radius);
    mode = small ? 2 : 1;
  }
  switch (taps.n) {
    case 3: return launch_nt_f32<3>(mode, g, taps, src, dst, stream);
    case 5: return launch_nt_f32<5>(mode, g, taps, src, dst, stream);
    case 7: return launch_nt_f32<7>(mode, g, taps, src, dst, stream);
    case 9: return launch_nt_f32<9>(mode, g, taps, src, dst, stream);
    case 13: return launch_nt_f32<13>(mode, g, taps, src, dst, stream);
    case 25: return launch_nt_f32<25>(mode, g, taps, src, dst, stream);
    case 27: return launch_nt_f32<27>(mode, g, taps, src, dst, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gbst
