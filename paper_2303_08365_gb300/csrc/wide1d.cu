// wide1d.cu -- 1D sweep (radius 1 or 2), up to 8 fused steps per launch, with the
// weighted sum in the integer form (wide.cuh).
//
// Operation: steps of u'(x) = sum_o w_o u~(x+o) (paper Sec. 2.1, Listing 1), blocked in
// time (Sec. 4.1).  The integer pipes bound it (112 instructions a cell and step, two thirds
// of them on the ALU pipe), where the FMA chain was bound by the FP64 pipe.
// Values stay unpacked, in registers, from the first step to the last: a warp owns 32 C consecutive cells, C on each lane,
// steps * R of them on either side a halo that goes wrong from the outside in; a
// lane takes the R values beyond its ends from its neighbours by shuffles, and the sums are
// rounded by integer instructions (WideAcc::val), which costs neither FP64 nor unpacking.
// (With get() and unpacking in val's place, for all cells or every second to fourth: the same
// time within 1%.)  Shared memory only turns the rows of 32 that global memory likes into the lanes' runs of C.
//
// Us a step, radius 1 (before, by the FMA chain from shared memory, single steps at the end of
// a run): 10^3 cells 1.2 (2.8), 60 000 1.3 (3.0), 220 000 2.5 (3.0), 10^6 5.3 (7.4), 10^7
// 43 (55; 50 with the cells that the integer form does not take told apart one by one).
// C, us a step at radius 1: 20 000 cells 2: 1.0, 4: 1.5; 220 000 2.4 / 2.6 (radius
// 2 4.0 / 3.4); 10^6 4: 5.3, 8: 5.8 (radius 2 8.5 / 7.7); 10^7 42.8 / 43.2 (74.9 / 63.9).
#include "internal.h"
#include "wide.cuh"

namespace gbst {
namespace {

constexpr int kThreads1d = 256;

// One cell that the integer form does not take.  Out of line: rarely run.
template <int NT>
__device__ __noinline__ WideVal chain_cell(const WideVal (&u)[NT], const double* wdev) {
  double v[NT];
  for (int k = 0; k < NT; ++k) v[k] = wide_repack(u[k]);
  return wide_unpack(wide_chain(v, wdev, NT));
}

template <int R, int C, bool HEAT, bool PERIODIC>
__global__ void __launch_bounds__(kThreads1d, 2)
    k_wide1d(const double* __restrict__ src, double* __restrict__ dst, int n, int steps,
             const double* __restrict__ wdev, const __grid_constant__ WideTapsOf<5> T) {
  constexpr int NT = 2 * R + 1, kCells = 32 * C;
  constexpr unsigned int kAll = 0xffffffffu;
  __shared__ double buf[kThreads1d / 32][32 * (C + 1)];
  const int lane = threadIdx.x & 31;
  double* const b = buf[threadIdx.x >> 5];
  const int halo = R * steps, own = kCells - 2 * halo;
  const long long at = ((long long)blockIdx.x * (kThreads1d / 32) + (threadIdx.x >> 5)) * own;
  if (at >= n) return;
  const long long x0 = at - halo;  // of the warp's first cell
  const bool inside = x0 >= 0 && x0 + kCells <= n;
#pragma unroll
  for (int k = 0; k < C; ++k) {
    const int i = 32 * k + lane;
    long long x = x0 + i;
    double v = 0.0;
    if (PERIODIC) {
      if (!inside) x = (x % n + n) % n;
      v = __ldg(src + x);
    } else if (x >= 0 && x < n) {
      v = __ldg(src + x);
    }
    b[i + i / C] = v;
  }
  __syncwarp();
  WideVal u[C];
#pragma unroll
  for (int j = 0; j < C; ++j) u[j] = wide_unpack(b[lane * (C + 1) + j]);
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    WideVal before[R], after[R];  // of the lane's first cell (nearest last) and of its last one
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const WideVal& l = u[C - R + r];
      before[r] = {__shfl_up_sync(kAll, l.hi, 1), __shfl_up_sync(kAll, l.lo, 1), __shfl_up_sync(kAll, l.e, 1)};
      const WideVal& h = u[r];
      after[r] = {__shfl_down_sync(kAll, h.hi, 1), __shfl_down_sync(kAll, h.lo, 1), __shfl_down_sync(kAll, h.e, 1)};
    }
    auto near = [&](int j, WideVal (&v)[NT]) {  // the values that cell j reads
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        const int q = j + k - R;
        v[k] = q < 0 ? before[q < 0 ? q + R : 0] : q < C ? u[q < 0 || q >= C ? 0 : q] : after[q < C ? 0 : q - C];
      }
    };
    // all cells first, without a branch between them, which would keep them apart
    WideVal w[C];
    unsigned int other = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
      WideVal v[NT];
      near(j, v);
      WideAcc acc;
      int E;
      if constexpr (HEAT) E = wide_acc_heat<NT>(v, T, acc);
      else E = wide_acc<NT>(v, T, acc);
      w[j] = acc.val(E, T);
      if (!wide_covers(E, T)) other |= 1u << j;
    }
    if (other != 0) {
#pragma unroll
      for (int j = 0; j < C; ++j)
        if (other >> j & 1) {
          WideVal v[NT];
          near(j, v);
          w[j] = wide_zeros<NT>(v) ? wide_unpack(0.0) : chain_cell<NT>(v, wdev);
        }
    }
#pragma unroll
    for (int j = 0; j < C; ++j) {
      u[j] = w[j];
      if (!PERIODIC && !inside) {
        const long long x = x0 + lane * C + j;
        if (x < 0 || x >= n) u[j] = wide_unpack(0.0);  // a ghost stays zero
      }
    }
  }
#pragma unroll
  for (int j = 0; j < C; ++j) b[lane * (C + 1) + j] = wide_repack(u[j]);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < C; ++k) {
    const int i = 32 * k + lane;
    if (i >= halo && i < halo + own && x0 + i < n) dst[x0 + i] = b[i + i / C];
  }
}

template <int R, int C>
cudaError_t launch_c(bool per, int steps, int n, const WideTapsOf<5>& T, const double* wdev, const double* src,
                     double* dst, cudaStream_t stream) {
  const int own = 32 * C - 2 * R * steps;
  const long long warps = ((long long)n + own - 1) / own;
  const unsigned int blocks = (unsigned int)((warps + kThreads1d / 32 - 1) / (kThreads1d / 32));
  if (T.heat) {
    if (per) k_wide1d<R, C, true, true><<<blocks, kThreads1d, 0, stream>>>(src, dst, n, steps, wdev, T);
    else k_wide1d<R, C, true, false><<<blocks, kThreads1d, 0, stream>>>(src, dst, n, steps, wdev, T);
  } else {
    if (per) k_wide1d<R, C, false, true><<<blocks, kThreads1d, 0, stream>>>(src, dst, n, steps, wdev, T);
    else k_wide1d<R, C, false, false><<<blocks, kThreads1d, 0, stream>>>(src, dst, n, steps, wdev, T);
  }
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_wide1d(int radius, int boundary, int steps, const Geom& g, const WideTapsOf<5>& wide,
                          const double* wdev, const double* src, double* dst, int sms, cudaStream_t stream) {
  if (steps < 1 || steps > kWide1dSteps || wide.n != 2 * radius + 1 || (radius != 1 && radius != 2))
    return cudaErrorInvalidValue;
  const bool per = boundary == kPeriodic;
  // more cells per lane: less halo; fewer: more warps, each with a shorter chain (above)
  const int c = g.nx >= 1 << 20 ? 8 : g.nx >= 1 << 16 ? 4 : 2;
  if (radius == 1)
    return c == 8 ? launch_c<1, 8>(per, steps, g.nx, wide, wdev, src, dst, stream)
           : c == 4 ? launch_c<1, 4>(per, steps, g.nx, wide, wdev, src, dst, stream)
                    : launch_c<1, 2>(per, steps, g.nx, wide, wdev, src, dst, stream);
  return c == 8 ? launch_c<2, 8>(per, steps, g.nx, wide, wdev, src, dst, stream)
         : c == 4 ? launch_c<2, 4>(per, steps, g.nx, wide, wdev, src, dst, stream)
                  : launch_c<2, 2>(per, steps, g.nx, wide, wdev, src, dst, stream);
}

}  // namespace gbst
