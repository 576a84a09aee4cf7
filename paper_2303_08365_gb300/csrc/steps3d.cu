// steps3d.cu -- all steps of a small 3D 7-point grid in ONE persistent cooperative launch,
// with the weighted sum in the integer form (wide.cuh).
//
// Operation: steps of u'(x) = sum_o w_o u~(x+o) (paper Sec. 2.1, Listing 1).  A launch per step
// costs more than the step where a grid has a few hundred thousand cells (64^3: 7.1 us, of which
// the integer pipes need about one).  So every CTA keeps a brick of up to 32 x 8 x 2 Z cells on
// the chip for the whole run, unpacked: in registers (Z cells along z per thread, two threads
// per column) and, for the neighbours, in shared memory with a shell of one cell.  Between steps
// only the cells on the brick's faces go through global memory (the caller's grid and its
// partner, by turns, each cell at its place), and a CTA waits only for the six bricks beside
// its own: progress words, a line each.  A brick that is a step ahead of a neighbour writes
// the faces of the level that the neighbour does not read.
//
// Every warp polls for itself, so that a step has two CTA barriers.  Every wait is bounded
// by wall time.
//
// Us a step of 100, heat, a launch per step before: 24^3 2.5 (4.4), 49^3 3.8 (6.2), 64^3 4.3
// (7.1), 65^3 6.5 (8.2), 70 x 80 x 90 6.6 (10.3), 64 x 64 x 128 7.0 (9.5).  About 1.8 us of
// each are the exchange, the rest 0.6 us for each of the Z cells.
#include <algorithm>

#include "internal.h"
#include "ptx.cuh"
#include "wide.cuh"

namespace gbst {
namespace {

constexpr int kBX = 32, kBY = 8;  // a warp is a row; 8 rows, twice along z
constexpr int kStepThreads = 512;
constexpr int kStepMaxZ = 8;

template <int Z>
struct __align__(16) Shell {
  long long m[2 * Z + 2][kBY + 2][kBX + 2];
  int e[2 * Z + 2][kBY + 2][kBX + 2];
  __device__ __forceinline__ void put(int z, int y, int x, const WideVal& u) {
    m[z][y][x] = (long long)(((unsigned long long)(unsigned int)u.hi << 32) | u.lo);
    e[z][y][x] = u.e;
  }
  __device__ __forceinline__ WideVal get(int z, int y, int x) const {
    const long long v = m[z][y][x];
    return {(int)(v >> 32), (unsigned int)v, e[z][y][x]};
  }
};

// One cell that the integer form does not take.  Out of line: rarely run.
template <int Z>
__device__ __noinline__ WideVal other_cell(const Shell<Z>& S, int z, int y, int x, const double* wdev) {
  const WideVal u[7] = {S.get(z - 1, y, x), S.get(z, y - 1, x), S.get(z, y, x - 1), S.get(z, y, x),
                        S.get(z, y, x + 1), S.get(z, y + 1, x), S.get(z + 1, y, x)};
  if (wide_zeros<7>(u)) return wide_unpack(0.0);
  double v[7];
  for (int k = 0; k < 7; ++k) v[k] = wide_repack(u[k]);
  return wide_unpack(wide_chain(v, wdev, 7));
}

template <int Z, bool HEAT>
__global__ void __launch_bounds__(kStepThreads) k_steps3d(const __grid_constant__ Steps3dLaunch L) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Shell<Z>& S = *reinterpret_cast<Shell<Z>*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int y = warp % kBY, zh = warp / kBY * Z;  // the thread's column, its first cell along z
  // the brick: cells [lo, lo + n) along each axis (x, y, z)
  const int N[3] = {L.nx, L.ny, L.nz};
  const int b[3] = {(int)blockIdx.x % L.bricks[0], (int)blockIdx.x / L.bricks[0] % L.bricks[1],
                    (int)blockIdx.x / (L.bricks[0] * L.bricks[1])};
  int lo[3], n[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lo[d] = (int)((long long)N[d] * b[d] / L.bricks[d]);
    n[d] = (int)((long long)N[d] * (b[d] + 1) / L.bricks[d]) - lo[d];
  }
  const int sy = L.nx, sz = L.nx * L.ny;
  // lanes 0..5 poll the progress of the bricks beside this one (-1: none)
  int beside = -1;
  if (lane < 6) {
    int c[3] = {b[0], b[1], b[2]};
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (lane / 2 == d) {
        c[d] += lane % 2 ? 1 : -1;
        if (L.periodic) c[d] = c[d] < 0 ? L.bricks[d] - 1 : c[d] == L.bricks[d] ? 0 : c[d];
        if (c[d] < 0 || c[d] >= L.bricks[d]) c[0] = -1 - (1 << 30);
      }
    beside = c[0] < 0 ? -1 : (c[2] * L.bricks[1] + c[1]) * L.bricks[0] + c[0];
  }
  // The thread's values of the shell: one of a z face, up to two of the y faces and one of
  // the x faces; at: index in the grid (-1: none, or a ghost), pos: place in the shell.
  constexpr int kH = 1 + (Z + 3) / 4 + 1;
  int at[kH], pz[kH], py[kH], px[kH];
  auto shell = [&](int k, int z, int yy, int x) {  // of the brick's cell (z, y, x), one coordinate beyond it
    int g[3] = {lo[0] + x, lo[1] + yy, lo[2] + z};
    bool in = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (L.periodic) g[d] = g[d] < 0 ? N[d] - 1 : g[d] == N[d] ? 0 : g[d];
      else in = in && g[d] >= 0 && g[d] < N[d];
    }
    at[k] = in ? g[2] * sz + g[1] * sy + g[0] : -1;
    pz[k] = z + 1;
    py[k] = yy + 1;
    px[k] = x + 1;
    if (!in) S.put(pz[k], py[k], px[k], wide_unpack(0.0));  // a ghost: zero from now on
  };
#pragma unroll
  for (int k = 0; k < kH; ++k) at[k] = -1;
  if (lane < n[0] && y < n[1]) shell(0, warp < kBY ? -1 : n[2], y, lane);
#pragma unroll
  for (int q = 0; q < (Z + 3) / 4; ++q) {
    const int z = (warp + 16 * q) / 2;
    if (lane < n[0] && z < n[2]) shell(1 + q, z, warp % 2 ? n[1] : -1, lane);
  }
  {
    const int t = (int)threadIdx.x, z = t / 16, yy = t % 16 / 2;
    if (z < n[2] && yy < n[1]) shell(kH - 1, z, yy, t % 2 ? n[0] : -1);
  }
  const bool mine = lane < n[0] && y < n[1];
  const int left = mine ? min(Z, n[2] - zh) : 0;  // the thread's cells
  const int own = (lo[2] + zh) * sz + (lo[1] + y) * sy + lo[0] + lane;
  const bool side = lane == 0 || lane == n[0] - 1 || y == 0 || y == n[1] - 1;  // all its cells are on a face
  WideVal u[Z];
#pragma unroll
  for (int k = 0; k < Z; ++k) {
    u[k] = wide_unpack(k < left ? __ldcg(L.a + own + k * sz) : 0.0);
    if (k < left) S.put(zh + k + 1, y + 1, lane + 1, u[k]);
  }
  // waits until the bricks beside this one have made `steps` steps; false: gave up
  auto wait_beside = [&](unsigned int steps) {
    bool ok = true;
    if (beside >= 0) {
      const unsigned int* word = L.progress + (int64_t)beside * kFlagWords;
      unsigned int was = 0;
      unsigned long long t0 = 0;
      for (unsigned int spin = 0;; ++spin) {
        unsigned int seen;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(word) : "memory");
        if (seen >= steps) break;
        if ((spin & 63) == 63) {
          const unsigned long long now = globaltimer_ns();
          if (t0 == 0 || seen != was) t0 = now;
          was = seen;
          if (*(volatile int*)L.status != 0) ok = false;
          else if ((long long)(now - t0) > L.spin_limit) {
            atomicCAS(L.status, 0, -5 /* STENCIL_ERR_TIMEOUT */);
            ok = false;
          }
          if (!ok) break;
        }
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    __syncwarp();  // what the polling lanes have acquired holds for the warp
    return ok;
  };
  auto publish = [&](unsigned int steps) {  // (after a CTA barrier)
    if (threadIdx.x == 0 && (int)blockIdx.x != L.mute) {
      __threadfence();
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(L.progress + (int64_t)blockIdx.x * kFlagWords), "r"(steps)
                   : "memory");
    }
  };
  for (int t = 0; t < L.T; ++t) {
    const double* src = t & 1 ? L.b : L.a;
    double* dst = t & 1 ? L.a : L.b;
    const bool ok = t == 0 || wait_beside((unsigned int)t);
    double h[kH];
#pragma unroll
    for (int k = 0; k < kH; ++k) h[k] = ok && at[k] >= 0 ? __ldcg(src + at[k]) : 0.0;
#pragma unroll
    for (int k = 0; k < kH; ++k)
      if (at[k] >= 0) S.put(pz[k], py[k], px[k], wide_unpack(h[k]));
    if (!__syncthreads_and(ok)) return;
    const bool last = t + 1 == L.T;
    WideVal before = S.get(zh, y + 1, lane + 1);
    const WideVal above = S.get(min(zh + Z, 2 * Z) + 1, y + 1, lane + 1);
    // all cells first, without a branch between them, which would keep them apart (64^3:
    // 5.7 us a step)
    unsigned int other = 0;
#pragma unroll
    for (int k = 0; k < Z; ++k) {
      const int z = zh + k + 1;
      WideVal after = above;
      if (k + 1 < Z) {
        after = u[k + 1 < Z ? k + 1 : 0];
        if (k + 1 == left) after = S.get(z + 1, y + 1, lane + 1);  // the shell is next to a ragged brick's last cell
      }
      const WideVal v[7] = {before,  S.get(z, y, lane + 1),     S.get(z, y + 1, lane), u[k], S.get(z, y + 1, lane + 2),
                            S.get(z, y + 2, lane + 1), after};
      before = u[k];
      WideAcc acc;
      int E;
      if constexpr (HEAT) E = wide_acc_heat<7>(v, L.wide, acc);
      else E = wide_acc<7>(v, L.wide, acc);
      u[k] = acc.val(E, L.wide);
      if (!wide_covers(E, L.wide)) other |= 1u << k;
    }
    other &= (1u << left) - 1;
    if (other != 0) {
#pragma unroll
      for (int k = 0; k < Z; ++k)
        if (other >> k & 1) u[k] = other_cell(S, zh + k + 1, y + 1, lane + 1, L.wdev);
    }
#pragma unroll
    for (int k = 0; k < Z; ++k)
      if (k < left && (last ? (L.T & 1) == 0 : side || zh + k == 0 || zh + k + 1 == n[2]))
        dst[own + k * sz] = wide_repack(u[k]);
    __syncthreads();  // the old level is read, the faces are stored
    publish((unsigned int)t + 1);
    if (!last) {
#pragma unroll
      for (int k = 0; k < Z; ++k)
        if (k < left) S.put(zh + k + 1, y + 1, lane + 1, u[k]);
    }
  }
  if (L.T & 1) {  // the result goes where the neighbours read the last step's level
    if (!wait_beside((unsigned int)L.T)) return;
#pragma unroll
    for (int k = 0; k < Z; ++k)
      if (k < left) L.a[own + k * sz] = wide_repack(u[k]);
  }
}

template <int Z, bool HEAT>
cudaError_t launch_z(const Steps3dLaunch& L, cudaStream_t stream) {
  auto kern = k_steps3d<Z, HEAT>;
  constexpr size_t bytes = sizeof(Shell<Z>);
  static std::atomic<int> cache[kMaxDeviceOrdinals];
  const int occ = cached_per_device(cache, [kern] {
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, kStepThreads, bytes) != cudaSuccess)
      n = 0;
    return n;
  });
  if (occ < 1) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(L.bricks[0] * L.bricks[1] * L.bricks[2]), 1, 1);
  cfg.blockDim = dim3(kStepThreads, 1, 1);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, L);
  if (e == cudaSuccess) g_launches.fetch_add(1, std::memory_order_relaxed);
  return e;
}

}  // namespace

int steps3d_cut(const Geom& g, int sms, int (&bricks)[3]) {
  bricks[0] = (g.nx + kBX - 1) / kBX;
  bricks[1] = (g.ny + kBY - 1) / kBY;
  // (products in 64 bits: this is asked of grids of any size)
  for (int z = 1; z <= kStepMaxZ; ++z) {
    bricks[2] = (g.nz + 2 * z - 1) / (2 * z);
    if ((int64_t)bricks[0] * bricks[1] <= sms && (int64_t)bricks[0] * bricks[1] * bricks[2] <= sms) return z;
  }
  return 0;
}

cudaError_t launch_steps3d(const Steps3dLaunch& L, int z, cudaStream_t stream) {
  if (L.T < 1 || L.wide.n != 7) return cudaErrorInvalidValue;
  const bool heat = L.wide.heat != 0;
  switch (z) {
    case 1: return heat ? launch_z<1, true>(L, stream) : launch_z<1, false>(L, stream);
    case 2: return heat ? launch_z<2, true>(L, stream) : launch_z<2, false>(L, stream);
    case 3: return heat ? launch_z<3, true>(L, stream) : launch_z<3, false>(L, stream);
    case 4: return heat ? launch_z<4, true>(L, stream) : launch_z<4, false>(L, stream);
    case 5: return heat ? launch_z<5, true>(L, stream) : launch_z<5, false>(L, stream);
    case 6: return heat ? launch_z<6, true>(L, stream) : launch_z<6, false>(L, stream);
    case 7: return heat ? launch_z<7, true>(L, stream) : launch_z<7, false>(L, stream);
    case 8: return heat ? launch_z<8, true>(L, stream) : launch_z<8, false>(L, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gbst
