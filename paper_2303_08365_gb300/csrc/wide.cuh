// wide.cuh -- the weighted sum of a sweep in integer arithmetic.
//
// This GPU issues 2 FP64 instructions per clock per SM but 64 of each of the
// integer kinds that the sum needs (measured per clock per SM: DFMA 1.98,
// 32 x 32 + 64 bit multiply-add 62, shift and logic 63, 64-bit shift 25), so
// sum_k w_k u_k over K taps costs K/2 clocks on the FP64 pipe and about 0.13 K
// + 0.2 on the integer pipes.  The sum is taken in fixed point, aligned cell by
// cell:
//   - u_k is unpacked into a signed 62-bit integer M_k (the 53-bit significand,
//     9 zero bits below it) and its exponent; w_k = W_k 2^x_k, W_k the 53-bit
//     significand, is split once on the host into two limbs of 27 and 26 bits;
//   - E = the largest exponent of any product w_k u_k; A_k = M_k >> (E - e_k),
//     so the low bits that a product loses lie 2^-62 below the largest one;
//   - S = sum_k A_k W_k, exactly, in four 64-bit accumulators of 32 x 32 bit
//     products, then R = S / 2^57 rounded, 56 bits or more for the largest product;
//   - R is rounded once to a double and its exponent is set.
// The error is one rounding of the result and about 2^-55 of the largest product
// (half a unit of R, and K/16 units from the bits that the alignment drops),
// against K roundings of partial sums in an FMA chain.  The result is
// a function of the K values alone: every kernel that takes it gives the same
// bits, whatever its tiles.  (One kernel of a class that has it does not: the overlapped temporal
// kernel for 2D boxes of equal weights, temporal.cu.)
//
// Boxes whose weights are all equal take one multiplication a cell, and share the alignment of
// a value between cells where a kernel can (WideSum).  For their results to be a function of
// the K values alone all the same, E is the next number of the form 4 n + 3 from the largest
// exponent on: neighbouring cells seldom differ in that.  (In the largest exponent itself they
// would differ wherever a field passes a power of two.)  With up to three bits fewer, the unit
// of A that a negative value's one's complement is short by would show over many steps (160 of
// a 9-point box: 2.2e-16 between a field and its negative), so theirs is a two's complement.
//
// It covers weights > 0.  Values whose largest exponent is out of the range in
// which that is safe (infinities, NaN, products near the largest or the
// smallest doubles, neighbourhoods that are all zero) take the FMA chain, cell by cell.
#pragma once

#include <cmath>
#include <cstdint>

#include "internal.h"
#include "taps.cuh"

namespace gbst {

// Splits the weights; false (and n = 0) when the integer form does not cover
// them: a weight that is not positive, or weights so far apart or so extreme
// that no range of exponents is left.
template <int N>
inline bool make_wide(const double* w, int n, WideTapsOf<N>& t, bool box = false) {
  t.n = t.heat = t.equal = 0;
  if (n < 1 || n > N) return false;
  int xmax = -100000, x[N];
  for (int k = 0; k < n; ++k) {
    if (!(w[k] > 0.0) || !std::isfinite(w[k])) return false;
    std::frexp(w[k], &x[k]);  // w = m 2^x, m in [0.5, 1)
    if (x[k] > xmax) xmax = x[k];
  }
  int ex_min = 0;
  for (int k = 0; k < n; ++k) {
    const int64_t W = (int64_t)std::ldexp(w[k], 53 - x[k]);  // [2^52, 2^53), exact
    const int64_t hi = W >> 26, lo = W - hi * (1 << 26);
    t.hi[k] = (int)hi;
    t.hi2[k] = (int)(2 * hi);
    t.lo[k] = (int)lo;
    t.ex[k] = x[k] - xmax;
    if (t.ex[k] < ex_min) ex_min = t.ex[k];
  }
  t.bias = 1080 - xmax;
  // a zero or subnormal value is unpacked as if it had a leading 1: E >= 64
  // shifts it out; the result's exponent stays within the normal range; an
  // infinity or NaN (exponent field 2047) is always above e_max
  const int e_min = t.bias - 1010 > 64 ? t.bias - 1010 : 64;
  const int e_max = 2046 + ex_min < 2030 - xmax ? 2046 + ex_min : 2030 - xmax;
  if (e_max < e_min + 256) return false;
  t.e_min = e_min;
  t.e_span = (unsigned)(e_max - e_min);
  t.heat = n >= 3 && n % 2 == 1;
  for (int k = 1; k < n; ++k)
    if (k != n / 2 && w[k] != w[0]) t.heat = 0;
  t.equal = box && t.heat && w[n / 2] == w[0];
  t.n = n;
  return true;
}

#ifdef __CUDACC__

// A value unpacked: the signed 62-bit integer (hi, lo) and its exponent field.
struct WideVal {
  int hi;
  unsigned int lo;
  int e;
};

__device__ __forceinline__ WideVal wide_unpack(double v) {
  const unsigned int hi = (unsigned int)__double2hiint(v), lo = (unsigned int)__double2loint(v);
  const int s = (int)hi >> 31;
  const unsigned int m = (hi & 0xfffffu) | 0x100000u;
  WideVal u;
  u.e = (int)((hi << 1) >> 21);
  // one's complement for negative values: 2^-62 of the value away
  u.hi = (int)(__funnelshift_l(lo, m, 9) ^ (unsigned int)s);
  u.lo = (lo << 9) ^ (unsigned int)s;
  return u;
}

// From and to two's complement for negative values (boxes of equal weights).
__device__ __forceinline__ WideVal wide_twos(WideVal u) {
  const int s = u.hi >> 31;
  const long long m = (long long)(((unsigned long long)(unsigned int)u.hi << 32) | u.lo) - s;
  u.hi = (int)(m >> 32);
  u.lo = (unsigned int)m;
  return u;
}
__device__ __forceinline__ WideVal wide_ones(WideVal u) {
  const long long v = (long long)(((unsigned long long)(unsigned int)u.hi << 32) | u.lo);
  const long long m = v + (v >> 63);
  u.hi = (int)(m >> 32);
  u.lo = (unsigned int)m;
  return u;
}

// Zero bits when the value is a zero.  Neighbourhoods of zeros, which the integer form
// does not take, are told apart first: whole grids of them are ordinary input (512^3 with
// one hot cell: 134 GStencil/s, the FMA chain for each 17; no zeros 170).
__device__ __forceinline__ unsigned int wide_nonzero(const WideVal& u) {
  const unsigned int s = (unsigned int)(u.hi >> 31);
  return ((unsigned int)u.hi ^ s ^ 0x20000000u) | (u.lo ^ s) | (unsigned int)u.e;
}
template <int NT>
__device__ __forceinline__ bool wide_zeros(const WideVal (&u)[NT]) {
  unsigned int any = 0;
#pragma unroll
  for (int k = 0; k < NT; ++k) any |= wide_nonzero(u[k]);
  return any == 0;
}

// The double that was unpacked (exact, whatever it was).
__device__ __forceinline__ double wide_repack(const WideVal& u) {
  const unsigned int s = (unsigned int)(u.hi >> 31);
  const unsigned int h = (unsigned int)u.hi ^ s, l = u.lo ^ s;
  return __hiloint2double((int)((s & 0x80000000u) | ((unsigned int)u.e << 20) | ((h >> 9) & 0xfffffu)),
                          (int)__funnelshift_r(l, h, 9));
}

// The FMA chain for the neighbourhoods that the integer form does not take
// (wdev: the weights as doubles, in global memory or among a kernel's parameters, so by plain
// loads: the read-only path takes global addresses alone).  Out of line: it is rarely run.
static __device__ __noinline__ double wide_chain(const double* v, const double* wdev, int n) {
  long long any = 0;
  for (int k = 0; k < n; ++k) any |= __double_as_longlong(v[k]) << 1;
  if (any == 0) return 0.0;  // every value is a zero
  double acc = 0.0;
  for (int k = 0; k < n; ++k) acc = fma(wdev[k], v[k], acc);
  return acc;
}

// Whether the integer form takes a cell whose largest product has exponent E.
template <class Taps>
__device__ __forceinline__ bool wide_covers(int E, const Taps& T) {
  return (unsigned int)(E - T.e_min) <= T.e_span;
}

// M >> d; an amount over 63 leaves the sign.
__device__ __forceinline__ long long wide_align(const WideVal& u, int d) {
  long long a;
  asm("{.reg .b64 t; mov.b64 t, {%2, %1}; shr.s64 %0, t, %3;}" : "=l"(a) : "r"(u.hi), "r"(u.lo), "r"(d));
  return a;
}

// R 2^x, rounded once to a double.
__device__ __forceinline__ double wide_double(long long R, int x) {
  // R to double: (2^84 + 2^63 + high) - (2^84 + 2^63 + 2^52) exactly, then one
  // rounding when the low word (2^52 + low) is added.  As FMAs on registers,
  // which run at the full FP64 rate (additions at 83%)
  double one, off;
  asm("mov.f64 %0, 0d3FF0000000000000;" : "=d"(one));
  asm("mov.f64 %0, 0dC530000080100000;" : "=d"(off));
  const double dh = __hiloint2double(0x45300000, (int)(R >> 32) ^ (int)0x80000000);
  const double dl = __hiloint2double(0x43300000, (int)(unsigned int)R);
  const double r = fma(dl, one, fma(dh, one, off));
  const int h = __double2hiint(r);
  return __hiloint2double(h != 0 ? h + (x << 20) : h, __double2loint(r));
}

// The same, rounded alike, unpacked: for a value that the next step reads, without the two FP64
// instructions (64 cycles each) between.
__device__ __forceinline__ WideVal wide_val(long long R, int x) {
  const long long s = R >> 63;
  const unsigned long long a = (unsigned long long)((R ^ s) - s);
  if (a == 0) return wide_unpack(0.0);
  const int lz = __clzll((long long)a);
  const unsigned long long n = a << lz;  // leading bit 63; 53 bits stay
  unsigned long long r = n + 0x3ff + ((n >> 11) & 1);
  const bool carry = r < n;
  r = carry ? 1ull << 63 : r;
  const unsigned long long m = ((r & ~0x7ffull) >> 2) ^ (unsigned long long)s;
  WideVal u;
  u.hi = (int)(m >> 32);
  u.lo = (unsigned int)m;
  u.e = x + (1023 + 63) - lz + (carry ? 1 : 0);
  return u;
}

// The accumulators of a cell: hh, hl, lh and ll count units of 2^57, 2^32, 2^26 and
// 1 of S (27 taps: below 2^63 each).
struct WideAcc {
  long long hh, hl;
  unsigned long long lh, ll;
  __device__ __forceinline__ WideAcc() : hh(0), hl(1 << 24 /* half a unit of R */), lh(0), ll(0) {}

  // Adds W_k a.
  template <class Taps>
  __device__ __forceinline__ void add(long long a, int k, const Taps& T) {
    const int ah = (int)(a >> 32);
    const unsigned int al = (unsigned int)a;
    // one multiply-add each (written in C, the addends cost moves: 149 against
    // 115 instructions for a 5-tap cell)
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hh) : "r"(ah), "r"(T.hi2[k]));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hl) : "r"(ah), "r"(T.lo[k]));
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(lh) : "r"(al), "r"(T.hi[k]));
    asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(ll) : "r"(al), "r"(T.lo[k]));
  }

  // Adds w_k u whose product lies d exponents below the cell's largest.
  template <class Taps>
  __device__ __forceinline__ void add(const WideVal& u, int k, int d, const Taps& T) {
    add(wide_align(u, d), k, T);
  }

  __device__ __forceinline__ long long rounded() const {  // R
    return hh + ((hl + (long long)((lh + (ll >> 26)) >> 6)) >> 25);
  }

  template <class Taps>
  __device__ __forceinline__ WideVal val(int E, const Taps& T) const {
    return wide_val(rounded(), E - T.bias);
  }

  // The sum as a double.
  template <class Taps>
  __device__ __forceinline__ double get(int E, const Taps& T) const {
    return wide_double(rounded(), E - T.bias);
  }
};

// sum_k w_k u_k of one cell (the file's head comment); ok = false, and a
// result without meaning, where the FMA chain has to take the cell.  wide_acc:
// the sum before its rounding; returns E.
template <int NT, class Taps>
__device__ __forceinline__ int wide_acc(const WideVal (&u)[NT], const Taps& T, WideAcc& acc) {
  int e[NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) e[k] = u[k].e + T.ex[k];
  int E = e[0];
#pragma unroll
  for (int k = 1; k < NT; ++k) E = max(E, e[k]);
#pragma unroll
  for (int k = 0; k < NT; ++k) acc.add(u[k], k, E - e[k], T);
  return E;
}
template <int NT, class Taps>
__device__ __forceinline__ double wide_sum(const WideVal (&u)[NT], const Taps& T, bool& ok) {
  WideAcc acc;
  const int E = wide_acc<NT>(u, T, acc);
  ok = wide_covers(E, T);
  return acc.get(E, T);
}

// The same for weights that are one value at the centre tap (NT / 2) and one at
// all the others (Eq. 3): one exponent for the neighbours, and their integers added
// in pairs (two of 62 bits fit 63) before the multiplication.  S is exact either
// way, so the result has the same bits.
template <int NT, class Taps>
__device__ __forceinline__ int wide_acc_heat(const WideVal (&u)[NT], const Taps& T, WideAcc& acc) {
  constexpr int C = NT / 2;  // NT - 1 neighbours: an even number
  auto nb = [&](int k) -> const WideVal& { return u[k < C ? k : k + 1]; };
  int en = nb(0).e;
#pragma unroll
  for (int k = 1; k + 1 < NT - 1; k += 2) en = __vimax3_s32(en, nb(k).e, nb(k + 1).e);
  en = max(en, nb(NT - 2).e);
  const int ec = u[C].e + T.ex[C];
  const int E = max(en + T.ex[0], ec);
  const int dn = E - T.ex[0];
#pragma unroll
  for (int k = 0; k < NT - 1; k += 2)
    acc.add(wide_align(nb(k), dn - nb(k).e) + wide_align(nb(k + 1), dn - nb(k + 1).e), 0, T);
  acc.add(u[C], C, E - ec, T);
  return E;
}
template <int NT, class Taps>
__device__ __forceinline__ double wide_sum_heat(const WideVal (&u)[NT], const Taps& T, bool& ok) {
  WideAcc acc;
  const int E = wide_acc_heat<NT>(u, T, acc);
  ok = wide_covers(E, T);
  return acc.get(E, T);
}

// The sum of aligned values (two's complement) of a box whose weights are all equal: up to 27
// of 63 bits, so the sum modulo 2^64, and the sum of the values' top bits (units of 2^37), which
// has the rest.  (Values cut to 58 bits, whose sum fits 64, lean to one side: spread from e^-4 to
// e^4, by 0.10 of 2^-53 a step of a 27-point box; so, 0.02.)
struct WideSum {
  long long s;
  int top;
  __device__ __forceinline__ WideSum() : s(0), top(0) {}
  __device__ __forceinline__ explicit WideSum(long long a) : s(a), top((int)(a >> 37)) {}
  __device__ __forceinline__ WideSum& operator+=(const WideSum& o) {
    s += o.s;
    top += o.top;
    return *this;
  }
  friend __device__ __forceinline__ WideSum operator+(WideSum a, const WideSum& o) { return a += o; }
  // The sum's bits from the 64th on.  From the 37th on the values' bits fall short of the sum's
  // by one a value at most, and 27 of the sum's are in s.
  __device__ __forceinline__ int over() const {
    return (top - (int)((unsigned long long)s >> 37) + (1 << 26)) >> 27;
  }
  // Times 2^g, g < 37.
  __device__ __forceinline__ void shift(int g) {
    const int high = (over() << 27) | (int)((unsigned long long)s >> 37);
    top = (high << g) | ((int)((unsigned long long)s >> (37 - g)) & ((1 << g) - 1));
    s <<= g;
  }
};

// A value's share of a sum of exponent E.
__device__ __forceinline__ WideSum wide_part(const WideVal& u, int E) { return WideSum(wide_align(u, E - u.e)); }

// What they need of the weights, one value, side by side in one line of a kernel's parameters
// (16384^2: 13.4 ms for ten steps; apart, 13.7 to 14.0).
struct alignas(16) WideEqualTaps {
  int lo[1], hi[1], hi2[1], bias, e_min;
  unsigned int e_span;
  template <int N>
  WideEqualTaps& operator=(const WideTapsOf<N>& t) {
    lo[0] = t.lo[0];
    hi[0] = t.hi[0];
    hi2[0] = t.hi2[0];
    bias = t.bias;
    e_min = t.e_min;
    e_span = t.e_span;
    return *this;
  }
};

// R = w S / 2^57 rounded, w the weights' one value.
template <class Taps>
__device__ __forceinline__ long long wide_equal(const WideSum& S, const Taps& T) {
  const int ext = S.over();  // S = ext 2^64 + s
  const unsigned int ah = (unsigned int)((unsigned long long)S.s >> 32), al = (unsigned int)S.s;
  const unsigned int lo = (unsigned int)T.lo[0], hi = (unsigned int)T.hi[0], hi2 = (unsigned int)T.hi2[0];
  // units of 2^57, 2^32, 2^26 and 1 of S W
  const unsigned long long lh = (unsigned long long)al * hi + ((unsigned long long)al * lo >> 26);
  const unsigned long long hl = (unsigned long long)ah * lo + (1 << 24) + (lh >> 6);
  const long long top = (long long)(ext << 7) * (int)lo + ((long long)(ext * (int)hi2) << 32);
  return (long long)((unsigned long long)ah * hi2 + (hl >> 25)) + top;
}
template <class Taps>
__device__ __forceinline__ double wide_equal_double(const WideSum& S, int E, const Taps& T) {
  return wide_double(wide_equal(S, T), E - T.bias);
}

// One cell: S and E.
template <int NT>
__device__ __forceinline__ int wide_acc_equal(const WideVal (&u)[NT], WideSum& S) {
  int E = u[0].e;
#pragma unroll
  for (int k = 1; k < NT; ++k) E = max(E, u[k].e);
  E |= 3;
#pragma unroll
  for (int k = 0; k < NT; ++k) S += wide_part(wide_twos(u[k]), E);
  return E;
}
template <int NT, class Taps>
__device__ __forceinline__ double wide_sum_equal(const WideVal (&u)[NT], const Taps& T, bool& ok) {
  WideSum S;
  const int E = wide_acc_equal<NT>(u, S);
  ok = wide_covers(E, T);
  return wide_equal_double(S, E, T);
}

// How a kernel takes the weighted sum of a cell, collected tap by tap: the FMA
// chain in tap order, or the integer form once every value is there (kHeat: for
// weights that wide_sum_heat takes, or a box whose weights are all equal).
enum SumForm : int { kChain = 0, kWide = 1, kHeat = 2 };

template <int NT, int FORM, class Taps = WideTaps>
struct TapSum {
  struct Acc {
    WideVal u[NT];
  };
  const Taps& T;
  const double* wdev;
  __device__ __forceinline__ TapSum(const double* __restrict__ w, const Taps& t) : T(t), wdev(w) {}
  __device__ __forceinline__ void tap(Acc& acc, int k, double v, int) const { acc.u[k] = wide_unpack(v); }
  // ok = false: the FMA chain has to take the cell
  __device__ __forceinline__ double get(const Acc& acc, bool& ok) const {
    if constexpr (FORM == kHeat && NT >= 9) return wide_sum_equal<NT>(acc.u, T, ok);
    else if constexpr (FORM == kHeat) return wide_sum_heat<NT>(acc.u, T, ok);
    else return wide_sum<NT>(acc.u, T, ok);
  }
  __device__ __forceinline__ double get(const Acc& acc) const {
    bool ok;
    const double r = get(acc, ok);
    if (ok) return r;
    if (wide_zeros<NT>(acc.u)) return 0.0;
    double v[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) v[k] = wide_repack(acc.u[k]);
    return wide_chain(v, wdev, NT);
  }
};

template <int NT, class Taps>
struct TapSum<NT, kChain, Taps> {
  using Acc = double;
  RegWeights<NT> W;
  __device__ __forceinline__ TapSum(const double* __restrict__ wdev, const Taps&) { W.load(wdev); }
  __device__ __forceinline__ void tap(Acc& acc, int k, double v, int c) const { W.tap(acc, k, v, c); }
  __device__ __forceinline__ double get(const Acc& acc, bool& ok) const {
    ok = true;
    return acc;
  }
  __device__ __forceinline__ double get(const Acc& acc) const { return acc; }
};

#endif  // __CUDACC__

}  // namespace gbst
