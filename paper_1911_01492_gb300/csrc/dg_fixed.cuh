// Block fixed-point arithmetic for the FP64 operator.
//
// GB300 issues an FP64 instruction for a warp once per 64 cycles and
// scheduler; a 32 x 32 + 64 bit integer multiply-add (mad.wide.s32) takes 4.  The
// FP64 operator is bound by its FP64 instructions (98-103 % of their rate), so
// the operator's contractions run on the integer pipe instead: the values of
// one cell share one exponent and are 64-bit integers, a product of two
// 60-bit numbers is three 32-bit products, and sums of 64-bit integers are two
// additions.  Measured on a dense 4 x 4 line contraction: 227 cycles against
// 1204 with FP64 multiply-adds.
//
// Number format.  A value v stands for v 2^E with E per cell.  A constant or
// coefficient T in (-2, 2) is stored as T 2^60 = h 2^30 + l with |l| <= 2^29
// (FxPair).  A value splits as v = h 2^30 + l with 0 <= l < 2^30.  Their product
// over 2^60 is h h' + (h l' + l h') / 2^30, where the l l' term (below 2^-1 of
// the last place) is left out: an absolute error of about one unit, 2^-59 of the
// cell's largest value, against 2^-53 of each partial sum in FP64.
//
// Ranges, which make every sum fit 64 bits whatever the data:
//   * |v| <= 2^60 (sums of a mirror pair 2^61), so |h| <= 2^31 exclusive;
//   * the entries of a table row are scaled so that the row's result obeys the
//     same bound (the bases are orthonormal: the transforms preserve the
//     2-norm of a cell, which starts at <= 2^60);
//   * low-order sums: at most 9 terms of 2^30 2^30 and 2^29 2^31 stay below 2^63.
#pragma once

#include "dg_apply_impl.cuh"

namespace dgk {

// cells whose data holds a NaN or an infinity carry this exponent
constexpr int FX_NAN = 1 << 24;

// Largest power of two S0 with n^{3/2} 2^S0 <= 2^60: values of magnitude below
// 2^S0 have a cell 2-norm of at most 2^60.
template <int N>
struct FxScale {
  static constexpr int S0 = N == 2 ? 58 : N == 3 ? 57 : N == 4 ? 57 : N <= 6 ? 56 : 55;
};

// shared-memory strides of a cell's n x n x n values (8-byte words): odd row
// strides keep the x- and y-line accesses of 16 lanes on different banks
template <int N>
struct FxPad {
  static constexpr int SY = N + (N % 2 == 0 ? 1 : 0), SZ = N * SY, SC = N * SZ;
};

struct FxVal { int h, l; };  // a value v = h 2^30 + l

__device__ __forceinline__ FxVal fx_split(long long v) {
  return {(int)(v >> 30), (int)v & 0x3fffffff};
}

// h: sum of h h'; m: sum of the cross products, starting at the rounding term
struct FxAcc { long long h, m; };

__device__ __forceinline__ long long fx_madw(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// acc += t v
__device__ __forceinline__ void fx_mac(FxAcc& acc, const FxPair& t, const FxVal& v) {
  acc.h = fx_madw(t.h, v.h, acc.h);
  acc.m = fx_madw(t.h, v.l, acc.m);
  acc.m = fx_madw(t.l, v.h, acc.m);
}

// SH: result times 2^SH
template <int SH = 0>
__device__ __forceinline__ FxAcc fx_zero() { return {0, 1ll << (29 - SH)}; }
template <int SH = 0>
__device__ __forceinline__ long long fx_value(const FxAcc& a) {
  return (a.h << SH) + (a.m >> (30 - SH));
}

__device__ __forceinline__ FxPair fx_pair(long long t) {
  const int h = (int)((t + (1ll << 29)) >> 30);
  return {h, (int)(t - ((long long)h << 30))};
}

__device__ __forceinline__ long long fx_shift(long long v, int s) {  // v 2^s, |s| < 64
  return s >= 0 ? v << s : v >> -s;
}

// exponent E with |x| < 2^E for every x whose high word without sign is at most
// hi; FX_NAN for NaN or infinity
__device__ __forceinline__ int fx_exponent(unsigned hi) {
  const int e = (int)(hi >> 20);
  if (e == 0) return (hi != 0 ? 64 - __clz((int)hi) : 32) - 1074;  // subnormal or zero
  return e == 2047 ? FX_NAN : e - 1022;
}

__device__ __forceinline__ unsigned fx_abs_hi(double x) {
  return (unsigned)__double2hiint(x) & 0x7fffffffu;
}

// round(x 2^k) for values whose largest magnitude is below 2^E (result < 2^(E + k))
__device__ __forceinline__ long long fx_from_double(double x, int k, int E) {
  if (E < -900) {  // subnormal numbers near: scale in two steps
    const int k1 = k / 2;
    return __double2ll_rn(scalbn(scalbn(x, k1), k - k1));
  }
  // 2^k by adding to the exponent; what is too small for that rounds to zero
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  const double s = __hiloint2double(hi + (int)((unsigned)k << 20), __double2loint(x));
  return e > (k < 0 ? -k : 0) ? __double2ll_rn(s) : 0;
}

// v 2^k
__device__ __forceinline__ double fx_to_double(long long v, int k) {
  const double d = (double)v;
  if (k > 900 || k < -900) return scalbn(d, k);
  return v != 0 ? __hiloint2double(__double2hiint(d) + (int)((unsigned)k << 20),
                                   __double2loint(d))
                : 0.0;
}

// magnitude's high word, for fx_bits of a maximum
__device__ __forceinline__ unsigned fx_mag_hi(long long v) {
  return (unsigned)((unsigned long long)(v < 0 ? ~v : v) >> 32);
}
// smallest b >= 32 with every magnitude below 2^b
__device__ __forceinline__ int fx_bits(unsigned mag_hi) { return 64 - __clz((int)mag_hi); }

// Largest v over the threads of the calling thread's cell.  Cells that lie
// inside one warp need no barrier; otherwise slots[CPB] (zeroed before an
// earlier barrier) collects the warps' maxima.  Every thread of the block calls it.
template <int N>
__device__ __forceinline__ unsigned fx_cell_max(unsigned v, int lc, unsigned* slots) {
  constexpr int N2 = N * N, T = Cfg<N>::THREADS;
  const int lane = threadIdx.x & 31, base = (int)threadIdx.x - lane;
  const int lo = lc * N2 > base ? lc * N2 - base : 0;
  int hi = (lc + 1) * N2 - base;
  const int lanes = T - base < 32 ? T - base : 32;
  if (hi > lanes) hi = lanes;
  const unsigned mask = (hi >= 32 ? 0xffffffffu : (1u << hi) - 1u) & ~((1u << lo) - 1u);
  v = __reduce_max_sync(mask, v);
  if constexpr (32 % N2 == 0) return v;
  if (lane == lo) atomicMax(slots + lc, v);
  __syncthreads();
  return slots[lc];
}

// u[a] = sum_i q[a][i] x[i], parity split (q[N-1-a][i] = (-1)^i q[a][i])
template <int N>
__device__ __forceinline__ void fx_fwd(const DGTabX& t, const long long (&x)[N],
                                       long long (&u)[N]) {
  FxVal s[N];
#pragma unroll
  for (int i = 0; i < N; ++i) s[i] = fx_split(x[i]);
#pragma unroll
  for (int a = 0; a < (N + 1) / 2; ++a) {
    FxAcc E = fx_zero();
#pragma unroll
    for (int i = 0; i < N; i += 2) fx_mac(E, t.q[a][i], s[i]);
    const long long e = fx_value(E);
    if (a == N - 1 - a) {
      u[a] = e;
    } else {
      FxAcc O = fx_zero();
#pragma unroll
      for (int i = 1; i < N; i += 2) fx_mac(O, t.q[a][i], s[i]);
      const long long o = fx_value(O);
      u[a] = e + o;
      u[N - 1 - a] = e - o;
    }
  }
}

// x[i] = sum_a q[a][i] r[a]
template <int N>
__device__ __forceinline__ void fx_bwd(const DGTabX& t, const long long (&r)[N],
                                       long long (&x)[N]) {
  constexpr int H = N / 2, P = (N + 1) / 2;
  FxVal e[P], o[H];
#pragma unroll
  for (int a = 0; a < H; ++a) {
    e[a] = fx_split(r[a] + r[N - 1 - a]);
    o[a] = fx_split(r[a] - r[N - 1 - a]);
  }
  if (N % 2 == 1) e[P - 1] = fx_split(r[H]);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    FxAcc A = fx_zero();
    if (i % 2 == 0) {
#pragma unroll
      for (int a = 0; a < P; ++a) fx_mac(A, t.q[a][i], e[a]);
    } else {
#pragma unroll
      for (int a = 0; a < H; ++a) fx_mac(A, t.q[a][i], o[a]);
    }
    x[i] = fx_value(A);
  }
}

}  // namespace dgk
