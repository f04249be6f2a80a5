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
// coefficient T is stored as T 2^60 = h 2^30 + l with |l| <= 2^29 (FxPair); h is a
// 32-bit integer, so T < 2 - 2^-31.  A value splits as v = h 2^30 + l with 0 <= l < 2^30.  Their product
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
//
// Ranges inside a cell.  One exponent per cell keeps 60 bits of its largest values
// and 60 - b of those 2^b below.  In the Legendre basis every result mixes the
// whole cell and FP64 rounds relative to it too.  In the point basis a point only
// sees its three lines, and FP64 keeps 53 bits of each: there a cell that may hold
// points whose lines are all small against the cell's largest one, in the vector
// (2^7) or in the operator (2^4), or that is outweighed by 2^9 by a neighbour with
// small lines towards it, is applied in FP64 (fx_cells_wide), as exact
// as FP64 throughout.  Lognormal fields of unit variance have no such cells (line
// operators of a cell within 2^3.2) and pay 3 % for the marks (64^3 Q3 345 -> 356
// us); a field of which every cell is marked takes 2.8 ms there, the FP64 kernels
// took 1.25.
#pragma once

#include "dg_apply_impl.cuh"

namespace dgk {

// cells whose data holds a NaN or an infinity carry this exponent
constexpr int FX_NAN = 1 << 24;
// added to the own exponent of a cell of the point basis that is applied in FP64
constexpr int FX_WIDE = 1 << 20;
// bit d of a cell's mark: it has a line along direction d below 2^-7 (vector) or
// 2^-4 (operator) of its largest; a point small in all three needs all bits
constexpr int FX_MARKS = 7;

// A transform preserves the 2-norm of a cell and no value of its stages exceeds it,
// so a cell is scaled until its norm, not its largest value times n^{3/2}, reaches
// 2^60: for a vector that one mode per cell dominates (any smooth one) that is up to
// 4.7 bits more.  Without them the noise in A x of such a vector was 17 times FP64's
// at degree 8 and twice at degree 4, and mixed solves of 48^3 Q4 to 1e-10 could
// stall above it; with them it is below FP64's at every degree.  They cost 3 % of an
// application (27^3 Q5 166 -> 171 us).  The norm comes from 11-bit magnitudes m
// (rounded up) under the exponent E of the cell's largest value: norm < 2^(E - 11)
// sqrt(sum of m^2).  fx_norm_bits: the bits that it takes above 2^(E - 11).
__device__ __forceinline__ int fx_norm_bits(unsigned sum) { return (33 - __clz((int)sum)) >> 1; }

// Shared memory of the two passes in a block of BT threads.
template <int N, int BT>
struct FxSmem {
  static constexpr int C = Cfg<N>::CPB;
  static constexpr int NS = (BT + N * N - 1) / (N * N);  // n^2 thread groups of the block
  static constexpr size_t trace = 8 * C * LinePad<N>::SC + 4 * 3 * NS;
  static constexpr size_t cell =
      8 * 2 * C * LinePad<N>::SC + 8 * 6 * C + 4 * (13 * C + 2 * NS);
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

// -2^61 - 2^29 <= t < 2^61 - 2^29.  Who calls it: values below 2^60 (face
// coefficients, metric terms, derivatives and traces, eigenbases), sums brought
// down to that, and line operator entries, whose row sums are at most 2^61 in
// three directions together.
__device__ __forceinline__ FxPair fx_pair(long long t) {
  const int h = (int)((t + (1ll << 29)) >> 30);
  return {h, (int)(t - ((long long)h << 30))};
}

__device__ __forceinline__ long long fx_shift(long long v, int s) {  // v 2^s, |s| < 64
  return s >= 0 ? v << s : v >> -s;
}

// v 2^-s to nearest, 0 <= s < 63
__device__ __forceinline__ long long fx_round(long long v, int s) {
  return (v + ((1ll << s) >> 1)) >> s;
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

// d 2^k, v 2^k
__device__ __forceinline__ double fx_scale(double d, int k) {
  if (k > 900 || k < -900) return scalbn(d, k);
  return d != 0.0 ? __hiloint2double(__double2hiint(d) + (int)((unsigned)k << 20),
                                     __double2loint(d))
                  : 0.0;
}
__device__ __forceinline__ double fx_to_double(long long v, int k) {
  return fx_scale((double)v, k);
}

// magnitude's high word, for fx_bits of a maximum
__device__ __forceinline__ unsigned fx_mag_hi(long long v) {
  return (unsigned)((unsigned long long)(v < 0 ? ~v : v) >> 32);
}
// smallest b >= 32 with every magnitude below 2^b
__device__ __forceinline__ int fx_bits(unsigned mag_hi) { return 64 - __clz((int)mag_hi); }

// Largest v, or the sum of v, over the threads of the calling thread's cell.
// Cells that lie inside one warp need no barrier and take shuffles (a reduction
// instruction runs once per cell of the warp: 64^3 Q3 464 against 435 us, 100^3 Q1
// 368 against 273); otherwise slots (zeroed before an earlier barrier) collects the
// warps' results.  Every thread of the block calls it.
template <int N, int BT, bool SUM>
__device__ __forceinline__ unsigned fx_cell_reduce(unsigned v, int lc, unsigned* slots) {
  constexpr int N2 = N * N;
  if constexpr (32 % N2 == 0) {
#pragma unroll
    for (int off = N2 / 2; off > 0; off >>= 1) {
      const unsigned o = __shfl_xor_sync(0xffffffffu, v, off);
      v = SUM ? v + o : max(v, o);
    }
    return v;
  }
  const int lane = threadIdx.x & 31, base = (int)threadIdx.x - lane;
  const int lo = lc * N2 > base ? lc * N2 - base : 0;
  int hi = (lc + 1) * N2 - base;
  const int lanes = BT - base < 32 ? BT - base : 32;
  if (hi > lanes) hi = lanes;
  const unsigned mask = (hi >= 32 ? 0xffffffffu : (1u << hi) - 1u) & ~((1u << lo) - 1u);
  v = SUM ? __reduce_add_sync(mask, v) : __reduce_max_sync(mask, v);
  if (lane == lo) {
    if (SUM)
      atomicAdd(slots + lc, v);
    else
      atomicMax(slots + lc, v);
  }
  __syncthreads();
  return slots[lc];
}
template <int N, int BT>
__device__ __forceinline__ unsigned fx_cell_max(unsigned v, int lc, unsigned* slots) {
  return fx_cell_reduce<N, BT, false>(v, lc, slots);
}

// k with cell 2-norm of x 2^k below 2^60, for |x| < 2^E.  The upper halves, with
// their exponents moved, are FP32 numbers in [0, 2^11] that are at most 2^-20
// below x 2^(11 - E); a thread's squares are added in FP32, with a margin for that
// and for its roundings, and the cell's in integers (at most 2^31.6).
template <int N, int BT>
__device__ __forceinline__ int fx_norm_scale(const double (&x)[N], int E, int lc,
                                             unsigned* slots) {
  float sum = 0.0f;
#pragma unroll
  for (int l = 0; l < N; ++l) {
    // subnormal numbers count as 2^11
    const int t = min((int)(fx_abs_hi(x[l]) - ((unsigned)(E + 885) << 20)), 138 << 20);
    const float f = __int_as_float(max(t, 0) << 3);
    sum = fmaf(f, f, sum);
  }
  const unsigned m = __float2uint_ru(sum * (1.0f + 0x1p-16f)) + 1u;
  return 71 - E - fx_norm_bits(fx_cell_reduce<N, BT, true>(m, lc, slots));
}
// The same for integers below 2^b: the shift that brings the cell's norm below
// 2^60, from the upper halves (b >= 32; those below 2^43 are taken as they are).
template <int N, int BT>
__device__ __forceinline__ int fx_norm_shift(const long long (&r)[N], int b, int lc,
                                             unsigned* slots) {
  b = max(b, 43);
  unsigned sum = 0;
#pragma unroll
  for (int l = 0; l < N; ++l) {
    const unsigned m = (fx_mag_hi(r[l]) >> (b - 43)) + 1u;
    sum += m * m;
  }
  return 71 - b - fx_norm_bits(fx_cell_reduce<N, BT, true>(sum, lc, slots));
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

// g[f] = sum_a Dh[f][a] u[a]  2^-cD
template <int N>
__device__ __forceinline__ void fx_deriv(const DGTabXGrad& t, const long long (&u)[N],
                                         long long (&g)[N]) {
  constexpr int H = N / 2, P = (N + 1) / 2;
  FxVal e[P], o[H];
#pragma unroll
  for (int a = 0; a < H; ++a) {
    e[a] = fx_split(u[a] + u[N - 1 - a]);
    o[a] = fx_split(u[a] - u[N - 1 - a]);
  }
  if (N % 2 == 1) e[P - 1] = fx_split(u[H]);
#pragma unroll
  for (int f = 0; f < P; ++f) {
    FxAcc Q = fx_zero();
#pragma unroll
    for (int a = 0; a < H; ++a) fx_mac(Q, t.Do[f][a], o[a]);
    const long long q = fx_value(Q);
    if (f == N - 1 - f) {
      g[f] = q;
    } else {
      FxAcc E = fx_zero();
#pragma unroll
      for (int a = 0; a < P; ++a) fx_mac(E, t.De[f][a], e[a]);
      const long long p = fx_value(E);
      g[f] = q + p;
      g[N - 1 - f] = q - p;
    }
  }
}

// ---------------------------------------------------------------------------
// The two passes (dg_fixed.cu), as functions of a block over a group of cells.
// ---------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ void fx_store_traces(const DGTabX& t, const long long (&u)[N],
                                                long long* __restrict__ tr, int dir, int pt) {
  constexpr int N2 = N * N, H = N / 2;
  FxAcc ve = fx_zero(), vo = fx_zero(), ae = fx_zero(), ao = fx_zero();
#pragma unroll
  for (int a = 0; a < H; ++a) {
    const FxVal e = fx_split(u[a] + u[N - 1 - a]), o = fx_split(u[a] - u[N - 1 - a]);
    fx_mac(ve, t.ve[a], e);
    fx_mac(ae, t.ae[a], e);
    fx_mac(vo, t.vo[a], o);
    fx_mac(ao, t.ao[a], o);
  }
  if (N % 2 == 1) {
    const FxVal e = fx_split(u[H]);
    fx_mac(ve, t.ve[H], e);
    fx_mac(ae, t.ae[H], e);
  }
  const long long v = fx_value(ve), w = fx_value(vo), a = fx_value(ae), b = fx_value(ao);
  tr[(4 * dir + 0) * N2 + pt] = v + w;  // lower face
  tr[(4 * dir + 1) * N2 + pt] = a + b;
  tr[(4 * dir + 2) * N2 + pt] = v - w;  // upper face
  tr[(4 * dir + 3) * N2 + pt] = b - a;
}

// Where pass 1 takes the vector from and pass 2 puts the result: functions of
// the DOF index, called once per DOF by the thread that owns it there.
struct FxLoad {
  const double* x;
  __device__ __forceinline__ void begin() const {}
  __device__ __forceinline__ double operator()(long long i) const { return x[i]; }
};
struct FxStore {
  double* y;
  __device__ __forceinline__ void operator()(long long i, double v) const { y[i] = v; }
};

// Pass 1 over the cells c0 .. c0+nblk-1 (nblk <= CPB) by the calling block of
// BT threads (at least CPB n^2; the others only take part in the barriers).
// smem: FxSmem<N, BT>::trace bytes.  Every thread of the block calls it; a
// barrier must follow before smem is used again.
// mark: the cells' marks of the vector (point basis).
template <int N, bool MODAL, int BT, typename XL>
__device__ __forceinline__ void fx_trace_cells(const XL& x, long long* __restrict__ U,
                                               long long* __restrict__ TR,
                                               int* __restrict__ expU, int* __restrict__ mark,
                                               long long c0, int nblk,
                                               const DGTabX& tab, long long* smem) {
  constexpr int C = Cfg<N>::CPB, N2 = N * N, N3 = N * N * N;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC;
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + lc;
  const bool live = BT <= Cfg<N>::THREADS || lc < C;
  long long* sc = smem + (live ? lc : 0) * SC;
  unsigned* slots = reinterpret_cast<unsigned*>(smem + C * SC);
  constexpr int NS = FxSmem<N, BT>::NS;
  if (32 % N2 != 0) {
    if (threadIdx.x < 3 * NS) slots[threadIdx.x] = 0;
    cell_sync<N>();
  }
  double xv[N];
  unsigned big = 0;
#pragma unroll
  for (int l = 0; l < N; ++l) {
    xv[l] = active ? x(c * N3 + l * N2 + q * N + p) : 0.0;
    const unsigned m = fx_abs_hi(xv[l]);
    big = m > big ? m : big;
  }
  const int E = fx_exponent(fx_cell_max<N, BT>(big, lc, slots));
  const bool zsmall = (int)(big >> 20) < E + 1016;  // the z-line is below 2^(E - 7)
  long long v[N], u[N];
  int eu;  // u[] 2^eu
  if (MODAL) {
    const int k = fx_norm_scale<N, BT>(xv, E, lc, slots + 2 * NS);
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = fx_from_double(xv[l], k, E);
    // along z: thread owns (i = p, j = q)
    fx_fwd<N>(tab, v, u);
#pragma unroll
    for (int e = 0; e < N; ++e)
      if (live) sc[e * SZ + q * SY + p] = u[e];
    cell_sync<N>();
    // along y: (i = p, e = q)
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = sc[q * SZ + j * SY + p];
    fx_fwd<N>(tab, v, u);
#pragma unroll
    for (int b = 0; b < N; ++b)
      if (live) sc[q * SZ + b * SY + p] = u[b];
    cell_sync<N>();
    // along x: (b = p, e = q)
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = sc[q * SZ + p * SY + i];
    fx_fwd<N>(tab, v, u);
    // the largest point value to [2^59, 2^60)
    big = 0;
#pragma unroll
    for (int a = 0; a < N; ++a) {
      const unsigned m = fx_mag_hi(u[a]);
      big = m > big ? m : big;
    }
    const int up = 60 - fx_bits(fx_cell_max<N, BT>(big, lc, slots + NS));
#pragma unroll
    for (int a = 0; a < N; ++a) {
      u[a] = fx_shift(u[a], up);
      if (live) sc[q * SZ + p * SY + a] = u[a];
    }
    eu = -k - up;
    if (active) fx_store_traces<N>(tab, u, TR + c * (12 * N2), 0, pt);
  } else {
#pragma unroll
    for (int l = 0; l < N; ++l) {
      u[l] = fx_from_double(xv[l], 60 - E, E);
      if (live) sc[l * SZ + q * SY + p] = u[l];
    }
    eu = E - 60;
  }
  if (E == FX_NAN) eu = FX_NAN;
  if (active && pt == 0) {
    expU[c] = eu;
    if (!MODAL) mark[c] = 0;
  }
  cell_sync<N>();
  if (!active) return;  // no barrier follows
  long long* tr = TR + c * (12 * N2);
  // whether a line's largest value is below 2^53, the cell's at least 2^59
  auto small = [](const long long (&w)[N]) {
    int m = 0;
#pragma unroll
    for (int e = 0; e < N; ++e) m |= (int)(w[e] >> 32) ^ (int)(w[e] >> 63);
    return m < 1 << 21;
  };
  int marks = 0;
  if (MODAL) {
#pragma unroll
    for (int e = 0; e < N; ++e) {
      u[e] = sc[e * SZ + q * SY + p];
      U[c * N3 + e * N2 + q * N + p] = u[e];
    }
  } else {
#pragma unroll
    for (int a = 0; a < N; ++a) v[a] = sc[q * SZ + p * SY + a];
    fx_store_traces<N>(tab, v, tr, 0, pt);
    marks = (small(v) ? 1 : 0) | (zsmall ? 4 : 0);
  }
  fx_store_traces<N>(tab, u, tr, 2, pt);
#pragma unroll
  for (int b = 0; b < N; ++b) v[b] = sc[q * SZ + b * SY + p];
  fx_store_traces<N>(tab, v, tr, 1, pt);
  if (!MODAL) {
    if (small(v)) marks |= 2;
    if (marks != 0 && E > -1042) atomicOr(mark + c, marks);  // E: the cell is not zero
  }
}

// What fx_cells_wide reads: h w_q K, h gamma [c][6], the marks of the vector, the
// FP64 tables of the scaled point basis.
struct FxWide {
  const double *kt, *gh;
  const int* mark;
  const DGTabN<double>* tn;
};

// Pass 2 in FP64 for the marked cells of a block (bit k of cells: c0 + k): y = sum
// over the directions of Dh^T (h K . Dh x) and the face terms, from x itself.
// Returns the thread's part of <x, A x> over these cells.  Every thread of the block
// calls it.  A chain of FP64 instructions is what a block with one marked cell waits
// for, so the n^2-thread groups of the block take a cell's three directions side by
// side (Kronecker solves in this basis, whose directions mark a few cells in most
// iterations, 12^3 Q4: 40.3 ms, one direction after the other 44.0, no cell marked
// 37.4).  Kept out of line, so that the fixed-point path keeps its registers.
template <int N, int BT>
__device__ __noinline__ double fx_cells_wide(const double* x, const double* kt, const double* gh,
                                             const DGTabN<double>* tn, double* y, long long c0,
                                             unsigned cells, int Nc, double* smem) {
  constexpr int C = Cfg<N>::CPB, N2 = N * N, N3 = N * N * N;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC;
  constexpr int ROOM = C / 2;  // cells at a time: x and the three directions' sums
  constexpr double sigma = 2.0 * N * N;
  const DGTabN<double>& t = *tn;
  const int group = threadIdx.x / N2, pt = threadIdx.x - group * N2;
  const int p = pt % N, q = pt / N;
  const unsigned nu = (unsigned)Nc;
  const double iw = t.isw[p] * t.isw[p] * (t.isw[q] * t.isw[q]);
  const int count = __popc(cells);
  auto cell = [&](int k) {  // the k-th marked one
    unsigned m = cells;
    for (; k > 0; --k) m &= m - 1;
    return c0 + (__ffs((int)m) - 1);
  };
  double dot = 0.0;
  for (int first = 0; first < count; first += ROOM) {
    const int here = min(count - first, ROOM);
    __syncthreads();
    for (int i = threadIdx.x; i < here * N3; i += BT) {
      const int k = i / N3, o = i - k * N3, e = o / N2, r = o - e * N2;
      const long long c = cell(first + k);
      smem[4 * k * SC + e * SZ + (r / N) * SY + r % N] = x[c * N3 + o];
    }
    __syncthreads();
    for (int task = group < C ? group : 3 * here; task < 3 * here; task += C) {
      const int k = task / 3, dir = task - 3 * k;
      const long long c = cell(first + k);
      const double* su = smem + 4 * k * SC;
      double* sr = smem + (4 * k + 1 + dir) * SC;
      // the thread's line: points at + f step of the cell, at2 + f step2 in smem
      const int at = dir == 2 ? pt : dir == 1 ? q * N2 + p : q * N2 + p * N;
      const int step = dir == 2 ? N2 : dir == 1 ? N : 1;
      const int at2 = dir == 2 ? q * SY + p : dir == 1 ? q * SZ + p : q * SZ + p * SY;
      const int step2 = dir == 2 ? SZ : dir == 1 ? SY : 1;
      const unsigned row = (unsigned)c / nu;
      const int at_dir = dir == 0   ? (int)((unsigned)c - row * nu)
                         : dir == 1 ? (int)(row % nu)
                                    : (int)(row / nu);
      const long long stride = dir == 0 ? 1 : dir == 1 ? Nc : (long long)Nc * Nc;
      double F[N], cv[2], cd[2];
      {
        double u[N], v0 = 0.0, v1 = 0.0, q0 = 0.0, q1 = 0.0;
#pragma unroll
        for (int f = 0; f < N; ++f) {
          u[f] = su[at2 + f * step2];
          // end values and outward half derivatives
          v0 = fma(t.l0[f], u[f], v0);
          v1 = fma(t.l1[f], u[f], v1);
          q0 = fma(-t.hdl0[f], u[f], q0);
          q1 = fma(t.hdl1[f], u[f], q1);
        }
#pragma unroll
        for (int f = 0; f < N; ++f) {
          double g = 0.0;
#pragma unroll
          for (int j = 0; j < N; ++j) g = fma(t.Dh[f][j], u[j], g);
          F[f] = kt[c * N3 + at + f * step] * (iw * (t.isw[f] * t.isw[f])) * g;
        }
#pragma unroll
        for (int up = 0; up < 2; ++up) {
          double J = up ? v1 : v0, S = 2.0 * (up ? q1 : q0), once = 2.0;
          if (up ? at_dir < Nc - 1 : at_dir > 0) {
            const double* xn = x + (up ? c + stride : c - stride) * N3 + at;
            double vn = 0.0, qn = 0.0;  // its outward direction is the opposite one
#pragma unroll
            for (int f = 0; f < N; ++f) {
              const double w = xn[f * step];
              vn = fma(up ? t.l0[f] : t.l1[f], w, vn);
              qn = fma(up ? t.hdl0[f] : -t.hdl1[f], w, qn);
            }
            J -= vn;
            S = (up ? q1 : q0) + qn;
            once = 1.0;
          }
          const double g = gh[c * 6 + 2 * dir + up];
          cv[up] = g * (sigma * J - S);
          cd[up] = g * once * J;
        }
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        double r = t.l0[i] * cv[0];
        r = fma(t.hdl0[i], cd[0], r);
        r = fma(t.l1[i], cv[1], r);
        r = fma(-t.hdl1[i], cd[1], r);
#pragma unroll
        for (int f = 0; f < N; ++f) r = fma(t.Dh[f][i], F[f], r);
        sr[at2 + i * step2] = r;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < here * N3; i += BT) {
      const int k = i / N3, o = i - k * N3, e = o / N2, r = o - e * N2;
      const long long c = cell(first + k);
      const double* sx = smem + 4 * k * SC + e * SZ + (r / N) * SY + r % N;
      const double v = (sx[3 * SC] + sx[2 * SC]) + sx[SC];
      y[c * N3 + o] = v;
      dot = fma(sx[0], v, dot);
    }
  }
  return dot;
}

__device__ __forceinline__ void fx_prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Pass 2 over the cells c0 .. c0+nblk-1, called like pass 1; smem:
// FxSmem<N, BT>::cell bytes.  xU: MODAL: the point values of pass 1 (integers);
// otherwise the vector itself, with FX_WIDE added to expM in the marked cells, and
// wd.  DOT: returns the thread's part of <x, A x>, formed from the point values and
// the sum r before Q^T (Q is orthogonal).
template <int N, bool MODAL, int BT, bool DOT = false>
__device__ __forceinline__ double fx_cell_cells(
    const void* xU, const long long* TR, const int* expU, const FxPair* __restrict__ lineop,
    const FxPair* __restrict__ gam, const int* __restrict__ expM, const int* __restrict__ expG,
    const FxWide wd, const FxStore y, long long c0, int nblk, int Nc, const DGTabX& tab,
    long long* smem) {
  constexpr int C = Cfg<N>::CPB, N2 = N * N, N3 = N * N * N, NP = N * (N + 1) / 2;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC;
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const bool live = BT <= Cfg<N>::THREADS || lc < C;
  const long long c = c0 + (active ? lc : 0);
  long long* su = smem + (live ? lc : 0) * SC;
  long long* sr = su + C * SC;
  FxPair(*sg)[6] = reinterpret_cast<FxPair(*)[6]>(smem + 2 * C * SC);  // face coefficients
  // exponents: six faces, own terms, the faces of neighbours with small lines
  int(*sexp)[13] = reinterpret_cast<int(*)[13]>(sg + C);
  unsigned* slots = reinterpret_cast<unsigned*>(sexp + C);
  // the block's operators to L2, while exponents and vectors arrive (odd sizes
  // would leave the 16-byte grid)
  if (NP * N2 % 2 == 0 && threadIdx.x == 0)
    fx_prefetch_l2(lineop + c0 * (3 * NP * N2), nblk * (3 * NP * N2) * 8);
  // cell coordinates: 32-bit divisions (n_cells <= 1024)
  const unsigned nu = (unsigned)Nc;
  const long long stride[3] = {1, Nc, (long long)Nc * Nc};
  // exponents of the seven contributions to a cell
  const unsigned row = (unsigned)c / nu;
  const int crd[3] = {(int)((unsigned)c - row * nu), (int)(row % nu), (int)(row / nu)};
  if (active) {
    for (int f = pt; f < 7; f += N2) {
      int e;
      if (f == 6) {
        e = expU[c] + expM[c];
        if (!MODAL && wd.mark[c] == FX_MARKS) e += FX_WIDE;
      } else {
        const int d = f >> 1, cd = d == 0 ? crd[0] : d == 1 ? crd[1] : crd[2];
        const long long st = d == 0 ? stride[0] : d == 1 ? stride[1] : stride[2];
        e = (f & 1 ? cd < Nc - 1 : cd > 0) ? expU[f & 1 ? c + st : c - st] + expG[c * 6 + f]
                                           : -4 * FX_NAN;
        sg[lc][f] = gam[c * 6 + f];
        if (!MODAL)  // an absent neighbour's own mark: the coefficient is zero
          sexp[lc][7 + f] = wd.mark[f & 1 ? (cd < Nc - 1 ? c + st : c) : (cd > 0 ? c - st : c)] &
                                    (1 << d)
                                ? e
                                : -4 * FX_NAN;
      }
      sexp[lc][f] = e;
    }
  }
  if (MODAL && 32 % N2 != 0 && threadIdx.x < 2 * FxSmem<N, BT>::NS) slots[threadIdx.x] = 0;
  if (!MODAL && threadIdx.x == 0) slots[0] = 0;  // the cells of the block applied in FP64
  long long u[N], r[N];
  // z-lines (a = p, b = q)
#pragma unroll
  for (int e = 0; e < N; ++e) {
    const long long at = c * N3 + e * N2 + q * N + p;
    u[e] = MODAL ? static_cast<const long long*>(xU)[at]
                 : __double_as_longlong(static_cast<const double*>(xU)[at]);
  }
  // their operators too, where the registers allow it (measured at 64^3 Q3:
  // 336 against 340 us; 40^3 Q4: 172 against 178 us; from n = 6 on it is slower)
  constexpr bool PRE = N == 4 || N == 5;
  FxPair Mz[PRE ? NP : 1];
  if constexpr (PRE) {
#pragma unroll
    for (int k = 0; k < NP; ++k) Mz[k] = lineop[((c * 3 + 2) * NP + k) * N2 + pt];
  }
  __syncthreads();  // the block's: its warps start on neighbouring cells together
  const int eown = sexp[active ? lc : 0][6];
  int eout = eown;
#pragma unroll
  for (int f = 0; f < 6; ++f) eout = max(eout, sexp[active ? lc : 0][f] + tab.bump);
  const bool bad = eout >= FX_NAN / 2;
  bool wide = false;
  if (!MODAL) {
    int enb = eown;
#pragma unroll
    for (int f = 7; f < 13; ++f) enb = max(enb, sexp[active ? lc : 0][f] + tab.bump);
    wide = active && !bad && (eown >= FX_WIDE / 2 || enb - eown > 9);
    if (wide && pt == 0) atomicOr(slots, 1u << lc);
  }
  for (int f = pt; f < 6; f += N2) {
    if (!active) break;
    const int down = min(eout - sexp[lc][f], 63);
    const FxPair g = sg[lc][f];
    sg[lc][f] = sexp[lc][f] == -4 * FX_NAN
                    ? FxPair{0, 0}
                    : fx_pair((((long long)g.h << 30) + g.l) >> down);
  }
  {
    const int down = min(eout - eown, 63);
    if (!MODAL) {
      const int E = (active ? expU[c] : 0) + 60;
#pragma unroll
      for (int e = 0; e < N; ++e) u[e] = fx_from_double(__longlong_as_double(u[e]), 60 - E, E);
    }
#pragma unroll
    for (int e = 0; e < N; ++e) {
      u[e] >>= down;
      if (live) su[e * SZ + q * SY + p] = u[e];
    }
  }
  __syncthreads();
  // r (= or +=) the line's terms: |r| < 2^62.3 in the end
  auto line = [&](int dir, bool first) {
    const FxPair* Mp = lineop + ((c * 3 + dir) * NP) * N2 + pt;
    FxPair Mv[PRE ? NP : 1];
    if constexpr (PRE) {
#pragma unroll
      for (int k = 0; k < NP; ++k) Mv[k] = dir == 2 ? Mz[k] : Mp[k * N2];
    }
    // absent neighbours: any value times a zero coefficient
    const long long* t0 =
        TR + (crd[dir] > 0 ? c - stride[dir] : c) * (12 * N2) + (4 * dir + 2) * N2 + pt;
    const long long* t1 =
        TR + (crd[dir] < Nc - 1 ? c + stride[dir] : c) * (12 * N2) + (4 * dir) * N2 + pt;
    const FxVal v0 = fx_split(t0[0]), a0 = fx_split(t0[N2]);
    const FxVal v1 = fx_split(t1[0]), a1 = fx_split(t1[N2]);
    FxVal us[N];
#pragma unroll
    for (int e = 0; e < N; ++e) us[e] = fx_split(u[e]);
    FxAcc R[N];
#pragma unroll
    for (int e = 0; e < N; ++e) R[e] = fx_zero();
#pragma unroll
    for (int e = 0; e < N; ++e) {
#pragma unroll
      for (int f = e; f < N; ++f) {
        const FxPair m = PRE ? Mv[PRE ? packed<N>(e, f) : 0] : Mp[packed<N>(e, f) * N2];
        fx_mac(R[e], m, us[f]);
        if (f != e) fx_mac(R[f], m, us[e]);
      }
    }
    const FxPair g0 = sg[active ? lc : 0][2 * dir], g1 = sg[active ? lc : 0][2 * dir + 1];
    FxAcc A0 = fx_zero(), B0 = fx_zero(), A1 = fx_zero(), B1 = fx_zero();
    fx_mac(A0, g0, a0);
    fx_mac(B0, g0, v0);
    fx_mac(A1, g1, a1);
    fx_mac(B1, g1, v1);
    const long long al0 = fx_value(A0), be0 = fx_value(B0), al1 = fx_value(A1),
                    be1 = fx_value(B1);
    const FxVal ad = fx_split(al0 - al1), as = fx_split(al0 + al1);
    const FxVal bs = fx_split(be0 + be1), bd = fx_split(be0 - be1);
#pragma unroll
    for (int a = 0; a < (N + 1) / 2; ++a) {
      FxAcc Pe = fx_zero();
      fx_mac(Pe, tab.le[a], ad);
      fx_mac(Pe, tab.de[a], bs);
      const long long pe = fx_value(Pe);
      if (a == N - 1 - a) {
        r[a] = first ? pe : r[a] + pe;
      } else {
        FxAcc Po = fx_zero();
        fx_mac(Po, tab.lo[a], as);
        fx_mac(Po, tab.dn[a], bd);
        const long long po = fx_value(Po);
        r[a] = first ? pe + po : r[a] + (pe + po);
        r[N - 1 - a] = first ? pe - po : r[N - 1 - a] + (pe - po);
      }
    }
#pragma unroll
    for (int e = 0; e < N; ++e) r[e] += fx_value(R[e]);
  };
  line(2, true);
#pragma unroll
  for (int e = 0; e < N; ++e)
    if (live) sr[e * SZ + q * SY + p] = r[e];
  cell_sync<N>();
  // y-lines (a = p, e = q)
#pragma unroll
  for (int b = 0; b < N; ++b) {
    u[b] = su[q * SZ + b * SY + p];
    r[b] = sr[q * SZ + b * SY + p];
  }
  line(1, false);
#pragma unroll
  for (int b = 0; b < N; ++b)
    if (live) sr[q * SZ + b * SY + p] = r[b];
  cell_sync<N>();
  // x-lines (b = p, e = q): the sum of all three directions
#pragma unroll
  for (int a = 0; a < N; ++a) {
    u[a] = su[q * SZ + p * SY + a];
    r[a] = sr[q * SZ + p * SY + a];
  }
  line(0, false);
  // u r / 2^60 in units 2^(eout - expM) 2^(eout - 1); r, below 2^62.3, three
  // bits down
  double dot = 0.0;
  if constexpr (DOT) {
    if (active) {
      FxAcc A = {0, 0};
#pragma unroll
      for (int a = 0; a < N; ++a) fx_mac(A, fx_pair(r[a] >> 3), fx_split(u[a]));
      dot = fx_scale(fma((double)A.m, 0x1p-30, (double)A.h), 2 * eout - expM[c] + 62);
    }
  }
  const double qnan = __longlong_as_double(0x7ff8000000000000ll);
  if (!MODAL) {
#pragma unroll
    for (int a = 0; a < N; ++a)
      if (live)
        sr[q * SZ + p * SY + a] =
            __double_as_longlong(bad ? qnan : fx_to_double(r[a], eout - 1));
    cell_sync<N>();
    if (active && !wide) {  // written from the z-lines: consecutive lanes, consecutive words
#pragma unroll
      for (int e = 0; e < N; ++e)
        y(c * N3 + e * N2 + q * N + p, __longlong_as_double(sr[e * SZ + q * SY + p]));
    }
    if (slots[0] != 0) {
      if (wide) dot = 0.0;
      dot += fx_cells_wide<N, BT>(static_cast<const double*>(xU), wd.kt, wd.gh, wd.tn, y.y, c0,
                                  slots[0], Nc, reinterpret_cast<double*>(smem));
    }
    return DOT && bad ? qnan : dot;
  }
  // the sum to a cell 2-norm of at most 2^60, then Q^T
  unsigned big = 0;
#pragma unroll
  for (int a = 0; a < N; ++a) {
    const unsigned m = fx_mag_hi(r[a]);
    big = m > big ? m : big;
  }
  const int up = fx_norm_shift<N, BT>(r, fx_bits(fx_cell_max<N, BT>(big, lc, slots)), lc,
                                      slots + FxSmem<N, BT>::NS);
#pragma unroll
  for (int a = 0; a < N; ++a) r[a] = fx_shift(r[a], up);
  fx_bwd<N>(tab, r, u);
#pragma unroll
  for (int i = 0; i < N; ++i)
    if (live) su[q * SZ + p * SY + i] = u[i];
  cell_sync<N>();
  // y: (i = p, e = q)
#pragma unroll
  for (int b = 0; b < N; ++b) r[b] = su[q * SZ + b * SY + p];
  fx_bwd<N>(tab, r, u);
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (live) su[q * SZ + j * SY + p] = u[j];
  cell_sync<N>();
  // z: (i = p, j = q)
#pragma unroll
  for (int e = 0; e < N; ++e) r[e] = su[e * SZ + q * SY + p];
  fx_bwd<N>(tab, r, u);
  if (active) {
#pragma unroll
    for (int l = 0; l < N; ++l)
      y(c * N3 + l * N2 + q * N + p, bad ? qnan : fx_to_double(u[l], eout - 1 - up));
  }
  return DOT && bad ? qnan : dot;
}

}  // namespace dgk
