// The FP64 operator in block fixed-point arithmetic (dg_fixed.cuh): two passes
// in the scaled Gauss-point basis (dg_nodal.cu), for vectors in that basis
// (Q A Q^T) and, with the orthogonal transforms Q and Q^T fused into the
// passes, for vectors of Legendre coefficients (A).
//
// Pass 1, per cell: the vector becomes 64-bit integers under one exponent (its
// largest magnitude), goes to point values, is brought up to the full range
// again, and leaves the face data its neighbours need: on each face the value v
// and the combination the neighbour's flux takes (sigma v + d on the lower face,
// d - sigma v on the upper one, d half the normal derivative).
// Pass 2, per cell: every line adds M u, M its precomputed operator (volume term
// and own-side face terms), and the neighbours' face terms; for Legendre
// coefficients the sum is brought up to the full range once more and
// transformed back; FP64 values leave.
//
// Every coefficient has its own scale: the line operators of a cell share an
// exponent, each face coefficient has one, and pass 2 brings the products to
// the largest exponent among its cell's own and its six neighbours' terms.  What
// is shifted out is below 2^-59 of the largest term.  A NaN or an infinity in a
// cell gives NaN in that cell and its face neighbours.
//
// Layouts: U[c][point] (integers), TR[c][6 faces][v, combination][n^2] as the FP64
// pass; line operators [c][x,y,z][packed entry][line], so that the lanes of a
// warp read consecutive words.
#include "dg_fixed.cuh"

namespace dgk {

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

template <int N, bool MODAL>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_trace_fx(const double* __restrict__ x, long long* __restrict__ U, long long* __restrict__ TR,
           int* __restrict__ expU, long long cbeg, long long cend, const int* __restrict__ skip,
           const __grid_constant__ DGTabX tab) {
  constexpr int C = Cfg<N>::CPB, N2 = N * N, N3 = N * N * N;
  constexpr int SY = FxPad<N>::SY, SZ = FxPad<N>::SZ, SC = FxPad<N>::SC;
  if (skip != nullptr && *skip) return;
  __shared__ long long s[C * SC];
  __shared__ unsigned slots[2][C];
  const long long c0 = cbeg + (long long)blockIdx.x * C;
  const int nblk = (int)((cend - c0) < C ? (cend - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + lc;
  long long* sc = s + lc * SC;
  if (32 % N2 != 0) {
    if (threadIdx.x < C) slots[0][threadIdx.x] = slots[1][threadIdx.x] = 0;
    __syncthreads();
  }
  double xv[N];
  unsigned big = 0;
#pragma unroll
  for (int l = 0; l < N; ++l) {
    xv[l] = active ? x[c * N3 + l * N2 + q * N + p] : 0.0;
    const unsigned m = fx_abs_hi(xv[l]);
    big = m > big ? m : big;
  }
  const int E = fx_exponent(fx_cell_max<N>(big, lc, slots[0]));
  long long v[N], u[N];
  int eu;  // u[] 2^eu
  if (MODAL) {
    constexpr int S0 = FxScale<N>::S0;
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = fx_from_double(xv[l], S0 - E, E);
    // along z: thread owns (i = p, j = q)
    fx_fwd<N>(tab, v, u);
#pragma unroll
    for (int e = 0; e < N; ++e) sc[e * SZ + q * SY + p] = u[e];
    __syncthreads();
    // along y: (i = p, e = q)
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = sc[q * SZ + j * SY + p];
    fx_fwd<N>(tab, v, u);
#pragma unroll
    for (int b = 0; b < N; ++b) sc[q * SZ + b * SY + p] = u[b];
    __syncthreads();
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
    const int up = 60 - fx_bits(fx_cell_max<N>(big, lc, slots[1]));
#pragma unroll
    for (int a = 0; a < N; ++a) {
      u[a] = fx_shift(u[a], up);
      sc[q * SZ + p * SY + a] = u[a];
    }
    eu = E - S0 - up;
    if (active) fx_store_traces<N>(tab, u, TR + c * (12 * N2), 0, pt);
  } else {
#pragma unroll
    for (int l = 0; l < N; ++l) {
      u[l] = fx_from_double(xv[l], 60 - E, E);
      sc[l * SZ + q * SY + p] = u[l];
    }
    eu = E - 60;
  }
  if (E == FX_NAN) eu = FX_NAN;
  if (active && pt == 0) expU[c] = eu;
  __syncthreads();
  if (!active) return;  // no barrier follows
  long long* tr = TR + c * (12 * N2);
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
  }
  fx_store_traces<N>(tab, u, tr, 2, pt);
#pragma unroll
  for (int b = 0; b < N; ++b) v[b] = sc[q * SZ + b * SY + p];
  fx_store_traces<N>(tab, v, tr, 1, pt);
}

// xU: MODAL: the point values of pass 1 (integers); otherwise the vector itself
template <int N, bool MODAL>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_cell_fx(const void* __restrict__ xU, const long long* __restrict__ TR,
          const int* __restrict__ expU, const FxPair* __restrict__ lineop,
          const FxPair* __restrict__ gam, const int* __restrict__ expM,
          const int* __restrict__ expG, double* __restrict__ y, long long cbeg, long long cend,
          int Nc, const int* __restrict__ skip, const __grid_constant__ DGTabX tab) {
  constexpr int C = Cfg<N>::CPB, N2 = N * N, N3 = N * N * N, NP = N * (N + 1) / 2, H = N / 2;
  constexpr int SY = FxPad<N>::SY, SZ = FxPad<N>::SZ, SC = FxPad<N>::SC;
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  long long* su = reinterpret_cast<long long*>(smem_raw);
  long long* sr = su + C * SC;
  __shared__ unsigned slots[C];
  const long long c0 = cbeg + (long long)blockIdx.x * C;
  const int nblk = (int)((cend - c0) < C ? (cend - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + lc;
  su += lc * SC;
  sr += lc * SC;
  if (MODAL && 32 % N2 != 0 && threadIdx.x < C) slots[threadIdx.x] = 0;
  // cell coordinates: 32-bit divisions (n_cells <= 1024)
  const unsigned cu = (unsigned)(active ? c : c0), nu = (unsigned)Nc;
  const unsigned row = cu / nu;
  const int crd[3] = {(int)(cu - row * nu), (int)(row % nu), (int)(row / nu)};
  const long long stride[3] = {1, Nc, (long long)Nc * Nc};
  // exponents: own terms and each neighbour's, then the common one
  int eown = 0, ef[6], eout = 0;
  if (active) {
    eown = expU[c] + expM[c];
    eout = eown;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int d = f >> 1;
      const bool in = (f & 1) ? crd[d] < Nc - 1 : crd[d] > 0;
      ef[f] = in ? expU[(f & 1) ? c + stride[d] : c - stride[d]] + expG[c * 6 + f]
                 : -4 * FX_NAN;
      eout = max(eout, ef[f] + (in ? tab.bump : 0));
    }
  }
  const bool bad = eout >= FX_NAN / 2;
  long long u[N], r[N];
  if (active) {  // z-lines (a = p, b = q)
    const int down = min(eout - eown, 63);
    const int E = expU[c] + 60;
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const long long at = c * N3 + e * N2 + q * N + p;
      u[e] = MODAL ? static_cast<const long long*>(xU)[at]
                   : fx_from_double(static_cast<const double*>(xU)[at], 60 - E, E);
      u[e] >>= down;
      su[e * SZ + q * SY + p] = u[e];
    }
  }
  // r (= or +=) the line's terms, doubled: |r| < 2^62.3 in the end
  auto line = [&](int dir, bool first) {
    const FxPair* Mp = lineop + ((c * 3 + dir) * NP) * N2 + pt;
    FxVal us[N];
#pragma unroll
    for (int e = 0; e < N; ++e) us[e] = fx_split(u[e]);
    long long al0 = 0, be0 = 0, al1 = 0, be1 = 0;
    auto face = [&](int f, long long cn, long long& al, long long& be) {
      const int down = min(eout - ef[f], 63);
      const long long* tr = TR + cn * (12 * N2) + (2 * (f ^ 1)) * N2 + pt;
      const FxPair g = gam[c * 6 + f];
      FxAcc A = fx_zero(), B = fx_zero();
      fx_mac(B, g, fx_split(tr[0] >> down));
      fx_mac(A, g, fx_split(tr[N2] >> down));
      al = fx_value(A);
      be = fx_value(B);
    };
    if (crd[dir] > 0) face(2 * dir, c - stride[dir], al0, be0);
    if (crd[dir] < Nc - 1) face(2 * dir + 1, c + stride[dir], al1, be1);
    const FxVal ad = fx_split(al0 - al1), as = fx_split(al0 + al1);
    const FxVal bs = fx_split(be0 + be1), bd = fx_split(be0 - be1);
#pragma unroll
    for (int a = 0; a < (N + 1) / 2; ++a) {
      FxAcc Pe = fx_zero<1>();
      fx_mac(Pe, tab.le[a], ad);
      fx_mac(Pe, tab.de[a], bs);
      const long long pe = fx_value<1>(Pe);
      if (a == N - 1 - a) {
        r[a] = first ? pe : r[a] + pe;
      } else {
        FxAcc Po = fx_zero<1>();
        fx_mac(Po, tab.lo[a], as);
        fx_mac(Po, tab.dn[a], bd);
        const long long po = fx_value<1>(Po);
        r[a] = first ? pe + po : r[a] + (pe + po);
        r[N - 1 - a] = first ? pe - po : r[N - 1 - a] + (pe - po);
      }
    }
    FxAcc R[N];
#pragma unroll
    for (int e = 0; e < N; ++e) R[e] = fx_zero<1>();
#pragma unroll
    for (int e = 0; e < N; ++e) {
#pragma unroll
      for (int f = e; f < N; ++f) {
        const FxPair m = Mp[packed<N>(e, f) * N2];
        fx_mac(R[e], m, us[f]);
        if (f != e) fx_mac(R[f], m, us[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < N; ++e) r[e] += fx_value<1>(R[e]);
  };
  if (active) {
    line(2, true);
#pragma unroll
    for (int e = 0; e < N; ++e) sr[e * SZ + q * SY + p] = r[e];
  }
  __syncthreads();
  if (active) {  // y-lines (a = p, e = q)
#pragma unroll
    for (int b = 0; b < N; ++b) {
      u[b] = su[q * SZ + b * SY + p];
      r[b] = sr[q * SZ + b * SY + p];
    }
    line(1, false);
#pragma unroll
    for (int b = 0; b < N; ++b) sr[q * SZ + b * SY + p] = r[b];
  }
  __syncthreads();
  if (active) {  // x-lines (b = p, e = q): the sum of all three directions
#pragma unroll
    for (int a = 0; a < N; ++a) {
      u[a] = su[q * SZ + p * SY + a];
      r[a] = sr[q * SZ + p * SY + a];
    }
    line(0, false);
  }
  const double qnan = __longlong_as_double(0x7ff8000000000000ll);
  if (!MODAL) {
    if (active) {
#pragma unroll
      for (int a = 0; a < N; ++a)
        sr[q * SZ + p * SY + a] = __double_as_longlong(bad ? qnan : fx_to_double(r[a], eout - 1));
    }
    __syncthreads();
    if (active) {  // written from the z-lines: consecutive lanes, consecutive words
#pragma unroll
      for (int e = 0; e < N; ++e)
        y[c * N3 + e * N2 + q * N + p] = __longlong_as_double(sr[e * SZ + q * SY + p]);
    }
    return;
  }
  // the sum to a cell 2-norm of at most 2^60, then Q^T
  unsigned big = 0;
  if (active) {
#pragma unroll
    for (int a = 0; a < N; ++a) {
      const unsigned m = fx_mag_hi(r[a]);
      big = m > big ? m : big;
    }
  }
  const int up = FxScale<N>::S0 - fx_bits(fx_cell_max<N>(big, lc, slots));
  if (active) {
#pragma unroll
    for (int a = 0; a < N; ++a) r[a] = fx_shift(r[a], up);
    fx_bwd<N>(tab, r, u);
#pragma unroll
    for (int i = 0; i < N; ++i) su[q * SZ + p * SY + i] = u[i];
  }
  __syncthreads();
  if (active) {  // y: (i = p, e = q)
#pragma unroll
    for (int b = 0; b < N; ++b) r[b] = su[q * SZ + b * SY + p];
    fx_bwd<N>(tab, r, u);
#pragma unroll
    for (int j = 0; j < N; ++j) su[q * SZ + j * SY + p] = u[j];
  }
  __syncthreads();
  if (active) {  // z: (i = p, j = q)
#pragma unroll
    for (int e = 0; e < N; ++e) r[e] = su[e * SZ + q * SY + p];
    fx_bwd<N>(tab, r, u);
#pragma unroll
    for (int l = 0; l < N; ++l)
      y[c * N3 + l * N2 + q * N + p] = bad ? qnan : fx_to_double(u[l], eout - 1 - up);
  }
}

// Line operators, face coefficients and their exponents from K and h gamma: one
// thread per cell, direction and line.  Integer arithmetic throughout: K in
// units of the cell's largest, h gamma < 2^(1 + exponents of h and K), both to
// 2^-59; products of the 1D tables are constants.
template <int N>
struct FxSetup {
  static constexpr int L = 3 * N * N;                    // lines of a cell
  static constexpr int C = N == 2 ? 12 : N == 3 ? 6 : N == 4 ? 4 : N == 5 ? 2 : 1;
  static constexpr int THREADS = C * L;
};

template <int N>
__global__ void __launch_bounds__(FxSetup<N>::THREADS)
k_lines_fx(const double* __restrict__ K, const double* __restrict__ gh,
           FxPair* __restrict__ lineop, FxPair* __restrict__ gam, int* __restrict__ expM,
           int* __restrict__ expG, long long ncells, int Nc, int cg,
           const __grid_constant__ DGTabXSetup t) {
  constexpr int C = FxSetup<N>::C, L = FxSetup<N>::L, T = FxSetup<N>::THREADS;
  constexpr int N2 = N * N, N3 = N * N * N, NP = N * (N + 1) / 2;
  __shared__ long long sk[C * N3];
  __shared__ unsigned kmax[C];
  __shared__ unsigned long long rmax[C][3];
  __shared__ int sbad[C];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  if (threadIdx.x < C) {
    kmax[threadIdx.x] = 0;
    sbad[threadIdx.x] = 0;
    for (int d = 0; d < 3; ++d) rmax[threadIdx.x][d] = 0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nblk * N3; i += T) {
    const double v = K[c0 * N3 + i];
    sk[i] = __double_as_longlong(v);
    atomicMax(&kmax[i / N3], fx_abs_hi(v));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nblk * N3; i += T) {
    const int E = fx_exponent(kmax[i / N3]);
    sk[i] = fx_from_double(__longlong_as_double(sk[i]), 59 - E, E);
  }
  __syncthreads();
  const int lc = threadIdx.x / L, t2 = threadIdx.x - lc * L;
  const int dir = t2 / N2, pt = t2 - dir * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + lc;
  const int eK = active ? fx_exponent(kmax[lc]) : 0;
  long long M[NP];
  bool bad = eK == FX_NAN;
  if (active) {
    const int step = dir == 0 ? 1 : dir == 1 ? N : N2;
    const int at = lc * N3 + (dir == 0 ? N * (p + N * q) : dir == 1 ? p + N2 * q : p + N * q);
    const unsigned cu = (unsigned)c, nu = (unsigned)Nc;
    const int crd = (int)(dir == 0 ? cu % nu : dir == 1 ? (cu / nu) % nu : cu / nu / nu);
    FxVal k[N];
#pragma unroll
    for (int f = 0; f < N; ++f) k[f] = fx_split(sk[at + f * step]);
    FxVal g[2];
    bool edge[2] = {crd == 0, crd == Nc - 1};
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const double w = gh[c * 6 + 2 * dir + m];
      bad = bad || fx_abs_hi(w) >= 0x7ff00000u;
      const int E = eK + t.ch + 1;
      g[m] = fx_split(fx_from_double(w, 60 - E, E));
      if (pt == 0) {
        // normalised to [2^59, 2^60), taking up the table scales 2^cg
        const double w2 = fx_abs_hi(w) < 0x00100000u ? w * 0x1p64 : w;
        const int e = (int)(fx_abs_hi(w2) >> 20);
        const long long mant = (__double_as_longlong(w2) & 0xfffffffffffffll) | 0x10000000000000ll;
        gam[c * 6 + 2 * dir + m] = w > 0.0 ? fx_pair(mant << 7) : FxPair{0, 0};
        expG[c * 6 + 2 * dir + m] =
            w > 0.0 ? e - 1022 - (fx_abs_hi(w) < 0x00100000u ? 64 : 0) + cg : -2 * FX_NAN;
      }
    }
    unsigned long long rs[N];
#pragma unroll
    for (int e = 0; e < N; ++e) rs[e] = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
      for (int j = i; j < N; ++j) {
        const int ij = packed<N>(i, j), ji = packed<N>(N - 1 - i, N - 1 - j);
        FxAcc A = fx_zero<1>();
#pragma unroll
        for (int f = 0; f < N; ++f) fx_mac(A, t.DD[f][ij], k[f]);
        fx_mac(A, edge[0] ? t.F[1][ij] : t.F[0][ij], g[0]);
        fx_mac(A, edge[1] ? t.F[1][ji] : t.F[0][ji], g[1]);
        const long long v = fx_value<1>(A);
        M[ij] = v;
        const unsigned long long mag = (unsigned long long)(v < 0 ? -v : v) >> 4;
        rs[i] += mag;
        if (i != j) rs[j] += mag;
      }
    }
    unsigned long long R = 0;
#pragma unroll
    for (int e = 0; e < N; ++e) R = rs[e] > R ? rs[e] : R;
    atomicMax(&rmax[lc][dir], R + N);
    if (bad) sbad[lc] = 1;
  }
  __syncthreads();
  if (!active) return;
  // largest row sum over the three directions to (2^59, 2^60]
  const int bits = 68 - __clzll((long long)(rmax[lc][0] + rmax[lc][1] + rmax[lc][2]));
  const int up = 60 - bits;
  if (t2 == 0) expM[c] = sbad[lc] ? FX_NAN : eK + t.cB - up;
  FxPair* out = lineop + ((c * 3 + dir) * NP) * N2 + pt;
#pragma unroll
  for (int k2 = 0; k2 < NP; ++k2) out[k2 * N2] = fx_pair(fx_shift(M[k2], up));
}

template <int N>
struct FixedF {
  static constexpr size_t SMEM = 2 * sizeof(long long) * Cfg<N>::CPB * FxPad<N>::SC;
  template <bool MODAL>
  static cudaError_t pass(const dg_mesh* m, int pass, const double* x, double* y, long long cbeg,
                          long long cend, const int* skip, cudaStream_t s) {
    if (cend <= cbeg) return cudaSuccess;
    const unsigned blocks = (unsigned)((cend - cbeg + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    long long* U = reinterpret_cast<long long*>(m->U64);
    long long* TR = reinterpret_cast<long long*>(m->TR64);
    if (pass == 1)
      k_trace_fx<N, MODAL><<<blocks, Cfg<N>::THREADS, 0, s>>>(x, U, TR, m->expU, cbeg, cend, skip,
                                                             m->tabX);
    else
      k_cell_fx<N, MODAL><<<blocks, Cfg<N>::THREADS, SMEM, s>>>(
          MODAL ? (const void*)U : (const void*)x, TR, m->expU, m->lineopX, m->gamX, m->expM,
          m->expG, y, cbeg, cend, m->N, skip, m->tabX);
    return cudaGetLastError();
  }
  template <typename T>
  static cudaError_t run(const dg_mesh* m, bool modal, int which, const double* x, double* y,
                         long long cbeg, long long cend, const int* skip, cudaStream_t s) {
    return modal ? pass<true>(m, which, x, y, cbeg, cend, skip, s)
                 : pass<false>(m, which, x, y, cbeg, cend, skip, s);
  }
};

template <int N>
struct FixedPrepF {
  template <typename T>
  static cudaError_t run() {
    cudaError_t e = cudaFuncSetAttribute(k_cell_fx<N, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)FixedF<N>::SMEM);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_cell_fx<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)FixedF<N>::SMEM);
    return e;
  }
};

template <int N>
struct FixedSetupF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, const double* K, cudaStream_t s) {
    using S = FxSetup<N>;
    k_lines_fx<N><<<(unsigned)((m->ncells + S::C - 1) / S::C), S::THREADS, 0, s>>>(
        K, m->gh64, m->lineopX, m->gamX, m->expM, m->expG, m->ncells, m->N, m->tabX.cg,
        m->tabXS);
    return cudaGetLastError();
  }
};

}  // namespace dgk

int dg_prepare_fixed(int n) {
  cudaError_t e = dgk::dispatch_n<double, dgk::FixedPrepF>(n);
  if (e != cudaSuccess) return dg_cuda_fail(e, "fixed-point apply kernel attributes");
  return DG_OK;
}

int dg_setup_fixed(dg_mesh* m, const double* K, cudaStream_t s) {
  cudaError_t e = dgk::dispatch_n<double, dgk::FixedSetupF>(m->n, (const dg_mesh*)m, K, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "line operators launch");
  return DG_OK;
}

int dg_launch_fixed_pass(const dg_mesh* m, bool modal, int pass, const double* x, double* y,
                         long long cbeg, long long cend, const int* skip, cudaStream_t s) {
  cudaError_t e = dgk::dispatch_n<double, dgk::FixedF>(m->n, m, modal, pass, x, y, cbeg, cend,
                                                       skip, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "apply (fp64) launch");
  return DG_OK;
}

int dg_launch_fixed_apply(const dg_mesh* m, bool modal, const double* x, double* y,
                          const int* skip, cudaStream_t s) {
  dg_timing_mark(m, 0, s);
  int rc = dg_launch_fixed_pass(m, modal, 1, x, y, 0, m->ncells, skip, s);
  if (rc) return rc;
  dg_timing_mark(m, 1, s);
  rc = dg_launch_fixed_pass(m, modal, 2, x, y, 0, m->ncells, skip, s);
  if (rc) return rc;
  dg_timing_mark(m, 2, s);
  return DG_OK;
}
