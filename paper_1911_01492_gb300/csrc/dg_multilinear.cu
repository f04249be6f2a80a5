// FP64 operator on a multilinear mesh (the paper's problem C, Section 3.3):
// the N^3 cells of the structured mesh with vertices at given positions, each
// cell the trilinear image of its reference cube, so the Jacobian J varies
// from point to point.  Written in reference gradients (the tensor basis on
// [0,1]^3), with physical quantities at every quadrature point:
//   volume:  sum_q h w_q K_q grad u . G_q grad v,   G_q = |det J_q| J_q^-1 J_q^-T / h;
//   face point p of a face with reference axis d (shared surface: the unit
//   normal n along +e_d and the area element A_p are the same from both
//   cells; each side's normal derivative is m_side . grad u_side with
//   m_side = J_side^-1 n):
//     W_p ( -{m . grad u}[v] - {m . grad v}[u] + (sigma / h_F)[u][v] ),
//     W_p = gamma_F A_p,  h_F = (|T-| + |T+|) / (2 |F|) inside, |T| / |F| on
//     the boundary (|T| cell volume, |F| face area).
// Affine vertices give the affine operator exactly.
//
// dg_set_vertices forms the per-point geometry once (k_geo_points,
// k_geo_penalty), dg_set_coefficient the products with the coefficient
// (k_ml_setup).  The operator runs in block fixed point (dg_fixed.cuh) in the
// scaled point basis: with g_d = Dh u along direction d (sqrt(w_q) times the
// reference derivative),
//   volume:  r += sum_d Dh^T F_d,  F_d = sum_e (h K G)_de g_e  per point;
//   faces:   a trace of a point field is its contraction with the scaled end
//            values l along the normal line, for u and for each g_j, so a
//            side's normal derivative is m . (traces of g).  With the weight
//            Ws = h gamma A / (h w_s w_t), J = u- - u+ and D = m . grad u summed
//            over the sides (halved inside),
//              r += +- l (Ws pen J - Ws D),   F_j += -l m_j Ws J  (halved inside);
//            the second line is the derivative of the test function, which
//            joins the volume flux before Dh^T.
// Pass 1 (k_trace_ml) leaves v and m . grad u on every face, each side with its
// own m; pass 2 (k_cell_ml) reads the neighbours'.  Every array has its own
// exponent (per cell, or per face for the face coefficients) and the sums take
// the largest.  The FP64 kernels executed 196 FP64 flops per DOF at one
// instruction per 64 cycles: 40^3 Q3 1003 us, now 266 us.
#include <cmath>
#include <vector>

#include "dg_fixed.cuh"

namespace {

// Trilinear map of one cell: Jacobian J[i][j] = d x_i / d xi_j at xi from the
// corner positions C[dz][dy][dx][3].
__device__ void tri_jacobian(const double (&C)[2][2][2][3], double x1, double x2, double x3,
                             double (&J)[3][3]) {
  const double s1[2] = {1.0 - x1, x1}, s2[2] = {1.0 - x2, x2}, s3[2] = {1.0 - x3, x3};
  const double ds[2] = {-1.0, 1.0};
  for (int i = 0; i < 3; ++i) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int dz = 0; dz < 2; ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx) {
          const double v = C[dz][dy][dx][i];
          a = fma(v, s3[dz] * s2[dy] * ds[dx], a);
          b = fma(v, s3[dz] * ds[dy] * s1[dx], b);
          c = fma(v, ds[dz] * s2[dy] * s1[dx], c);
        }
    J[i][0] = a;
    J[i][1] = b;
    J[i][2] = c;
  }
}

// inverse by cofactors; returns det J
__device__ double inv3(const double (&J)[3][3], double (&Ji)[3][3]) {
  const double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                     J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                     J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
  const double r = 1.0 / det;
  Ji[0][0] = (J[1][1] * J[2][2] - J[1][2] * J[2][1]) * r;
  Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) * r;
  Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) * r;
  Ji[1][0] = (J[1][2] * J[2][0] - J[1][0] * J[2][2]) * r;
  Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) * r;
  Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) * r;
  Ji[2][0] = (J[1][0] * J[2][1] - J[1][1] * J[2][0]) * r;
  Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) * r;
  Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) * r;
  return det;
}

struct GaussPts {
  double xi[DG_MAXN];
};

// One thread per cell: volume metric and |det J| at the volume Gauss points,
// area element / h and J^-1 n at the face points, cell volume and face areas.
// A non-positive det J raises *flag.
__global__ void k_geo_points(const double* __restrict__ V, int Nc, int n, double h,
                             double* __restrict__ gvol, double* __restrict__ gdet,
                             double* __restrict__ gface, double* __restrict__ cellvol,
                             double* __restrict__ facearea, int* flag,
                             const __grid_constant__ GaussPts gp,
                             const __grid_constant__ DGTab<double> tab) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nc = (long long)Nc * Nc * Nc;
  if (c >= nc) return;
  const int cx = (int)(c % Nc), cy = (int)((c / Nc) % Nc), cz = (int)(c / ((long long)Nc * Nc));
  const long long V1 = Nc + 1;
  double C[2][2][2][3];
  for (int dz = 0; dz < 2; ++dz)
    for (int dy = 0; dy < 2; ++dy)
      for (int dx = 0; dx < 2; ++dx) {
        const long long v = ((cz + dz) * V1 + (cy + dy)) * V1 + (cx + dx);
        for (int i = 0; i < 3; ++i) C[dz][dy][dx][i] = V[3 * v + i];
      }
  const int n2 = n * n, n3 = n2 * n;
  double vol = 0.0;
  bool bad = false;
  for (int q = 0; q < n3; ++q) {
    const int a = q % n, b = (q / n) % n, e = q / n2;
    double J[3][3], Ji[3][3];
    tri_jacobian(C, gp.xi[a], gp.xi[b], gp.xi[e], J);
    const double det = inv3(J, Ji);
    if (!(det > 0.0)) bad = true;
    const double ad = fabs(det);
    // G = |det J| J^-1 J^-T / h, components xx, yy, zz, xy, xz, yz
    const int ii[6] = {0, 1, 2, 0, 0, 1}, jj[6] = {0, 1, 2, 1, 2, 2};
    for (int t = 0; t < 6; ++t) {
      double s = 0.0;
      for (int k = 0; k < 3; ++k) s = fma(Ji[ii[t]][k], Ji[jj[t]][k], s);
      gvol[(c * 6 + t) * n3 + q] = ad * s / h;
    }
    gdet[c * n3 + q] = ad;
    vol = fma(tab.w[a] * tab.w[b] * tab.w[e], ad, vol);
  }
  cellvol[c] = vol;
  for (int f = 0; f < 6; ++f) {
    const int d = f >> 1, sd = f & 1;
    const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
    double area = 0.0;
    for (int p = 0; p < n2; ++p) {
      const int s1 = p % n, s2 = p / n;
      double xi3[3];
      xi3[d] = (double)sd;
      xi3[t1] = gp.xi[s1];
      xi3[t2] = gp.xi[s2];
      double J[3][3], Ji[3][3];
      tri_jacobian(C, xi3[0], xi3[1], xi3[2], J);
      const double det = inv3(J, Ji);
      if (!(det > 0.0)) bad = true;
      // J^-T e_d = row d of J^-1; unit normal n; m = J^-1 n
      const double v0 = Ji[d][0], v1 = Ji[d][1], v2 = Ji[d][2];
      const double len = sqrt(v0 * v0 + v1 * v1 + v2 * v2);
      const double nn[3] = {v0 / len, v1 / len, v2 / len};
      const double A = fabs(det) * len * tab.w[s1] * tab.w[s2];
      area += A;
      double* gf = gface + (c * 6 + f) * 4 * n2;
      gf[p] = A / h;
      for (int i = 0; i < 3; ++i)
        gf[(1 + i) * n2 + p] = Ji[i][0] * nn[0] + Ji[i][1] * nn[1] + Ji[i][2] * nn[2];
    }
    facearea[c * 6 + f] = area;
  }
  if (bad) atomicOr(flag, 1);
}

// sigma / h_F per cell face: h_F = (|T-| + |T+|) / (2 |F|) inside, |T| / |F| on
// the boundary.
__global__ void k_geo_penalty(const double* __restrict__ cellvol,
                              const double* __restrict__ facearea, double* __restrict__ pen,
                              int Nc, double sigma) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nc = (long long)Nc * Nc * Nc;
  if (c >= nc) return;
  const int crd[3] = {(int)(c % Nc), (int)((c / Nc) % Nc), (int)(c / ((long long)Nc * Nc))};
  const long long stride[3] = {1, Nc, (long long)Nc * Nc};
  for (int f = 0; f < 6; ++f) {
    const int d = f >> 1;
    const bool upper = f & 1;
    const bool inside = upper ? crd[d] < Nc - 1 : crd[d] > 0;
    const double F = facearea[c * 6 + f];
    const double T = inside ? 0.5 * (cellvol[c] + cellvol[upper ? c + stride[d] : c - stride[d]])
                            : cellvol[c];
    pen[c * 6 + f] = sigma * F / T;
  }
}

}  // namespace

namespace dgk {

// F[e] = sum_f Dh[f][e] G[f]  2^-cD
template <int N>
__device__ __forceinline__ void fx_deriv_t(const DGTabXGrad& t, const long long (&G)[N],
                                           long long (&r)[N]) {
  constexpr int H = N / 2, P = (N + 1) / 2;
  FxVal e[P], o[H];
#pragma unroll
  for (int f = 0; f < H; ++f) {
    e[f] = fx_split(G[f] + G[N - 1 - f]);
    o[f] = fx_split(G[f] - G[N - 1 - f]);
  }
  if (N % 2 == 1) e[P - 1] = fx_split(G[H]);
#pragma unroll
  for (int a = 0; a < P; ++a) {
    FxAcc E = fx_zero();
#pragma unroll
    for (int f = 0; f < H; ++f) fx_mac(E, t.De[f][a], o[f]);
    const long long p = fx_value(E);
    if (a == N - 1 - a) {
      r[a] = p;
    } else {
      FxAcc Q = fx_zero();
#pragma unroll
      for (int f = 0; f < P; ++f) fx_mac(Q, t.Do[f][a], e[f]);
      const long long q = fx_value(Q);
      r[a] = p + q;
      r[N - 1 - a] = p - q;
    }
  }
}

// the field's values at both ends of the line, 2^-cv
template <int N>
__device__ __forceinline__ void fx_ends(const DGTabX& t, const long long (&u)[N], long long& lo,
                                        long long& up) {
  constexpr int H = N / 2;
  FxAcc E = fx_zero(), O = fx_zero();
#pragma unroll
  for (int a = 0; a < H; ++a) {
    fx_mac(E, t.ve[a], fx_split(u[a] + u[N - 1 - a]));
    fx_mac(O, t.vo[a], fx_split(u[a] - u[N - 1 - a]));
  }
  if (N % 2 == 1) fx_mac(E, t.ve[H], fx_split(u[H]));
  const long long e = fx_value(E), o = fx_value(O);
  lo = e + o;
  up = e - o;
}

// u[a] += l[a] lo + l[n-1-a] up, l 2^-cl
template <int N>
__device__ __forceinline__ void fx_lift(const DGTabX& t, long long lo, long long up,
                                        long long (&u)[N]) {
  const FxVal s = fx_split(lo + up), d = fx_split(lo - up);
#pragma unroll
  for (int a = 0; a < (N + 1) / 2; ++a) {
    FxAcc E = fx_zero();
    fx_mac(E, t.le[a], s);
    const long long e = fx_value(E);
    if (a == N - 1 - a) {
      u[a] += e;
    } else {
      FxAcc O = fx_zero();
      fx_mac(O, t.lo[a], d);
      const long long o = fx_value(O);
      u[a] += e + o;
      u[N - 1 - a] += e - o;
    }
  }
}

// Per-mesh data of the fixed-point operator on curved cells.  V: h K G [c][xx, yy,
// zz, xy, xz, yz][n^3], exponent eV; per face point [c][6][8][n^2]: m (3),
// exponent em per cell, then -m Ws (halved inside; 3), Ws (halved inside) and
// Ws pen, exponents ef[c][6][3].
struct MlData {
  FxPair *V, *F;
  int *eV, *em, *ef;
};

template <int N>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_ml_setup(const double* __restrict__ kt, const double* __restrict__ gh,
           const double* __restrict__ gvol, const double* __restrict__ gface,
           const double* __restrict__ gpen, MlData md, long long ncells, int Nc,
           const __grid_constant__ DGTabXGrad tab) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS, N2 = N * N, N3 = N * N * N;
  constexpr int NS = FxSmem<N, T>::NS;
  __shared__ unsigned slots[20][NS];
  for (int i = threadIdx.x; i < 20 * NS; i += T) slots[i / NS][i % NS] = 0;
  __syncthreads();
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + (active ? lc : 0);
  const double is = tab.iw[p] * tab.iw[q];
  double M[6];
  auto metric = [&](int e) {  // h K G at point e of the thread's z-line
    const int o = e * N2 + pt;
    const double k = kt[c * N3 + o] * (is * tab.iw[e]);
#pragma unroll
    for (int t = 0; t < 6; ++t) M[t] = k * gvol[(c * 6 + t) * N3 + o];
  };
  unsigned big = 0;
  for (int e = 0; e < N; ++e) {
    metric(e);
    const double x = fabs(M[3]), y = fabs(M[4]), z = fabs(M[5]);
    big = max(big, fx_abs_hi(fmax(M[0] + x + y, fmax(M[1] + x + z, M[2] + y + z))));
  }
  const int EV = fx_exponent(fx_cell_max<N, T>(big, lc, slots[0]));
  if (active) {
    for (int e = 0; e < N; ++e) {
      metric(e);
#pragma unroll
      for (int t = 0; t < 6; ++t)
        md.V[(c * 6 + t) * N3 + e * N2 + pt] = fx_pair(fx_from_double(M[t], 60 - EV, EV));
    }
    if (pt == 0) md.eV[c] = EV;
  }
  const unsigned nu = (unsigned)Nc, row = (unsigned)c / nu;
  const int crd[3] = {(int)((unsigned)c - row * nu), (int)(row % nu), (int)(row / nu)};
  auto geo = [&](int f, int k) { return gface[((c * 6 + f) * 4 + k) * N2 + pt]; };
  big = 0;
  for (int f = 0; f < 6; ++f)
    big = max(big, fx_abs_hi(fabs(geo(f, 1)) + fabs(geo(f, 2)) + fabs(geo(f, 3))));
  const int Em = fx_exponent(fx_cell_max<N, T>(big, lc, slots[1]));
  if (active && pt == 0) md.em[c] = Em;
  for (int f = 0; f < 6; ++f) {
    const int d = f >> 1;
    const bool in = f & 1 ? crd[d] < Nc - 1 : crd[d] > 0;
    const double W = gh[c * 6 + f] * geo(f, 0) * is, Wh = in ? 0.5 * W : W;
    const double v[8] = {geo(f, 1),       geo(f, 2),       geo(f, 3), -Wh * geo(f, 1),
                         -Wh * geo(f, 2), -Wh * geo(f, 3), Wh,        W * gpen[c * 6 + f]};
    unsigned b[3] = {max(fx_abs_hi(v[3]), max(fx_abs_hi(v[4]), fx_abs_hi(v[5]))),
                     fx_abs_hi(v[6]), fx_abs_hi(v[7])};
    int E[4] = {Em, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      E[k + 1] = fx_exponent(fx_cell_max<N, T>(b[k], lc, slots[2 + 3 * f + k]));
      if (active && pt == 0) md.ef[(c * 6 + f) * 3 + k] = E[k + 1];
    }
    if (active) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int e = E[k < 3 ? 0 : k < 6 ? 1 : k - 4];
        md.F[((c * 6 + f) * 8 + k) * N2 + pt] = fx_pair(fx_from_double(v[k], 60 - e, e));
      }
    }
  }
}

// Pass 1: the point values U under one exponent, and per face v and m . grad u
// (exponents expU + cv, and expU + em + cD + cv).
template <int N>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_trace_ml(const double* __restrict__ x, long long* __restrict__ U, long long* __restrict__ TR,
           int* __restrict__ expU, const FxPair* __restrict__ F, long long ncells,
           const int* __restrict__ skip, const __grid_constant__ DGTabX tab,
           const __grid_constant__ DGTabXGrad tg) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS, N2 = N * N, N3 = N * N * N;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC;
  constexpr int NS = FxSmem<N, T>::NS;
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned slots[3 * NS];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + (active ? lc : 0);
  // u, then its derivatives along x, y, z
  long long* su = reinterpret_cast<long long*>(smem_raw) + lc * 4 * SC;
  long long* sd[3] = {su + SC, su + 2 * SC, su + 3 * SC};
  for (int i = threadIdx.x; i < 3 * NS; i += T) slots[i] = 0;
  __syncthreads();
  double xv[N];
  unsigned big = 0;
#pragma unroll
  for (int l = 0; l < N; ++l) {
    xv[l] = active ? x[c * N3 + l * N2 + q * N + p] : 0.0;
    big = max(big, fx_abs_hi(xv[l]));
  }
  const int E = fx_exponent(fx_cell_max<N, T>(big, lc, slots));
  const int k = fx_norm_scale<N, T>(xv, E, lc, slots + 2 * NS);
  const int zl = q * SY + p, yl = q * SZ + p, xl = q * SZ + p * SY;
  long long v[N], u[N];
#pragma unroll
  for (int l = 0; l < N; ++l) v[l] = fx_from_double(xv[l], k, E);
  fx_fwd<N>(tab, v, u);
#pragma unroll
  for (int e = 0; e < N; ++e) su[zl + e * SZ] = u[e];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = su[yl + j * SY];
  fx_fwd<N>(tab, v, u);
#pragma unroll
  for (int b = 0; b < N; ++b) su[yl + b * SY] = u[b];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = su[xl + i];
  fx_fwd<N>(tab, v, u);
  big = 0;
#pragma unroll
  for (int a = 0; a < N; ++a) big = max(big, fx_mag_hi(u[a]));
  const int up = 60 - fx_bits(fx_cell_max<N, T>(big, lc, slots + NS));
#pragma unroll
  for (int a = 0; a < N; ++a) {
    u[a] = fx_shift(u[a], up);
    su[xl + a] = u[a];
  }
  fx_deriv<N>(tg, u, v);
#pragma unroll
  for (int a = 0; a < N; ++a) sd[0][xl + a] = v[a];
  if (active && pt == 0) expU[c] = E == FX_NAN ? FX_NAN : -k - up;
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) u[b] = su[yl + b * SY];
  fx_deriv<N>(tg, u, v);
#pragma unroll
  for (int b = 0; b < N; ++b) sd[1][yl + b * SY] = v[b];
#pragma unroll
  for (int e = 0; e < N; ++e) {
    u[e] = su[zl + e * SZ];
    if (active) U[c * N3 + e * N2 + pt] = u[e];
  }
  fx_deriv<N>(tg, u, v);
#pragma unroll
  for (int e = 0; e < N; ++e) sd[2][zl + e * SZ] = v[e];
  __syncthreads();
  if (!active) return;  // no barrier follows
  long long* tr = TR + c * (12 * N2) + pt;
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    const int at = dir == 0 ? xl : dir == 1 ? yl : zl, step = dir == 0 ? 1 : dir == 1 ? SY : SZ;
    FxAcc A[2] = {fx_zero(), fx_zero()};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int e = 0; e < N; ++e) u[e] = su[k * SC + at + e * step];
      long long end[2];
      fx_ends<N>(tab, u, end[0], end[1]);
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        if (k == 0)
          tr[(4 * dir + 2 * f) * N2] = end[f];
        else
          fx_mac(A[f], F[((c * 6 + 2 * dir + f) * 8 + k - 1) * N2 + pt], fx_split(end[f]));
      }
    }
#pragma unroll
    for (int f = 0; f < 2; ++f) tr[(4 * dir + 2 * f + 1) * N2] = fx_value(A[f]);
  }
}

template <int N>
struct MlSmem {
  static constexpr int C = Cfg<N>::CPB;
  static constexpr size_t trace = 8 * 4 * C * LinePad<N>::SC;
  // u / r, the flux; per cell: nine shifts and exponents per face, then those of
  // the volume flux and the largest of F's and of r's lifted terms
  static constexpr int SH = 6 * 9 + 3;
  static constexpr size_t cell = 8 * 5 * C * LinePad<N>::SC + 4 * (SH * C);
};

// Registers for one block per SM more than they would allow by themselves (n = 6-8).
template <int N>
__global__ void __launch_bounds__(Cfg<N>::THREADS, N == 8 ? 4 : N == 6 || N == 7 ? 3 : 0)
k_cell_ml(const long long* __restrict__ U, const long long* __restrict__ TR,
          const int* __restrict__ expU, MlData md, double* __restrict__ y, long long ncells,
          int Nc, const int* __restrict__ skip, const __grid_constant__ DGTabX tab,
          const __grid_constant__ DGTabXGrad tg) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS, N2 = N * N, N3 = N * N * N;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC;
  constexpr int NS = FxSmem<N, T>::NS, SH = MlSmem<N>::SH;
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned slots[3 * NS];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + (active ? lc : 0);
  long long* su = reinterpret_cast<long long*>(smem_raw) + lc * 5 * SC;  // u
  long long* sF = su + SC;                                              // F_x, F_y, F_z
  long long* sr = su + 4 * SC;                                          // r
  int* sh = reinterpret_cast<int*>(reinterpret_cast<long long*>(smem_raw) + 5 * C * SC) +
            (active ? lc : 0) * SH;
  const unsigned nu = (unsigned)Nc, row = (unsigned)c / nu;
  const int crd[3] = {(int)((unsigned)c - row * nu), (int)(row % nu), (int)(row / nu)};
  const long long stride[3] = {1, Nc, (long long)Nc * Nc};
  for (int i = threadIdx.x; i < 3 * NS; i += T) slots[i] = 0;
  // Exponents and shifts, one thread per cell; EF and ER, those of F and r, follow
  // once the cell's largest derivative is known.  F sums the volume flux, halved
  // (<= 2^59), and six lifted terms (each below 2^61, five bits down): below
  // 2^60.  r sums Dh^T F in three directions and six lifted terms three bits
  // down: below 2^62.5.
  if (active && pt == 0) {
    const int Eo = expU[c], em = md.em[c];
    int EF = -4 * FX_NAN, ER = -4 * FX_NAN, eJ, eD;
    bool nan = Eo >= FX_NAN / 2 || md.eV[c] >= FX_NAN / 2;
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int d = f >> 1;
      const bool in = f & 1 ? crd[d] < Nc - 1 : crd[d] > 0;
      const long long cn = in ? (f & 1 ? c + stride[d] : c - stride[d]) : c;
      const int En = expU[cn], mn = md.em[cn];
      nan = nan || En >= FX_NAN / 2 || md.ef[(c * 6 + f) * 3] >= FX_NAN / 2;
      eJ = max(Eo, En) + 1;
      eD = max(Eo + em, En + mn) + 1;
      sh[9 * f + 0] = min(eJ - Eo, 63);
      sh[9 * f + 1] = min(eJ - En, 63);
      sh[9 * f + 2] = min(eD - Eo - em, 63);
      sh[9 * f + 3] = min(eD - En - mn, 63);
      eJ += tg.cv;
      eD += tg.cv + tg.cD;
      // exponents of the lifted terms of F, and of the two of r
      const int* ef = md.ef + (c * 6 + f) * 3;
      sh[9 * f + 4] = ef[0] + eJ + tg.cl;
      sh[9 * f + 5] = ef[2] + eJ + tg.cl;
      sh[9 * f + 6] = ef[1] + eD + tg.cl;
      EF = max(EF, sh[9 * f + 4] + 5);
      ER = max(ER, max(sh[9 * f + 5], sh[9 * f + 6]) + 3);
    }
    sh[54] = md.eV[c] + tg.cD + Eo;
    sh[55] = EF;
    sh[56] = ER;
    sh[7] = nan;
  }
  const int zl = q * SY + p, yl = q * SZ + p, xl = q * SZ + p * SY;
  long long u[N], v[N], F[3][N], r[N];
#pragma unroll
  for (int e = 0; e < N; ++e) {
    u[e] = U[c * N3 + e * N2 + pt];
    su[zl + e * SZ] = u[e];
  }
  unsigned top = 0;
  auto largest = [&](const long long (&w)[N]) {
#pragma unroll
    for (int e = 0; e < N; ++e) top = max(top, fx_mag_hi(w[e]));
  };
  fx_deriv<N>(tg, u, F[2]);
  largest(F[2]);
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) u[b] = su[yl + b * SY];
  fx_deriv<N>(tg, u, v);
  largest(v);
#pragma unroll
  for (int b = 0; b < N; ++b) sF[SC + yl + b * SY] = v[b];
#pragma unroll
  for (int a = 0; a < N; ++a) u[a] = su[xl + a];
  fx_deriv<N>(tg, u, v);
  largest(v);
#pragma unroll
  for (int a = 0; a < N; ++a) sF[xl + a] = v[a];
  // The derivatives of a smooth field are small against their bound: the flux is
  // kept `spare` bits finer, the low halves' products included, so that points of
  // small K do not take the rounding of the cell's largest one.
  const int spare =
      min(max(60 - fx_bits(fx_cell_max<N, T>(top, lc, slots + 2 * NS)), 0), 28);
  if (32 % N2 == 0) __syncthreads();
  const int EF = max(sh[54] + 1 - spare, sh[55]), ER = max(sh[56], EF + tg.cD);
  // the flux at the points of the z-line
  {
    const FxPair* V = md.V + c * 6 * N3 + pt;
    const int down = min(EF - sh[54], 63), finer = max(-down, 0), coarser = max(down, 0);
    auto flux = [&](const FxPair& a, const FxVal& x, const FxPair& b, const FxVal& y,
                    const FxPair& d, const FxVal& z) {
      FxAcc A = {0, 1ll << (29 - finer)};
      fx_mac(A, a, x);
      fx_mac(A, b, y);
      fx_mac(A, d, z);
      const long long low = fx_madw(a.l, x.l, fx_madw(b.l, y.l, fx_madw(d.l, z.l, 0)));
      const long long m = A.m + (low >> 30);
      return ((A.h << finer) + (m >> (30 - finer))) >> coarser;
    };
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const FxVal gx = fx_split(sF[zl + e * SZ]), gy = fx_split(sF[SC + zl + e * SZ]),
                  gz = fx_split(F[2][e]);
      const FxPair xx = V[e * N2], yy = V[N3 + e * N2], zz = V[2 * N3 + e * N2],
                   xy = V[3 * N3 + e * N2], xz = V[4 * N3 + e * N2], yz = V[5 * N3 + e * N2];
      F[0][e] = flux(xx, gx, xy, gy, xz, gz);
      F[1][e] = flux(xy, gx, yy, gy, yz, gz);
      F[2][e] = flux(xz, gx, yz, gy, zz, gz);
    }
  }
  // both faces of the thread's line: their terms into F and r of the line
  auto faces = [&](int dir) {
    long long t[2][3], w[2];
#pragma unroll
    for (int up = 0; up < 2; ++up) {
      const int f = 2 * dir + up;
      const bool in = up ? crd[dir] < Nc - 1 : crd[dir] > 0;
      const long long cn = in ? (up ? c + stride[dir] : c - stride[dir]) : c;
      const long long* to = TR + c * (12 * N2) + (2 * f) * N2 + pt;
      const long long* tn = TR + cn * (12 * N2) + (2 * (in ? f ^ 1 : f)) * N2 + pt;
      const FxPair* W = md.F + (c * 6 + f) * 8 * N2 + pt;
      const int* s = sh + 9 * f;
      const long long vo = to[0] >> s[0], vn = in ? tn[0] >> s[1] : 0;
      const long long D = (to[N2] >> s[2]) + (in ? tn[N2] >> s[3] : 0);
      const FxVal J = fx_split(up ? vo - vn : vn - vo);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        FxAcc A = fx_zero();
        fx_mac(A, W[(3 + j) * N2], J);
        t[up][j] = fx_value(A) >> min(EF - s[4], 63);
      }
      FxAcc A = fx_zero(), B = fx_zero();
      fx_mac(A, W[7 * N2], J);
      fx_mac(B, W[6 * N2], fx_split(D));
      const long long cv =
          (fx_value(A) >> min(ER - s[5], 63)) - (fx_value(B) >> min(ER - s[6], 63));
      w[up] = up ? cv : -cv;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) fx_lift<N>(tab, t[0][j], t[1][j], F[j]);
    fx_lift<N>(tab, w[0], w[1], r);
  };
#pragma unroll
  for (int e = 0; e < N; ++e) r[e] = 0;
  faces(2);
#pragma unroll
  for (int e = 0; e < N; ++e) {
    sr[zl + e * SZ] = r[e];
#pragma unroll
    for (int j = 0; j < 3; ++j) sF[j * SC + zl + e * SZ] = F[j][e];
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) {
    r[b] = sr[yl + b * SY];
#pragma unroll
    for (int j = 0; j < 3; ++j) F[j][b] = sF[j * SC + yl + b * SY];
  }
  faces(1);
#pragma unroll
  for (int b = 0; b < N; ++b) {
    sr[yl + b * SY] = r[b];
#pragma unroll
    for (int j = 0; j < 3; ++j) sF[j * SC + yl + b * SY] = F[j][b];
  }
  __syncthreads();
#pragma unroll
  for (int a = 0; a < N; ++a) {
    r[a] = sr[xl + a];
#pragma unroll
    for (int j = 0; j < 3; ++j) F[j][a] = sF[j * SC + xl + a];
  }
  faces(0);
  const int down = min(ER - EF - tg.cD, 63);
  fx_deriv_t<N>(tg, F[0], v);
#pragma unroll
  for (int a = 0; a < N; ++a) {
    sr[xl + a] = r[a] + (v[a] >> down);
    sF[SC + xl + a] = F[1][a];
    sF[2 * SC + xl + a] = F[2][a];
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) u[b] = sF[SC + yl + b * SY];
  fx_deriv_t<N>(tg, u, v);
#pragma unroll
  for (int b = 0; b < N; ++b) sr[yl + b * SY] += v[b] >> down;
  __syncthreads();
#pragma unroll
  for (int e = 0; e < N; ++e) u[e] = sF[2 * SC + zl + e * SZ];
  fx_deriv_t<N>(tg, u, v);
  unsigned big = 0;
#pragma unroll
  for (int e = 0; e < N; ++e) {
    r[e] = sr[zl + e * SZ] + (v[e] >> down);
    big = max(big, fx_mag_hi(r[e]));
  }
  // Q^T along z, y, x, then out through the z-lines
  const int up = fx_norm_shift<N, T>(r, fx_bits(fx_cell_max<N, T>(big, lc, slots)), lc,
                                     slots + NS);
#pragma unroll
  for (int e = 0; e < N; ++e) r[e] = fx_shift(r[e], up);
  fx_bwd<N>(tab, r, u);
#pragma unroll
  for (int l = 0; l < N; ++l) su[zl + l * SZ] = u[l];
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) r[b] = su[yl + b * SY];
  fx_bwd<N>(tab, r, u);
#pragma unroll
  for (int j = 0; j < N; ++j) su[yl + j * SY] = u[j];
  __syncthreads();
#pragma unroll
  for (int a = 0; a < N; ++a) r[a] = su[xl + a];
  fx_bwd<N>(tab, r, u);
#pragma unroll
  for (int i = 0; i < N; ++i) su[xl + i] = u[i];
  __syncthreads();
  if (active) {
    const bool nan = sh[7] != 0;
#pragma unroll
    for (int l = 0; l < N; ++l)
      y[c * N3 + l * N2 + pt] = nan ? __longlong_as_double(0x7ff8000000000000ll)
                                    : fx_to_double(su[zl + l * SZ], ER - up);
  }
}

template <int N>
struct MlApplyF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, const double* x, double* yv, const int* skip,
                         cudaStream_t s) {
    const unsigned blocks = (unsigned)((m->ncells + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    long long* U = reinterpret_cast<long long*>(m->U64);
    long long* TR = reinterpret_cast<long long*>(m->TR64);
    const MlData md{m->mlV, m->mlF, m->mlExpV, m->mlExpM, m->mlExpF};
    dg_timing_mark(m, 0, s);
    k_trace_ml<N><<<blocks, Cfg<N>::THREADS, MlSmem<N>::trace, s>>>(
        x, U, TR, m->expU, m->mlF, m->ncells, skip, m->tabX, m->tabXG);
    dg_timing_mark(m, 1, s);
    k_cell_ml<N><<<blocks, Cfg<N>::THREADS, MlSmem<N>::cell, s>>>(
        U, TR, m->expU, md, yv, m->ncells, m->N, skip, m->tabX, m->tabXG);
    dg_timing_mark(m, 2, s);
    return cudaGetLastError();
  }
};

template <int N>
struct MlSetupF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, cudaStream_t s) {
    const unsigned blocks = (unsigned)((m->ncells + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    k_ml_setup<N><<<blocks, Cfg<N>::THREADS, 0, s>>>(
        m->kt64, m->gh64, m->geo_vol, m->geo_face, m->geo_pen,
        MlData{m->mlV, m->mlF, m->mlExpV, m->mlExpM, m->mlExpF}, m->ncells, m->N, m->tabXG);
    return cudaGetLastError();
  }
};

template <int N>
struct MlPrepareF {
  template <typename T>
  static cudaError_t run() {
    cudaError_t e = cudaFuncSetAttribute(
        k_trace_ml<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MlSmem<N>::trace);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_cell_ml<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)MlSmem<N>::cell);
    return e;
  }
};

}  // namespace dgk

int dg_setup_multilinear(dg_mesh* m, cudaStream_t s) {
  const size_t n3 = (size_t)m->n * m->n * m->n, n2 = (size_t)m->n * m->n;
  const size_t nc = (size_t)m->ncells;
  if (m->mlV == nullptr) DG_CUDA(cudaMalloc((void**)&m->mlV, sizeof(FxPair) * 6 * n3 * nc));
  if (m->mlF == nullptr) DG_CUDA(cudaMalloc((void**)&m->mlF, sizeof(FxPair) * 48 * n2 * nc));
  if (m->mlExpV == nullptr) DG_CUDA(cudaMalloc((void**)&m->mlExpV, sizeof(int) * nc));
  if (m->mlExpM == nullptr) DG_CUDA(cudaMalloc((void**)&m->mlExpM, sizeof(int) * nc));
  if (m->mlExpF == nullptr) DG_CUDA(cudaMalloc((void**)&m->mlExpF, sizeof(int) * 18 * nc));
  cudaError_t e = dgk::dispatch_n<double, dgk::MlSetupF>(m->n, (const dg_mesh*)m, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "multilinear coefficient data: launch");
  return DG_OK;
}

int dg_launch_apply_multilinear(const dg_mesh* m, const double* x, double* y, const int* skip,
                                cudaStream_t s) {
  cudaError_t e = dgk::dispatch_n<double, dgk::MlApplyF>(m->n, m, x, y, skip, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "multilinear apply: launch");
  return DG_OK;
}

extern "C" int dg_set_vertices(dg_mesh* m, const double* X) {
  if (m == nullptr || X == nullptr)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_set_vertices: NULL mesh or vertices");
  const long long nv = (long long)(m->N + 1) * (m->N + 1) * (m->N + 1);
  for (long long i = 0; i < 3 * nv; ++i)
    if (!std::isfinite(X[i]))
      return dg_fail(DG_ERR_INVALID_ARG, "dg_set_vertices: vertex coordinate %lld not finite", i);
  const size_t n3 = (size_t)m->n * m->n * m->n, n2 = (size_t)m->n * m->n;
  const size_t nc = (size_t)m->ncells;
  if (m->geo_vol == nullptr) {
    DG_CUDA(cudaMalloc((void**)&m->geo_vol, sizeof(double) * 6 * n3 * nc));
    DG_CUDA(cudaMalloc((void**)&m->geo_det, sizeof(double) * n3 * nc));
    DG_CUDA(cudaMalloc((void**)&m->geo_face, sizeof(double) * 24 * n2 * nc));
    DG_CUDA(cudaMalloc((void**)&m->geo_pen, sizeof(double) * 6 * nc));
  }
  double *dV = nullptr, *dvol = nullptr, *darea = nullptr;
  cudaError_t e = cudaMalloc((void**)&dV, sizeof(double) * 3 * nv);
  if (e == cudaSuccess) e = cudaMalloc((void**)&dvol, sizeof(double) * nc);
  if (e == cudaSuccess) e = cudaMalloc((void**)&darea, sizeof(double) * 6 * nc);
  if (e == cudaSuccess) e = cudaMemcpy(dV, X, sizeof(double) * 3 * nv, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(m->dflag, 0, sizeof(int));
  GaussPts gp = {};
  double w[DG_MAXN];
  dg_gauss_points(m->n, gp.xi, w);
  const unsigned blocks = (unsigned)((nc + 127) / 128);
  if (e == cudaSuccess) {
    k_geo_points<<<blocks, 128>>>(dV, m->N, m->n, m->h, m->geo_vol, m->geo_det, m->geo_face,
                                  dvol, darea, m->dflag, gp, m->tab64);
    k_geo_penalty<<<blocks, 128>>>(dvol, darea, m->geo_pen, m->N, m->sigma);
    e = cudaGetLastError();
  }
  int flag = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&flag, m->dflag, sizeof(int), cudaMemcpyDeviceToHost);
  cudaFree(dV);
  cudaFree(dvol);
  cudaFree(darea);
  if (e != cudaSuccess) return dg_cuda_fail(e, "dg_set_vertices");
  if (flag) {
    // the mesh is the cube again, under the coefficient that it has: a curved mesh
    // has not formed the cube's operators from it
    if (m->multilinear && m->has_coef) {
      m->has_coef = false;
      if (int rc = dg_restore_fixed(m, nullptr)) return rc;
      DG_CUDA(cudaDeviceSynchronize());
      m->has_coef = true;
    }
    m->multilinear = false;
    return dg_fail(DG_ERR_INVALID_ARG,
                   "dg_set_vertices: a cell's Jacobian determinant is not positive (inverted "
                   "or degenerate cell)");
  }
  cudaError_t ea = dgk::dispatch_n<double, dgk::MlPrepareF>(m->n);
  if (ea != cudaSuccess) return dg_cuda_fail(ea, "multilinear apply: kernel attributes");
  m->multilinear = true;
  m->affine = false;
  m->geomDet = 1.0;
  m->has_coef = false;
  m->has_diag = false;
  m->has_block = false;
  m->has_kron = false;
  return DG_OK;
}
