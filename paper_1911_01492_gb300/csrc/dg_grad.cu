// Gradient of v^T A(K) u with respect to log K at the volume Gauss points.
//
// With Kt_q = h w_q K_q the volume part of v^T A u is sum_q Kt_q grad u . grad v
// (reference gradients), so its derivative by log K_q is that product.  The
// face part is sum_F gamma_F b_F(u, v) with b_F the face form for gamma = 1
// (-{d_n u}[v] - {d_n v}[u] + sigma [u][v] weighted by h w_s w_t); gamma_F
// depends on K only through the cells' Kbar = exp(sum_q w_q log K_q), hence
//   g_q = Kt_q grad u . grad v + w_q sum_{F of the cell} (d gamma_F / d log Kbar_c) b_F(u, v).
//
// Both parts are formed in block fixed point (dg_fixed.cuh) from pass 1 of u and
// of v in the scaled point basis: there Dh u Dh v = w_q du dv at point q, and the
// products of two face traces carry w_s w_t.  With the traces J = u- - u+ and
// the combinations P = (d - sigma u)- + (sigma u + d)+ that pass 1 stores (d half
// the normal derivative), an interior face point gives
//   -(Pu Jv + Pv Ju) - sigma Ju Jv = -(Gu Jv + Gv Ju),  G = P + sigma J / 2;
// a boundary point is the same with the other side's value zero, P twice the own
// combination and 3 sigma / 2 in place of sigma / 2.
// Precision.  The gradient of a smooth field is small against the field, so a
// product of two gradients, rounded to the last place of the cell's largest
// value, would lose twice the digits that each factor has lost.  Every factor is
// therefore brought up to the full range by itself before it is multiplied
// (fx_top) and a point's sum carries its own exponent: what the products add is
// below 2^-59 of each of them.
// FP64 is left to 10 instructions per DOF (the FP64 kernel executed 60); 32^3 Q3:
// pass 1 of both and this kernel 445 -> 117 us (102 without the full range).
#include "dg_fixed.cuh"

namespace dgk {

template <int N>
struct GradCfg {
  static constexpr int C = Cfg<N>::CPB, N2 = N * N;
  // u, v, the volume products; per-line and per-row face sums; exponents of the
  // neighbours and of the points' products
  static constexpr size_t SMEM =
      8 * (3 * C * LinePad<N>::SC + C * (N2 + N)) + 4 * (14 * C + C * LinePad<N>::SC);
};

// v 2^s with |v| 2^s in [2^59, 2^60) (s <= 28 when the upper half is zero); e -= s
__device__ __forceinline__ long long fx_top(long long v, int& e) {
  const int s = 60 - fx_bits(fx_mag_hi(v));
  e -= s;
  return fx_shift(v, s);
}

// a b / 2^60 with both factors at the top of the range
__device__ __forceinline__ long long fx_product(long long a, long long b) {
  FxAcc A = fx_zero();
  fx_mac(A, fx_pair(a), fx_split(b));
  return fx_value(A);
}

// r 2^er + v 2^ev under the larger exponent, left in er
__device__ __forceinline__ long long fx_sum(long long r, int& er, long long v, int ev) {
  const int e = max(er, ev);
  const long long t = (r >> min(e - er, 63)) + (v >> min(e - ev, 63));
  er = e;
  return t;
}

template <int N>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_coeff_grad(const long long* __restrict__ Uu, const long long* __restrict__ TRu,
             const int* __restrict__ eu, const long long* __restrict__ Uv,
             const long long* __restrict__ TRv, const int* __restrict__ ev,
             const double* __restrict__ kt, const double* __restrict__ dgam, double h,
             double* __restrict__ g, long long ncells, int Nc,
             const __grid_constant__ DGTabXGrad tab) {
  constexpr int C = Cfg<N>::CPB, N2 = N * N, N3 = N * N * N;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int p = pt % N, q = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + (active ? lc : 0);
  long long* su = reinterpret_cast<long long*>(smem_raw) + lc * SC;
  long long* sv = su + C * SC;
  long long* sg = sv + C * SC;
  double* sf = reinterpret_cast<double*>(smem_raw) + 3 * C * SC + lc * (N2 + N);
  int(*sexp)[14] =
      reinterpret_cast<int(*)[14]>(reinterpret_cast<double*>(smem_raw) + 3 * C * SC + C * (N2 + N));
  int* se2 = reinterpret_cast<int*>(sexp + C) + lc * SC;  // exponents of sg
  const unsigned nu = (unsigned)Nc;
  const long long stride[3] = {1, Nc, (long long)Nc * Nc};
  const unsigned row = (unsigned)c / nu;
  const int crd[3] = {(int)((unsigned)c - row * nu), (int)(row % nu), (int)(row / nu)};
  // exponents of u (0..6) and v (7..13): six neighbours, own
  if (active) {
    for (int k = pt; k < 14; k += N2) {
      const int f = k % 7, d = f >> 1, cd = d == 0 ? crd[0] : d == 1 ? crd[1] : crd[2];
      const long long st = d == 0 ? stride[0] : d == 1 ? stride[1] : stride[2];
      const bool in = f < 6 && ((f & 1) ? cd < Nc - 1 : cd > 0);
      sexp[lc][k] = (k < 7 ? eu : ev)[in ? ((f & 1) ? c + st : c - st) : c];
    }
  }
  long long u[N], v[N];
#pragma unroll
  for (int e = 0; e < N; ++e) {  // z-lines (a = p, b = q)
    const long long at = c * N3 + e * N2 + q * N + p;
    u[e] = Uu[at];
    v[e] = Uv[at];
    su[e * SZ + q * SY + p] = u[e];
    sv[e * SZ + q * SY + p] = v[e];
  }
  __syncthreads();
  const int* se = sexp[active ? lc : 0];
  int top = 0;
#pragma unroll
  for (int k = 0; k < 14; ++k) top = max(top, se[k]);
  const bool bad = top >= FX_NAN / 2;
  double s = 0.0;  // the line's six face points, weighted by d gamma
  // the volume products of the line, added to r 2^er (or replacing it)
  auto line = [&](int dir, long long (&r)[N], int (&er)[N], bool first) {
    long long gu[N], gv[N];
    fx_deriv<N>(tab, u, gu);
    fx_deriv<N>(tab, v, gv);
#pragma unroll
    for (int e = 0; e < N; ++e) {
      int ep = 0;
      const long long a = fx_top(gu[e], ep), b = fx_top(gv[e], ep);
      const long long pr = fx_product(a, b);
      if (first) {
        r[e] = pr;
        er[e] = ep;
      } else {
        r[e] = fx_sum(r[e], er[e], pr, ep);
      }
    }
#pragma unroll
    for (int up = 0; up < 2; ++up) {
      const int f = 2 * dir + up;
      const bool in = up ? crd[dir] < Nc - 1 : crd[dir] > 0;
      const long long cn = in ? (up ? c + stride[dir] : c - stride[dir]) : c;
      const long long o = c * (12 * N2) + (2 * f) * N2 + pt;
      const long long on = cn * (12 * N2) + (2 * (in ? f ^ 1 : f)) * N2 + pt;
      // J = u- - u+ and P of one vector under the common exponent e, 2^-3
      auto side = [&](const long long* __restrict__ TR, int eo, int en, long long& J,
                      long long& P, int& e) {
        e = max(eo, en) + 3;
        const int so = min(e - eo, 63), sn = min(e - en, 63);
        const long long vo = TR[o] >> so, ao = TR[o + N2] >> so;
        const long long vn = in ? TR[on] >> sn : 0, an = TR[on + N2] >> sn;
        J = up ? vo - vn : vn - vo;
        P = ao + an;
      };
      long long Ju, Pu, Jv, Pv;
      int e1, e2;
      side(TRu, se[6], se[f], Ju, Pu, e1);
      side(TRv, se[13], se[7 + f], Jv, Pv, e2);
      FxAcc A = fx_zero<2>(), B = fx_zero<2>();
      fx_mac(A, tab.cj[in ? 0 : 1], fx_split(Ju));
      fx_mac(B, tab.cj[in ? 0 : 1], fx_split(Jv));
      int e3 = 0, e4 = 0;
      const long long Gu = fx_top(Pu + fx_value<2>(A), e3), ju = fx_top(Ju, e4);
      const long long Gv = fx_top(Pv + fx_value<2>(B), e4), jv = fx_top(Jv, e3);
      const long long F = fx_sum(fx_product(Gu, jv), e3, fx_product(Gv, ju), e4);
      s = fma(dgam[c * 6 + f], fx_to_double(F, e1 + e2 + e3 + 60 + tab.cva), s);
    }
  };
  long long r[N];
  int er[N];
  line(2, r, er, true);
#pragma unroll
  for (int e = 0; e < N; ++e) {
    sg[e * SZ + q * SY + p] = r[e];
    se2[e * SZ + q * SY + p] = er[e];
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) {  // y-lines (a = p, e = q)
    u[b] = su[q * SZ + b * SY + p];
    v[b] = sv[q * SZ + b * SY + p];
    r[b] = sg[q * SZ + b * SY + p];
    er[b] = se2[q * SZ + b * SY + p];
  }
  line(1, r, er, false);
#pragma unroll
  for (int b = 0; b < N; ++b) {
    sg[q * SZ + b * SY + p] = r[b];
    se2[q * SZ + b * SY + p] = er[b];
  }
  __syncthreads();
#pragma unroll
  for (int a = 0; a < N; ++a) {  // x-lines (b = p, e = q)
    u[a] = su[q * SZ + p * SY + a];
    v[a] = sv[q * SZ + p * SY + a];
    r[a] = sg[q * SZ + p * SY + a];
    er[a] = se2[q * SZ + p * SY + a];
  }
  line(0, r, er, false);
#pragma unroll
  for (int a = 0; a < N; ++a) {
    sg[q * SZ + p * SY + a] = r[a];
    se2[q * SZ + p * SY + a] = er[a];
  }
  // the cell's face sum in a fixed order: rows of n threads, then n rows
  sf[pt] = s;
  __syncthreads();
  if (q == 0) {
    double t = sf[p];
    for (int k = 1; k < N; ++k) t += sf[k * N + p];
    sf[N2 + p] = t;
  }
  __syncthreads();
  if (!active) return;
  s = sf[N2];
#pragma unroll
  for (int k = 1; k < N; ++k) s += sf[N2 + k];
  // each thread writes the n points of its z-line
  const double ws = -h * s * (tab.w[p] * tab.w[q]);
  const double is = tab.iw[p] * tab.iw[q];
  const int ex = se[6] + se[13] + 60 + 2 * tab.cD;
#pragma unroll
  for (int e = 0; e < N; ++e) {
    const long long at = c * N3 + e * N2 + q * N + p;
    const int o = e * SZ + q * SY + p;
    const double vol = fx_to_double(sg[o], ex + se2[o]);
    const double val = fma(kt[at] * (is * tab.iw[e]), vol, ws * tab.w[e]);
    g[at] = bad ? __longlong_as_double(0x7ff8000000000000ll) : val;
  }
}

template <int N>
struct GradF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, double* g, cudaStream_t s) {
    const unsigned blocks = (unsigned)((m->ncells + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    auto ll = [](double* p) { return reinterpret_cast<const long long*>(p); };
    k_coeff_grad<N><<<blocks, Cfg<N>::THREADS, GradCfg<N>::SMEM, s>>>(
        ll(m->U64), ll(m->TR64), m->expU, ll(m->U64b), ll(m->TR64b), m->expUb, m->kt64, m->dgam,
        m->h, g, m->ncells, m->N, m->tabXG);
    return cudaGetLastError();
  }
};

template <int N>
struct GradPrepF {
  template <typename T>
  static cudaError_t run() {
    return cudaFuncSetAttribute(k_coeff_grad<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)GradCfg<N>::SMEM);
  }
};

}  // namespace dgk

int dg_prepare_grad(int n) {
  cudaError_t e = dgk::dispatch_n<double, dgk::GradPrepF>(n);
  if (e != cudaSuccess) return dg_cuda_fail(e, "coefficient gradient kernel attributes");
  return DG_OK;
}

int dg_launch_coeff_grad(const dg_mesh* m, double* g, cudaStream_t s) {
  cudaError_t e = dgk::dispatch_n<double, dgk::GradF>(m->n, m, g, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "coefficient gradient launch");
  return DG_OK;
}
