// Kronecker cell-block preconditioner (DG_CG_PRECOND_KRON): a reading of the
// paper's factorised cell-block solves (Section 3.4, block preconditioners on
// the cells' subspaces V_T).  Each cell block of A is replaced by the block of
// the operator with K set to its Gauss-weighted mean over the cell.  In the
// orthonormal Legendre basis (mass matrix h^3 I) that block is the Kronecker
// sum S_x (+) S_y (+) S_z of three n x n matrices,
//   S_d = h Kmean S1 + lower-face and upper-face own-side terms (Section 4.1),
// S1 the 1D stiffness matrix.  It is inverted by fast diagonalisation: with
// S_d = Q_d diag(lambda_d) Q_d^T,
//   M^-1 = (Q_z x Q_y x Q_x) diag(1 / (lx_i + ly_j + lz_l)) (Q_z x Q_y x Q_x)^T,
// six line contractions and a pointwise scaling per cell: 12n flops and
// (3n^2 + 3n) / n^3 stored values per DOF, against 2n^3 flops and n^3 values
// for the exact cell blocks.
//
// k_kron_setup: one thread per (cell, direction) forms S_d in FP64 and its
//   eigen-decomposition by cyclic Jacobi rotations; stores Q_d and lambda_d in
//   FP64 and FP32 ([c][ Q_x Q_y Q_z (row-major [i][j], column j the j-th
//   eigenvector) | l_x l_y l_z ]).
// k_kron_apply (FP32): z = M^-1 r for a group of cells per block (one thread per
//   plane of lines, the 1D factor in registers, in place in shared memory),
//   <z, r> formed in the scaling phase and reduced by the last block.
// k_kron_apply_fx (FP64): the same with the contractions in block fixed point
//   (dg_fixed.cuh), one thread per line.
#include "dg_fixed.cuh"

namespace dgk {
namespace {

template <int N>
__global__ void __launch_bounds__(128)
k_kron_setup(const double* __restrict__ kt, const double* __restrict__ gh,
             double* __restrict__ K64, float* __restrict__ K32, long long ncells, int Nc,
             int* flag, const __grid_constant__ DGTab<double> tab) {
  constexpr int N2 = N * N, N3 = N * N * N, KS = 3 * N2 + 3 * N;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 3 * ncells) return;
  const long long c = t / 3;
  const int d = (int)(t - 3 * c);
  const long long coord = d == 0 ? c % Nc : d == 1 ? (c / Nc) % Nc : c / ((long long)Nc * Nc);
  // h Kmean = sum_q h w_q K_q
  double hk = 0.0;
  for (int q = 0; q < N3; ++q) hk += kt[c * N3 + q];
  const double glo = gh[c * 6 + 2 * d], ghi = gh[c * 6 + 2 * d + 1];  // h gamma (0: zero flux)
  const double elo = coord > 0 ? 0.5 : 1.0, ehi = coord < Nc - 1 ? 0.5 : 1.0;
  const double sg = tab.sigma;
  double A[N][N], V[N][N];
  double scale = 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      double s1 = 0.0;
      for (int a = 0; a < N; ++a) s1 += tab.w[a] * tab.Bd[a][i] * tab.Bd[a][j];
      const double lo =
          sg * tab.a0[i] * tab.a0[j] + elo * (tab.d0[i] * tab.a0[j] + tab.a0[i] * tab.d0[j]);
      const double hi =
          sg * tab.a1[i] * tab.a1[j] - ehi * (tab.d1[i] * tab.a1[j] + tab.a1[i] * tab.d1[j]);
      A[i][j] = hk * s1 + glo * lo + ghi * hi;
      V[i][j] = i == j ? 1.0 : 0.0;
      scale += A[i][j] * A[i][j];
    }
  }
  // cyclic Jacobi: A <- J^T A J zeroes A[p][q] with the rotation in the (p, q)
  // plane, t = tan of the angle the smaller root of t^2 + 2 theta t - 1 = 0;
  // V <- V J accumulates the eigenvectors
  for (int sweep = 0; sweep < 16; ++sweep) {
    double off = 0.0;
#pragma unroll
    for (int p = 0; p < N; ++p)
#pragma unroll
      for (int q = p + 1; q < N; ++q) off += A[p][q] * A[p][q];
    if (off <= 1e-32 * scale) break;
#pragma unroll
    for (int p = 0; p < N; ++p) {
#pragma unroll
      for (int q = p + 1; q < N; ++q) {
        const double apq = A[p][q];
        if (fabs(apq) <= 1e-300) continue;
        const double theta = (A[q][q] - A[p][p]) / (2.0 * apq);
        const double tt = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
        const double cs = 1.0 / sqrt(tt * tt + 1.0), sn = tt * cs;
#pragma unroll
        for (int k = 0; k < N; ++k) {  // columns p, q of A J
          const double akp = A[k][p], akq = A[k][q];
          A[k][p] = cs * akp - sn * akq;
          A[k][q] = sn * akp + cs * akq;
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {  // rows p, q of J^T (A J)
          const double apk = A[p][k], aqk = A[q][k];
          A[p][k] = cs * apk - sn * aqk;
          A[q][k] = sn * apk + cs * aqk;
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const double vkp = V[k][p], vkq = V[k][q];
          V[k][p] = cs * vkp - sn * vkq;
          V[k][q] = sn * vkp + cs * vkq;
        }
      }
    }
  }
  double* o64 = K64 + c * KS;
  float* o32 = K32 + c * KS;
  bool ok = true;
#pragma unroll
  for (int i = 0; i < N; ++i) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      o64[d * N2 + i * N + j] = V[i][j];
      o32[d * N2 + i * N + j] = (float)V[i][j];
    }
    // a direction whose two faces are both zero-flux boundary faces (one cell
    // across) has the singular factor h Kmean S1: its zero eigenvalue, up to
    // rounding, is kept at zero (the sum over the three directions stays
    // positive as long as another direction has a face with gamma > 0)
    double lam = A[i][i];
    if (lam < 0.0 && lam > -1e-12 * sqrt(scale)) lam = 0.0;
    ok = ok && lam >= 0.0 && isfinite(lam);
    o64[3 * N2 + d * N + i] = lam;
    o32[3 * N2 + d * N + i] = (float)lam;
  }
  if (!ok) atomicExch(flag, 1);
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& t) {
  s = a + b;
  const float bb = s - a;
  t = (a - (s - bb)) + (b - bb);
}

// Cells per block of the apply: one thread per plane of lines (N threads per
// cell, ~128 threads), shared memory for the work array and the factors
// within 40 KB (48 KB with the reduction arrays); at least Cfg<N>::CPB so the
// block count fits the mesh's per-block partials.
template <int N>
struct KronCfg {
  static constexpr int KS = 3 * N * N + 3 * N;
  static constexpr int PER_CELL = (N * N * N + KS) * (int)sizeof(float);
  static constexpr int BY_THREADS = 128 / N, BY_SMEM = 40960 / PER_CELL;
  static constexpr int C = BY_THREADS < BY_SMEM ? BY_THREADS : BY_SMEM;  // cells per block
  static constexpr int THREADS = C * N;
  static_assert(C >= Cfg<N>::CPB, "more blocks than the mesh's partials");
};

// The grid reduction of <z, r>: each block publishes its partial, the last
// block sums them in a fixed order and sets the CG scalars by MODE: 0 FP64
// iteration (beta = <z,r> / rho, rho = <z,r>); 1 FP64 initialisation (rho = <z,r>,
// runs even when done; the first direction update takes z with beta = 0); 2 FP32
// mixed iteration (rho_new = <z,r>, beta = 0 on a restart, else <z,r> / rho).
template <int NT, int MODE>
__device__ __forceinline__ void kron_finish(double part, double* __restrict__ partials,
                                            DGCGState* st, double* rd) {
  __shared__ bool is_last;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = part;
    __threadfence();
    is_last = (atomicAdd(&st->ticket, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const double tot = last_block_total<NT>(partials, (int)gridDim.x, rd);
  if (threadIdx.x == 0) {
    if (!isfinite(tot)) {
      st->breakdown = 1;
      st->done = 1;
      st->ru_skip = 1;
    } else if (MODE == 1) {
      st->rho = tot;
    } else if (MODE == 0) {
      st->beta = tot / st->rho;
      st->rho = tot;
    } else {
      st->rho_new = tot;
      st->beta = st->restart ? 0.0 : tot / st->rho;
    }
    st->ticket = 0u;
  }
}

// z = M^-1 r on the block's cells, in place in sw (the cells' values in their
// own order; sq holds their factors): thread (cell lc, plane t) contracts the
// N lines of plane t in each phase with the cell's 1D factor in registers.
// Returns the thread's part of <z, r> = sum over the transformed values t of
// t^2 / (lx + ly + lz), formed where the scaling is applied; the terms are
// positive, so per-thread sums (FP32 in the FP32 kernels) stay within n u
// relative, and threads and blocks are added in FP64.  In FP32 the scaling
// uses a fast reciprocal (two ulps: the preconditioner only needs to be a
// fixed symmetric positive definite operator).  Every thread of the block
// calls it; it synchronises before returning.
template <int N>
__device__ __forceinline__ float kron_solve_cells(float* sw, const float* sq, int nblk) {
  constexpr int N2 = N * N, N3 = N * N * N, KS = 3 * N2 + 3 * N;
  const int lc = threadIdx.x / N;
  const int t = threadIdx.x - lc * N;
  const bool active = lc < nblk;
  float* w = sw + lc * N3;
  const float* Qx = sq + lc * KS;
  const float* Qy = Qx + N2;
  const float* Qz = Qy + N2;
  const float* lam = Qx + 3 * N2;
  float q[N][N];
  auto load_q = [&](const float* Q) {
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int k = 0; k < N; ++k) q[i][k] = Q[i * N + k];
  };
  // one line of w (first element f, stride sd): w <- Q^float w (TR) or Q w
  auto line = [&](int f, int sd, bool tr) {
    float v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = w[f + i * sd];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      float a = (tr ? q[0][k] : q[k][0]) * v[0];
#pragma unroll
      for (int i = 1; i < N; ++i) a = fma(tr ? q[i][k] : q[k][i], v[i], a);
      w[f + k * sd] = a;
    }
  };
  if (active) {  // (Q_x)^float along the x-lines (j, l = t)
    load_q(Qx);
#pragma unroll
    for (int j = 0; j < N; ++j) line(t * N2 + j * N, 1, true);
  }
  __syncthreads();
  if (active) {  // (Q_y)^float along the y-lines (i, l = t)
    load_q(Qy);
#pragma unroll
    for (int i = 0; i < N; ++i) line(t * N2 + i, N, true);
  }
  __syncthreads();
  float acc = 0.0f;
  if (active) {  // z-lines (i, j = t): (Q_z)^T, the scaling, Q_z
    load_q(Qz);
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float v[N], u[N];
#pragma unroll
      for (int l = 0; l < N; ++l) v[l] = w[l * N2 + t * N + i];
      const float lxy = lam[i] + lam[N + t];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        float a = q[0][k] * v[0];
#pragma unroll
        for (int l = 1; l < N; ++l) a = fma(q[l][k], v[l], a);
        u[k] = a * __fdividef(1.0f, lxy + lam[2 * N + k]);
        acc = fma(a, u[k], acc);
      }
#pragma unroll
      for (int l = 0; l < N; ++l) {
        float a = q[l][0] * u[0];
#pragma unroll
        for (int k = 1; k < N; ++k) a = fma(q[l][k], u[k], a);
        w[l * N2 + t * N + i] = a;
      }
    }
  }
  __syncthreads();
  if (active) {  // Q_y along the y-lines
    load_q(Qy);
#pragma unroll
    for (int i = 0; i < N; ++i) line(t * N2 + i, N, false);
  }
  __syncthreads();
  if (active) {  // Q_x along the x-lines
    load_q(Qx);
#pragma unroll
    for (int j = 0; j < N; ++j) line(t * N2 + j * N, 1, false);
  }
  __syncthreads();
  return acc;
}

// Sum of one double per thread over the block, fixed order; valid in warp 0.
template <int NT>
__device__ __forceinline__ double block_total(double v, double* rd) {
  rd[threadIdx.x] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    for (int i = threadIdx.x; i < NT; i += 32) s += rd[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  }
  __syncthreads();
  return s;
}

// The FP32 form, of the mixed iteration (kron_finish MODE 2).
template <int N>
__global__ void __launch_bounds__(KronCfg<N>::THREADS)
k_kron_apply(const float* __restrict__ KD, const float* __restrict__ r, float* __restrict__ z,
             long long ncells, double* __restrict__ partials, DGCGState* st) {
  using KC = KronCfg<N>;
  constexpr int C = KC::C, N3 = N * N * N, NT = KC::THREADS, KS = KC::KS;
  if (st->done || st->ru_skip == 0) return;  // ru_skip = 0: an FP64 refinement is pending
  __shared__ float sw[C * N3], sq[C * KS];
  __shared__ double rd[NT];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  for (int i = threadIdx.x; i < nblk * N3; i += NT) sw[i] = r[c0 * N3 + i];
  for (int i = threadIdx.x; i < nblk * KS; i += NT) sq[i] = KD[c0 * KS + i];
  __syncthreads();
  const float acc = kron_solve_cells<N>(sw, sq, nblk);
  for (int i = threadIdx.x; i < nblk * N3; i += NT) z[c0 * N3 + i] = sw[i];
  const double part = block_total<NT>((double)acc, rd);
  kron_finish<NT, 2>(part, partials, st, rd);
}

// z = M^-1 r in FP64 vectors, contractions in block fixed point: in FP64 the
// 6n multiply-adds and the division per DOF kept the FP64 pipe busy for
// 6n + 12 instructions (0.94 ms at 48^3 Q4); here they are 6n integer
// products of 12 issue cycles each and the divisions are done once,
// in k_kron_fix.  KX: the 1D factors [c][x,y,z][i][j] 2^60; winv: 1 / (lx + ly
// + lz) [c][i][j + n l].  The transformed residual t is scaled to w t with the
// cell's 2-norm again below 2^60, whatever the spread of the eigenvalues; <z, r> =
// sum w t^2 accumulates in 64-bit integers per thread.
template <int N, int MODE>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_kron_apply_fx(const FxPair* __restrict__ KX, const double* __restrict__ winv,
                const double* __restrict__ r, double* __restrict__ z, long long ncells,
                double* __restrict__ partials, DGCGState* st) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS, N2 = N * N, N3 = N * N * N;
  constexpr int SY = LinePad<N>::SY, SZ = LinePad<N>::SZ, SC = LinePad<N>::SC, NS = FxSmem<N, T>::NS;
  if (MODE != 1 && st->done) return;
  __shared__ long long s[C * SC];
  __shared__ FxPair sq[C * 3 * N2];
  __shared__ double rd[T];
  __shared__ unsigned slots[4 * NS];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  const int lc = threadIdx.x / N2, pt = threadIdx.x - lc * N2;
  const int pp = pt % N, qq = pt / N;
  const bool active = lc < nblk;
  const long long c = c0 + (active ? lc : 0);
  long long* sc = s + lc * SC;
  const FxPair* Q = sq + lc * 3 * N2;
  double rv[N], w[N];
#pragma unroll
  for (int l = 0; l < N; ++l) rv[l] = active ? r[c * N3 + l * N2 + pt] : 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) w[i] = winv[c * N3 + i * N2 + pt];
  for (int i = threadIdx.x; i < nblk * 3 * N2; i += T) sq[i] = KX[c0 * 3 * N2 + i];
  for (int i = threadIdx.x; i < 4 * NS; i += T) slots[i] = 0;
  unsigned big = 0;
#pragma unroll
  for (int l = 0; l < N; ++l) big = max(big, fx_abs_hi(rv[l]));
  __syncthreads();
  const int E = fx_exponent(fx_cell_max<N, T>(big, lc, slots));
  const int k0 = fx_norm_scale<N, T>(rv, E, lc, slots + 2 * NS);
  long long v[N], u[N];
#pragma unroll
  for (int l = 0; l < N; ++l) v[l] = fx_from_double(rv[l], k0, E);
  // u[k] = sum_i Q[i][k] v[i] (tr) or sum_i Q[k][i] v[i]
  auto line = [&](int d, bool tr) {
    FxVal e[N];
#pragma unroll
    for (int i = 0; i < N; ++i) e[i] = fx_split(v[i]);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      FxAcc A = fx_zero();
#pragma unroll
      for (int i = 0; i < N; ++i) fx_mac(A, Q[d * N2 + (tr ? i * N + k : k * N + i)], e[i]);
      u[k] = fx_value(A);
    }
  };
  auto put = [&](int at, int step) {
#pragma unroll
    for (int i = 0; i < N; ++i) sc[at + i * step] = u[i];
    cell_sync<N>();
  };
  auto get = [&](int at, int step) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = sc[at + i * step];
  };
  const int zl = qq * SY + pp, yl = qq * SZ + pp, xl = qq * SZ + pp * SY;
  line(2, true);  // z-lines
  put(zl, SZ);
  get(yl, SY);
  line(1, true);
  put(yl, SY);
  get(xl, 1);
  line(0, true);
  // w t: mantissa of w in [2^59, 2^60), its exponent with the magnitude of t
  unsigned top = 0;
  int ew[N];
  FxVal m[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const long long b = __double_as_longlong(w[i]);
    ew[i] = (int)(b >> 52) - 1022;
    m[i] = fx_split(((b & 0xfffffffffffffll) | 0x10000000000000ll) << 7);
    // biased to stay positive
    top = max(top, (unsigned)(fx_bits(fx_mag_hi(u[i])) + ew[i] + 4096));
  }
  const int B = (int)fx_cell_max<N, T>(top, lc, slots + NS) - 4096;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    FxAcc A = fx_zero();
    fx_mac(A, fx_pair(u[i]), m[i]);
    const int sh = ew[i] + 60 - B;
    v[i] = fx_shift(fx_value(A), sh < -63 ? -63 : sh);
  }
  const int up = fx_norm_shift<N, T>(v, 60, lc, slots + 3 * NS);
  FxAcc dot = {0, 0};
#pragma unroll
  for (int i = 0; i < N; ++i) {
    v[i] = fx_shift(v[i], up);
    fx_mac(dot, fx_pair(u[i]), fx_split(v[i]));
  }
  // v stands for v 2^(B - 60 - up - k0); <z, r> sums t v, t 2^-k0
  const bool bad = E >= FX_NAN;
  const double qnan = __longlong_as_double(0x7ff8000000000000ll);
  const int ez = B - 60 - up - k0;
  const double acc = !active ? 0.0
                     : bad   ? qnan
                             : fx_scale(fma((double)dot.m, 0x1p-30, (double)dot.h),
                                        ez - k0 + 60);
  line(0, false);
  put(xl, 1);
  get(yl, SY);
  line(1, false);
  put(yl, SY);
  get(zl, SZ);
  line(2, false);
  if (active) {
#pragma unroll
    for (int l = 0; l < N; ++l) {
      const double zv = bad ? qnan : fx_to_double(u[l], ez);
      z[c * N3 + l * N2 + pt] = zv;
    }
  }
  const double part = block_total<T>(acc, rd);
  kron_finish<T, MODE>(part, partials, st, rd);
}

// Factors of the FP64 application from the FP64 ones: the eigenbases as
// fixed-point pairs, one reciprocal per DOF.  One thread per DOF.  A cell whose
// three factors share a zero eigenvalue (every face coefficient zero) has no
// inverse: its reciprocal raises *flag, since the application reads mantissas
// and would take an infinity for a number.
template <int N>
__global__ void k_kron_fix(const double* __restrict__ K64, FxPair* __restrict__ KX,
                           double* __restrict__ winv, long long ncells, int* flag) {
  constexpr int N2 = N * N, N3 = N * N * N, KS = 3 * N2 + 3 * N;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ncells * N3) return;
  const long long c = t / N3;
  const int k = (int)(t - c * N3);
  const double* L = K64 + c * KS + 3 * N2;
  const int i = k / N2, j = k % N, l = (k / N) % N;
  const double w = 1.0 / (L[i] + L[N + j] + L[2 * N + l]);
  winv[t] = w;
  if (!(w > 0.0) || !isfinite(w)) atomicOr(flag, 1);
  for (int e = k; e < 3 * N2; e += N3)
    KX[c * 3 * N2 + e] = fx_pair(__double2ll_rn(K64[c * KS + e] * 0x1p60));
}

template <int N>
struct KronFixF {
  template <typename T>
  static cudaError_t run(const double* K64, FxPair* KX, double* winv, long long ncells,
                         int* flag, cudaStream_t s) {
    const long long n = ncells * N * N * N;
    k_kron_fix<N><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(K64, KX, winv, ncells, flag);
    return cudaGetLastError();
  }
};

// The factors in the scaled Gauss-point basis: per cell and direction
// Qhat = q Q with q[a][i] = sqrt(w_a) L_i(xi_a) (orthogonal), the eigenvalues
// unchanged: Q M Q^T is again a Kronecker sum with these eigenbases.  One
// thread per (cell, direction).
template <int N>
__global__ void k_kron_rotate(const double* __restrict__ K64, double* __restrict__ KN64,
                              float* __restrict__ KN32, long long ncells,
                              const __grid_constant__ DGTab<double> tab) {
  constexpr int N2 = N * N, KS = 3 * N2 + 3 * N;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 3 * ncells) return;
  const long long c = t / 3;
  const int d = (int)(t - 3 * c);
  const double* Q = K64 + c * KS + d * N2;
  double* Q64 = KN64 + c * KS + d * N2;
  float* Q32 = KN32 + c * KS + d * N2;
  for (int a = 0; a < N; ++a) {
    const double sw = sqrt(tab.w[a]);
    for (int j = 0; j < N; ++j) {
      double acc = 0.0;
      for (int i = 0; i < N; ++i) acc = fma(tab.B[a][i], Q[i * N + j], acc);
      Q64[a * N + j] = sw * acc;
      Q32[a * N + j] = (float)(sw * acc);
    }
  }
  const double* L = K64 + c * KS + 3 * N2 + d * N;
  for (int j = 0; j < N; ++j) {
    KN64[c * KS + 3 * N2 + d * N + j] = L[j];
    KN32[c * KS + 3 * N2 + d * N + j] = (float)L[j];
  }
}

template <int N>
struct KronRotateF {
  template <typename T>
  static cudaError_t run(dg_mesh* m, cudaStream_t s) {
    const long long threads = 3 * m->ncells;
    k_kron_rotate<N><<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(
        m->kron64, m->kronN64, m->kronN32, m->ncells, m->tab64);
    return cudaGetLastError();
  }
};

template <int N>
struct KronSetupF {
  template <typename T>
  static cudaError_t run(dg_mesh* m, cudaStream_t s) {
    const long long threads = 3 * m->ncells;
    k_kron_setup<N><<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(
        m->kt64, m->gh64, m->kron64, m->kron32, m->ncells, m->N, m->dflag, m->tab64);
    return cudaGetLastError();
  }
};

template <int N>
struct KronApplyF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, const void* r, void* z, int mode, cudaStream_t s) {
    using K32 = KronCfg<N>;
    // inside a solve in the scaled Gauss-point basis: the rotated factors
    const FxPair* fx = m->nodal_op ? m->kronNX : m->kronX;
    const float* f32 = m->nodal_op ? m->kronN32 : m->kron32;
    const unsigned bx = (unsigned)((m->ncells + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    const unsigned b32 = (unsigned)((m->ncells + K32::C - 1) / K32::C);
    switch (mode) {
      case DG_KRON_FP64:
        k_kron_apply_fx<N, 0><<<bx, Cfg<N>::THREADS, 0, s>>>(
            fx, m->kronW, (const double*)r, (double*)z, m->ncells, m->partials_cells, m->state);
        break;
      case DG_KRON_FP64_INIT:
        k_kron_apply_fx<N, 1><<<bx, Cfg<N>::THREADS, 0, s>>>(
            fx, m->kronW, (const double*)r, (double*)z, m->ncells, m->partials_cells, m->state);
        break;
      default:
        k_kron_apply<N><<<b32, K32::THREADS, 0, s>>>(f32, (const float*)r, (float*)z, m->ncells,
                                                     m->partials_cells, m->state);
        break;
    }
    return cudaGetLastError();
  }
};

}  // namespace
}  // namespace dgk

int dg_ensure_kron(dg_mesh* m, cudaStream_t s) {
  if (m->has_kron) return DG_OK;
  const size_t KS = (size_t)(3 * m->n * m->n + 3 * m->n);
  if (m->kron64 == nullptr) {
    cudaError_t e = cudaMalloc((void**)&m->kron64, sizeof(double) * KS * (size_t)m->ncells);
    if (e == cudaSuccess)
      e = cudaMalloc((void**)&m->kron32, sizeof(float) * KS * (size_t)m->ncells);
    if (e != cudaSuccess) return dg_cuda_fail(e, "Kronecker cell blocks: storage");
  }
  DG_CUDA(cudaMemsetAsync(m->dflag, 0, sizeof(int), s));
  cudaError_t e = dgk::dispatch_n<double, dgk::KronSetupF>(m->n, m, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "Kronecker cell blocks: setup");
  int flag = 0;
  DG_CUDA(cudaMemcpyAsync(&flag, m->dflag, sizeof(int), cudaMemcpyDeviceToHost, s));
  DG_CUDA(cudaStreamSynchronize(s));
  if (flag)
    return dg_fail(DG_ERR_BREAKDOWN,
                   "Kronecker cell blocks: a 1D factor has a negative eigenvalue");
  m->has_kron = true;
  return DG_OK;
}

int dg_ensure_kron_nodal(dg_mesh* m, cudaStream_t s) {
  int rc = dg_ensure_kron(m, s);
  if (rc || m->has_kron_nodal) return rc;
  const size_t KS = (size_t)(3 * m->n * m->n + 3 * m->n);
  if (m->kronN64 == nullptr) {
    cudaError_t e = cudaMalloc((void**)&m->kronN64, sizeof(double) * KS * (size_t)m->ncells);
    if (e == cudaSuccess)
      e = cudaMalloc((void**)&m->kronN32, sizeof(float) * KS * (size_t)m->ncells);
    if (e != cudaSuccess) return dg_cuda_fail(e, "Kronecker cell blocks (point basis): storage");
  }
  cudaError_t e = dgk::dispatch_n<double, dgk::KronRotateF>(m->n, m, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "Kronecker cell blocks (point basis): rotation");
  m->has_kron_nodal = true;
  return DG_OK;
}

// The fixed-point factors of the FP64 application in the current basis.
static int ensure_kron_fx(dg_mesh* m, cudaStream_t s) {
  bool& has = m->nodal_op ? m->has_kron_nx : m->has_kron_x;
  FxPair*& X = m->nodal_op ? m->kronNX : m->kronX;
  if (has) return DG_OK;
  const size_t nq = (size_t)(3 * m->n * m->n) * (size_t)m->ncells;
  if (X == nullptr) DG_CUDA(cudaMalloc((void**)&X, sizeof(FxPair) * nq));
  if (m->kronW == nullptr)
    DG_CUDA(cudaMalloc((void**)&m->kronW, sizeof(double) * (size_t)m->ndofs));
  DG_CUDA(cudaMemsetAsync(m->dflag, 0, sizeof(int), s));
  cudaError_t e = dgk::dispatch_n<double, dgk::KronFixF>(
      m->n, (const double*)(m->nodal_op ? m->kronN64 : m->kron64), X, m->kronW, m->ncells,
      m->dflag, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "Kronecker cell blocks: fixed-point factors");
  int flag = 0;
  DG_CUDA(cudaMemcpyAsync(&flag, m->dflag, sizeof(int), cudaMemcpyDeviceToHost, s));
  DG_CUDA(cudaStreamSynchronize(s));
  if (flag)
    return dg_fail(DG_ERR_BREAKDOWN, "Kronecker cell blocks: a cell's block is singular");
  has = true;
  return DG_OK;
}

int dg_launch_kron_apply(const dg_mesh* m, const void* r, void* z, int mode, cudaStream_t s) {
  if (mode == DG_KRON_FP64_INIT)  // runs before the iterations are captured
    if (int rc = ensure_kron_fx(const_cast<dg_mesh*>(m), s)) return rc;
  cudaError_t e = dgk::dispatch_n<double, dgk::KronApplyF>(m->n, m, r, z, mode, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "Kronecker cell blocks: apply");
  return DG_OK;
}
