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

// XL: FxLoad, or FxDirection inside a CG iteration (then x.begin() reads beta)
template <int N, bool MODAL, typename XL>
__global__ void __launch_bounds__(Cfg<N>::THREADS)
k_trace_fx(XL x, long long* __restrict__ U, long long* __restrict__ TR,
           int* __restrict__ expU, int* __restrict__ mark, long long cbeg, long long cend,
           const int* skip, const __grid_constant__ DGTabX tab) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS;
  dg_release_next();
  dg_wait_before();
  if (skip != nullptr && *skip) return;
  __shared__ long long smem[(FxSmem<N, T>::trace + 7) / 8];
  x.begin();
  const long long c0 = cbeg + (long long)blockIdx.x * C;
  const int nblk = (int)((cend - c0) < C ? (cend - c0) : C);
  fx_trace_cells<N, MODAL, T>(x, U, TR, expU, mark, c0, nblk, tab, smem);
}

// Kernel parameter with the data of fx_cells_wide: in the point basis only.
template <bool MODAL>
struct FxWideArg {
  __device__ __forceinline__ FxWide get() const { return {}; }
};
template <>
struct FxWideArg<false> {
  const double *kt, *gh;
  const int* mark;
  DGTabN<double> tn;
  __device__ __forceinline__ FxWide get() const { return {kt, gh, mark, &tn}; }
};
template <bool MODAL>
FxWideArg<MODAL> wide_arg(const dg_mesh* m) {
  if constexpr (MODAL)
    return {};
  else
    return {m->kt64, m->gh64, m->markU, m->tabN64};
}

// Resident blocks per SM that the register allocation of pass 2 aims at.  It
// waits for memory most of the time, so more warps help until values spill.
// Measured (us; no aim / chosen / one more): 64^3 Q3 370 / 340 / 354,
// 27^3 Q5 144 / 127 / 128, 24^3 Q6 201 / 156 / 161, 22^3 Q7 201 / 170 / 190,
// 20^3 Q8 231 / 227 / 227; with ten in place of one more (Legendre, point basis):
// 100^3 Q1 181 / 201 / 186, 214 / 198 / 185, 64^3 Q2 166 / 167 / 162,
// 168 / 151 / 146, 40^3 Q4 193 / 185 / 226, 193 / 169 / 218.
template <int N>
struct FxCellBlocks {
  static constexpr int value = N <= 5 ? 8 : N == 6 ? 5 : N == 7 ? 4 : N == 8 ? 5 : 3;
};

template <int N, bool MODAL>
__global__ void __launch_bounds__(Cfg<N>::THREADS, FxCellBlocks<N>::value)
k_cell_fx(const void* xU, const long long* TR, const int* expU,
          const FxPair* __restrict__ lineop,
          const FxPair* __restrict__ gam, const int* __restrict__ expM,
          const int* __restrict__ expG, double* __restrict__ y, long long cbeg, long long cend,
          int Nc, const int* skip, const __grid_constant__ DGTabX tab,
          const __grid_constant__ FxWideArg<MODAL> wd) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS;
  dg_release_next();
  dg_wait_before();
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const long long c0 = cbeg + (long long)blockIdx.x * C;
  const int nblk = (int)((cend - c0) < C ? (cend - c0) : C);
  fx_cell_cells<N, MODAL, T>(xU, TR, expU, lineop, gam, expM, expG, wd.get(), FxStore{y}, c0,
                             nblk, Nc, tab, reinterpret_cast<long long*>(smem_raw));
}

// Inside a CG iteration (Section 2.4) the passes take the vector work along.
// With FP64 passes that was slower than separate kernels (they shared the FP64
// pipe); the fixed-point passes leave that pipe idle, and the two vector kernels,
// their traffic (40 B per DOF) and their launches go.  32^3 Q3 with Jacobi:
// 236 -> 190 ms per solve, together with the shorter pass 2 and reductions.
// Pass 1 of p = z + beta p, z = r, dinv r (PC) or M^-1 r already formed.
template <bool PC>
struct FxDirection {
  double* p;
  const double *z, *dinv;
  const DGCGState* st;
  double beta;
  __device__ __forceinline__ void begin() { beta = st->beta; }
  __device__ __forceinline__ double operator()(long long i) const {
    const double v = fma(beta, p[i], PC ? dinv[i] * z[i] : z[i]);
    p[i] = v;
    return v;
  }
};

// Pass 2 with <p, q> and alpha = rho / <p, q>: the products of point values are
// integers already there (from p and q in FP64 they were 8 bytes of traffic and an
// FP64 instruction per DOF: 201 -> 190 ms per solve); one partial per block, added
// by the last block in a fixed order.
template <int N, bool MODAL>
__global__ void __launch_bounds__(Cfg<N>::THREADS, FxCellBlocks<N>::value)
k_cell_dot_fx(const void* xU, const long long* TR, const int* expU,
              const FxPair* __restrict__ lineop,
              const FxPair* __restrict__ gam, const int* __restrict__ expM,
              const int* __restrict__ expG, double* __restrict__ q, long long ncells, int Nc,
              double* __restrict__ partials, DGCGState* st, const __grid_constant__ DGTabX tab,
              const __grid_constant__ FxWideArg<MODAL> wd) {
  constexpr int C = Cfg<N>::CPB, T = Cfg<N>::THREADS;
  dg_release_next();
  dg_wait_before();
  if (st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ bool is_last;
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  const double acc = fx_cell_cells<N, MODAL, T, true>(
      xU, TR, expU, lineop, gam, expM, expG, wd.get(), FxStore{q}, c0, nblk, Nc, tab,
      reinterpret_cast<long long*>(smem_raw));
  __syncthreads();
  double* rd = reinterpret_cast<double*>(smem_raw);
  static_assert(FxSmem<N, T>::cell >= sizeof(double) * T, "reduction scratch");
  rd[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = 0.0;
    for (int i = threadIdx.x; i < T; i += 32) t += rd[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (threadIdx.x == 0) {
      partials[blockIdx.x] = t;
      __threadfence();
      is_last = (atomicAdd(&st->ticket, 1u) == gridDim.x - 1);
    }
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const double tot = last_block_total<T>(partials, (int)gridDim.x, rd);
  if (threadIdx.x == 0) {
    st->pq = tot;
    if (!(tot > 0.0) || !isfinite(tot)) {
      st->breakdown = 1;
      st->done = 1;
      st->ru_skip = 1;
    } else {
      st->alpha = st->rho / tot;
    }
    st->ticket = 0u;
  }
}

// Line operators, face coefficients and their exponents from K and h gamma: one
// thread per cell, direction and line.  Integer arithmetic throughout: the volume
// part with K in units of the cell's largest, the faces' part with the 53 bits of
// h gamma, each a product with constants of the 1D tables under a scale of its own,
// rounded to the larger one.  (Under one scale the faces' bound, sigma times
// the volume part's, took up to 7 bits from an operator whose K is large at few
// points, and then a smooth vector, whose terms cancel, lost more than in FP64.)
template <int N>
struct FxSetup {
  static constexpr int L = 3 * N * N;                    // lines of a cell
  static constexpr int C = N == 2 ? 12 : N == 3 ? 6 : N == 4 ? 4 : N == 5 ? 2 : 1;
  static constexpr int THREADS = C * L;
};

// Registers for six (n = 3) and five (n = 4) blocks per SM, which cost no spill.
template <int N>
__global__ void __launch_bounds__(FxSetup<N>::THREADS, N == 3 ? 6 : N == 4 ? 5 : 0)
k_lines_fx(const double* __restrict__ K, const double* __restrict__ gh,
           FxPair* __restrict__ lineop, FxPair* __restrict__ gam, int* __restrict__ expM,
           int* __restrict__ expN, int* __restrict__ expG, long long ncells, int Nc, int cg,
           const __grid_constant__ DGTabXSetup t) {
  constexpr int C = FxSetup<N>::C, L = FxSetup<N>::L, T = FxSetup<N>::THREADS;
  constexpr int N2 = N * N, N3 = N * N * N, NP = N * (N + 1) / 2;
  __shared__ long long sk[C * N3];
  __shared__ unsigned kmax[C];
  __shared__ unsigned long long rmax[C][3];
  __shared__ int sbad[C], stop[C], smark[C];
  const long long c0 = (long long)blockIdx.x * C;
  const int nblk = (int)((ncells - c0) < C ? (ncells - c0) : C);
  if (threadIdx.x < C) {
    kmax[threadIdx.x] = 0;
    sbad[threadIdx.x] = 0;
    smark[threadIdx.x] = 0;
    stop[threadIdx.x] = -FX_NAN;
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
  bool edge[2] = {false, false};
  long long mant[2] = {0, 0};                // h gamma 2^(60 - eg), in [2^59, 2^60)
  int eg[2] = {-(1 << 20), -(1 << 20)};
  if (active) {
    const unsigned cu = (unsigned)c, nu = (unsigned)Nc;
    const int crd = (int)(dir == 0 ? cu % nu : dir == 1 ? (cu / nu) % nu : cu / nu / nu);
    edge[0] = crd == 0;
    edge[1] = crd == Nc - 1;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const double w = gh[c * 6 + 2 * dir + m];
      bad = bad || fx_abs_hi(w) >= 0x7ff00000u;
      const bool sub = fx_abs_hi(w) < 0x00100000u;
      const double w2 = sub ? w * 0x1p64 : w;
      if (w > 0.0) {
        mant[m] = ((__double_as_longlong(w2) & 0xfffffffffffffll) | 0x10000000000000ll) << 7;
        eg[m] = (int)(fx_abs_hi(w2) >> 20) - 1022 - (sub ? 64 : 0);
      }
      if (pt == 0) {  // an octave higher a mantissa could round to 2^61, past a pair's end
        gam[c * 6 + 2 * dir + m] = fx_pair(mant[m]);
        expG[c * 6 + 2 * dir + m] = w > 0.0 ? eg[m] + 1 + cg : -2 * FX_NAN;
      }
    }
    if (pt == 0) atomicMax(&stop[lc], max(eg[0], eg[1]) + t.cF);
  }
  __syncthreads();
  // the common exponent: volume part and two faces, each at most 2^60
  const int E0 = active ? max(eK + t.cV, stop[lc]) : 0;
  unsigned long long R = 0;  // the line's largest row sum
  if (active) {
    const int step = dir == 0 ? 1 : dir == 1 ? N : N2;
    const int at = lc * N3 + (dir == 0 ? N * (p + N * q) : dir == 1 ? p + N2 * q : p + N * q);
    FxVal k[N];
#pragma unroll
    for (int f = 0; f < N; ++f) k[f] = fx_split(sk[at + f * step]);
    const int egm = max(eg[0], eg[1]);  // both faces under the larger exponent
    const FxVal g[2] = {fx_split(mant[0] >> min(egm - eg[0], 63)),
                        fx_split(mant[1] >> min(egm - eg[1], 63))};
    const int sV = min(E0 - eK - t.cV, 62), sF = min(E0 - egm - t.cF, 62);
    unsigned long long rs[N];
#pragma unroll
    for (int e = 0; e < N; ++e) rs[e] = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
      for (int j = i; j < N; ++j) {
        const int ij = packed<N>(i, j), ji = packed<N>(N - 1 - i, N - 1 - j);
        FxAcc A = fx_zero<1>(), B = fx_zero();
#pragma unroll
        for (int f = 0; f < N; ++f) fx_mac(A, t.DD[f][ij], k[f]);
        fx_mac(B, edge[0] ? t.F[1][ij] : t.F[0][ij], g[0]);
        fx_mac(B, edge[1] ? t.F[1][ji] : t.F[0][ji], g[1]);
        const long long v = fx_round(fx_value<1>(A), sV) + fx_round(fx_value(B), sF);
        M[ij] = v;
        const unsigned long long mag = (unsigned long long)(v < 0 ? -v : v) >> 4;
        rs[i] += mag;
        if (i != j) rs[j] += mag;
      }
    }
#pragma unroll
    for (int e = 0; e < N; ++e) R = rs[e] > R ? rs[e] : R;
    atomicMax(&rmax[lc][dir], R + N);
    if (bad) sbad[lc] = 1;
  }
  __syncthreads();
  if (active && R < max(rmax[lc][0], max(rmax[lc][1], rmax[lc][2])) >> 4)
    atomicOr(&smark[lc], 1 << dir);
  __syncthreads();
  if (!active) return;
  // the sum of the directions' largest row sums to (2^60, 2^61]: each direction
  // holds the cell's largest K against table rows of similar size (within 2^6 for
  // every n), so an entry stays clear of a pair's upper end
  const int bits = 68 - __clzll((long long)(rmax[lc][0] + rmax[lc][1] + rmax[lc][2]));
  const int up = 61 - bits;
  if (t2 == 0) {
    const int e = sbad[lc] ? FX_NAN : E0 - up + 1;
    expM[c] = e;
    expN[c] = e + (smark[lc] == FX_MARKS ? FX_WIDE : 0);
  }
  FxPair* out = lineop + ((c * 3 + dir) * NP) * N2 + pt;
#pragma unroll
  for (int k2 = 0; k2 < NP; ++k2)
    out[k2 * N2] = fx_pair(up < 0 ? fx_round(M[k2], -up) : M[k2] << up);
}

// K from the kept h w_q K.
__global__ void k_point_coefficient(const double* __restrict__ kt, double* __restrict__ K,
                                    long long ndofs, int n, double h,
                                    const __grid_constant__ DGTab<double> tab) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ndofs) return;
  const int q = (int)(t % ((long long)n * n * n));
  K[t] = kt[t] / (h * (tab.w[q % n] * tab.w[(q / n) % n] * tab.w[q / (n * n)]));
}

template <int N>
struct FixedF {
  static constexpr size_t SMEM = FxSmem<N, Cfg<N>::THREADS>::cell;
  template <bool MODAL>
  static cudaError_t pass(const dg_mesh* m, int pass, const double* x, double* y, long long cbeg,
                          long long cend, const int* skip, cudaStream_t s) {
    if (cend <= cbeg) return cudaSuccess;
    const unsigned blocks = (unsigned)((cend - cbeg + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    long long* U = reinterpret_cast<long long*>(m->U64);
    long long* TR = reinterpret_cast<long long*>(m->TR64);
    if (pass == 1)
      return dg_launch_after(k_trace_fx<N, MODAL, FxLoad>, blocks, Cfg<N>::THREADS, 0, s, FxLoad{x},
                             U, TR, m->expU, m->markU, cbeg, cend, skip, m->tabX);
    return dg_launch_after(k_cell_fx<N, MODAL>, blocks, Cfg<N>::THREADS, SMEM, s,
                           MODAL ? (const void*)U : (const void*)x, TR, m->expU, m->lineopX,
                           m->gamX, MODAL ? m->expM : m->expN, m->expG, y, cbeg, cend, m->N, skip,
                           m->tabX, wide_arg<MODAL>(m));
  }
  template <typename T>
  static cudaError_t run(const dg_mesh* m, bool modal, int which, const double* x, double* y,
                         long long cbeg, long long cend, const int* skip, cudaStream_t s) {
    return modal ? pass<true>(m, which, x, y, cbeg, cend, skip, s)
                 : pass<false>(m, which, x, y, cbeg, cend, skip, s);
  }
};

// q = A p with p = z + beta p and alpha, on the mesh's solver state.
template <int N>
struct FixedCgF {
  template <bool MODAL, bool PC>
  static cudaError_t go(const dg_mesh* m, const double* z, const double* dinv, double* p,
                        double* q, cudaStream_t s) {
    const unsigned blocks = (unsigned)((m->ncells + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    long long* U = reinterpret_cast<long long*>(m->U64);
    long long* TR = reinterpret_cast<long long*>(m->TR64);
    cudaError_t e = dg_launch_after(
        k_trace_fx<N, MODAL, FxDirection<PC>>, blocks, Cfg<N>::THREADS, 0, s,
        FxDirection<PC>{p, z, dinv, m->state, 0.0}, U, TR, m->expU, m->markU, 0ll, m->ncells,
        &m->state->done, m->tabX);
    if (e != cudaSuccess) return e;
    return dg_launch_after(k_cell_dot_fx<N, MODAL>, blocks, Cfg<N>::THREADS, FixedF<N>::SMEM, s,
                           MODAL ? (const void*)U : (const void*)p, TR, m->expU, m->lineopX,
                           m->gamX, MODAL ? m->expM : m->expN, m->expG, q, m->ncells, m->N,
                           m->partials_cells, m->state, m->tabX, wide_arg<MODAL>(m));
  }
  template <typename T>
  static cudaError_t run(const dg_mesh* m, const double* z, const double* dinv, double* p,
                         double* q, cudaStream_t s) {
    if (m->nodal_op)
      return dinv ? go<false, true>(m, z, dinv, p, q, s) : go<false, false>(m, z, dinv, p, q, s);
    return dinv ? go<true, true>(m, z, dinv, p, q, s) : go<true, false>(m, z, dinv, p, q, s);
  }
};

template <int N>
struct FixedTraceF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, const double* x, long long* U, long long* TR,
                         int* expU, cudaStream_t s) {
    const unsigned blocks = (unsigned)((m->ncells + Cfg<N>::CPB - 1) / Cfg<N>::CPB);
    k_trace_fx<N, true><<<blocks, Cfg<N>::THREADS, 0, s>>>(FxLoad{x}, U, TR, expU, nullptr, 0,
                                                          m->ncells, nullptr, m->tabX);
    return cudaGetLastError();
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
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_cell_dot_fx<N, true>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FixedF<N>::SMEM);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_cell_dot_fx<N, false>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FixedF<N>::SMEM);
    return e;
  }
};

template <int N>
struct FixedSetupF {
  template <typename T>
  static cudaError_t run(const dg_mesh* m, const double* K, cudaStream_t s) {
    using S = FxSetup<N>;
    k_lines_fx<N><<<(unsigned)((m->ncells + S::C - 1) / S::C), S::THREADS, 0, s>>>(
        K, m->gh64, m->lineopX, m->gamX, m->expM, m->expN, m->expG, m->ncells, m->N, m->tabX.cg,
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

int dg_restore_fixed(dg_mesh* m, cudaStream_t s) {
  double* K = m->U64;  // the point values of an application: free between calls
  dgk::k_point_coefficient<<<(unsigned)((m->ndofs + 255) / 256), 256, 0, s>>>(
      m->kt64, K, m->ndofs, m->n, m->h, m->tab64);
  DG_CUDA(cudaGetLastError());
  return dg_setup_fixed(m, K, s);
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

int dg_launch_fixed_cg(const dg_mesh* m, const double* z, const double* dinv, double* p,
                       double* q, cudaStream_t s) {
  cudaError_t e = dgk::dispatch_n<double, dgk::FixedCgF>(m->n, m, z, dinv, p, q, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "CG operator (fp64) launch");
  return DG_OK;
}

int dg_launch_fixed_trace(const dg_mesh* m, const double* x, double* U, double* TR, int* expU,
                          cudaStream_t s) {
  cudaError_t e = dgk::dispatch_n<double, dgk::FixedTraceF>(
      m->n, m, x, reinterpret_cast<long long*>(U), reinterpret_cast<long long*>(TR), expU, s);
  if (e != cudaSuccess) return dg_cuda_fail(e, "trace (fp64) launch");
  return DG_OK;
}
