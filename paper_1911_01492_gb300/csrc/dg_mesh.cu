// Mesh handle, coefficient setup, error reporting and the apply entry points.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "dg_apply_impl.cuh"

// ---------------------------------------------------------------------------
// error reporting
// ---------------------------------------------------------------------------
static thread_local char g_err[512] = "";

int dg_fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}

int dg_cuda_fail(cudaError_t e, const char* what) {
  int code = (e == cudaErrorMemoryAllocation) ? DG_ERR_OOM : DG_ERR_CUDA;
  return dg_fail(code, "%s: %s (%s)", what, cudaGetErrorName(e), cudaGetErrorString(e));
}

extern "C" const char* dg_last_error(void) { return g_err; }

// ---------------------------------------------------------------------------
// coefficient setup kernels
// ---------------------------------------------------------------------------

// cells per block of k_coef_cells: about 128 mirror groups, at most 24 KB of K
static __host__ __device__ constexpr int coef_cells(int n) {
  return n == 2 ? 128 : n <= 4 ? 16 : n <= 6 ? 8 : n <= 8 ? 4 : 2;
}

// Kt = h w_q K (FP64, and FP32 unless kt32 is NULL), Kbar = exp(sum_q w_q log K)
// on coef_cells(n) cells per block.  Invalid K (<= 0, NaN, inf) raises bit 0 of
// *flag.  A logarithm costs about 30 FP64 instructions at one per 64 cycles, so
// the points that mirror each other about the cell's middle planes, which
// share their weight, are multiplied first and one logarithm serves the
// (up to) eight of them: mantissas in [1, 2) and the sum of the exponents, so
// that nothing over- or underflows.  The product's rounding, 2^-53 per factor,
// weighs w_q once, less than the eight roundings of separate logarithms.
// 32^3 Q3: 179 -> 49 us.
__global__ void __launch_bounds__(256)
k_coef_cells(const double* __restrict__ K, double* __restrict__ kt64, float* __restrict__ kt32,
             double* __restrict__ kbar, long long ncells, int n, double h, int* flag,
             const __grid_constant__ DGTab<double> tab) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n2 = n * n, n3 = n2 * n, H = (n + 1) / 2, H2 = H * H, H3 = H2 * H;
  const int CB = coef_cells(n);
  double* sk = reinterpret_cast<double*>(smem_raw);  // K of the block's cells
  double* hw = sk + CB * n3;                         // h w_q per point
  double* term = hw + n3;                            // w log(product) per mirror group
  const long long c0 = (long long)blockIdx.x * CB;
  const int nblk = (int)((ncells - c0) < CB ? (ncells - c0) : CB);
  for (int q = threadIdx.x; q < n3; q += blockDim.x)
    hw[q] = h * (tab.w[q % n] * tab.w[(q / n) % n] * tab.w[q / n2]);
  __syncthreads();
  bool bad = false;
  for (int i = threadIdx.x; i < nblk * n3; i += blockDim.x) {
    const double Kq = K[c0 * n3 + i];
    if (!(Kq > 0.0) || !(Kq < INFINITY)) bad = true;
    sk[i] = Kq;
    const double v = hw[i % n3] * Kq;
    kt64[c0 * n3 + i] = v;
    if (kt32 != nullptr) kt32[c0 * n3 + i] = (float)v;
  }
  if (bad) atomicOr(flag, 1);
  __syncthreads();
  for (int i = threadIdx.x; i < nblk * H3; i += blockDim.x) {
    const int cell = i / H3, o = i - cell * H3;
    const int a = o % H, b = (o / H) % H, e = o / H2;
    double prod = 1.0;
    int ex = 0;
    for (int m = 0; m < 8; ++m) {
      const int a2 = m & 1 ? n - 1 - a : a, b2 = m & 2 ? n - 1 - b : b,
                e2 = m & 4 ? n - 1 - e : e;
      // a middle point is its own mirror image
      if (((m & 1) && a2 == a) || ((m & 2) && b2 == b) || ((m & 4) && e2 == e)) continue;
      double v = sk[cell * n3 + a2 + n * b2 + n2 * e2];
      if (v < 0x1p-1022) {
        v *= 0x1p64;
        ex -= 64;
      }
      const int hi = __double2hiint(v);
      ex += (hi >> 20) - 1023;
      prod *= __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(v));
    }
    const double lg = ex > -1000 && ex < 1000 ? log(scalbn(prod, ex))
                                              : fma((double)ex, 0.69314718055994530942, log(prod));
    term[i] = tab.w[a] * tab.w[b] * tab.w[e] * lg;
  }
  __syncthreads();
  for (int cell = threadIdx.x; cell < nblk; cell += blockDim.x) {
    double acc = 0.0;
    for (int o = 0; o < H3; ++o) acc += term[cell * H3 + o];
    kbar[c0 + cell] = exp(acc);
  }
}

// launch of k_coef_cells
cudaError_t dg_launch_coef_cells(const double* K, double* kt64, float* kt32, double* kbar,
                                 long long ncells, int n, double h, int* flag,
                                 const DGTab<double>& tab, cudaStream_t s) {
  const int n3 = n * n * n, H = (n + 1) / 2, CB = coef_cells(n);
  const size_t smem = sizeof(double) * ((size_t)CB * n3 + n3 + (size_t)CB * H * H * H);
  k_coef_cells<<<(unsigned)((ncells + CB - 1) / CB), 256, smem, s>>>(K, kt64, kt32, kbar, ncells,
                                                                     n, h, flag, tab);
  return cudaGetLastError();
}

// One thread per cell: h*gamma (FP64, and FP32 unless gh32 is NULL) and, unless
// dgam is NULL, d gamma / d log Kbar_c on its six faces.  A boundary face on a
// side whose bit is clear in dmask carries zero flux (homogeneous Neumann): no
// face term at all, i.e. gamma = 0 there.
__global__ void k_coef_faces(const double* __restrict__ kbar, double* __restrict__ gh64,
                             float* __restrict__ gh32, float2* __restrict__ gh32s,
                             double* __restrict__ dgam, int Nc, double h, int dmask) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nc = (long long)Nc * Nc * Nc;
  if (c >= nc) return;
  const int crd[3] = {(int)(c % Nc), (int)((c / Nc) % Nc), (int)(c / ((long long)Nc * Nc))};
  const long long stride[3] = {1, Nc, (long long)Nc * Nc};
  const double k = kbar[c];
  for (int f = 0; f < 6; ++f) {
    const int d = f >> 1;
    const bool upper = f & 1;
    const bool interior = upper ? (crd[d] < Nc - 1) : (crd[d] > 0);
    double g, dg;
    if (interior) {
      const double kn = kbar[upper ? c + stride[d] : c - stride[d]];
      g = 2.0 * k * kn / (k + kn);
      dg = g * kn / (k + kn);
    } else if ((dmask >> f) & 1) {
      g = k;
      dg = k;
    } else {
      g = 0.0;
      dg = 0.0;
    }
    gh64[c * 6 + f] = h * g;
    if (gh32 != nullptr) {
      const float hi = (float)(h * g);
      gh32[c * 6 + f] = hi;
      gh32s[c * 6 + f] = make_float2(hi, isfinite(hi) ? (float)(h * g - (double)hi) : 0.0f);
    }
    if (dgam != nullptr) dgam[c * 6 + f] = dg;
  }
}

// ---------------------------------------------------------------------------
// mesh lifetime
// ---------------------------------------------------------------------------
template <typename P>
static cudaError_t dmalloc(P** p, size_t count) {
  return cudaMalloc((void**)p, count * sizeof(P));
}

static void free_all(dg_mesh* m) {
  void* ptrs[] = {m->kt64, m->kt32, m->gh64, m->gh32, m->gh32s, m->dgam, m->kbar, m->dflag, m->lineopX, m->gamX, m->expM, m->expG, m->expU, m->expN, m->markU, m->expUb, m->diag64, m->dinv64, m->dinv32, m->binv64, m->kron64, m->kron32, m->kronX, m->kronNX, m->kronW, m->dinvN64, m->dinvN32, m->bN64, m->xN64, m->hk32, m->kronN64, m->kronN32, m->geo_vol, m->geo_det, m->geo_face, m->geo_pen, m->mlV, m->mlF, m->mlExpV, m->mlExpM, m->mlExpF,
                  m->U64,  m->X64,  m->TR64, m->TR32, m->U64b,
                  m->TR64b, m->hx_dev, m->hy_dev, m->r64, m->p64, m->q64,
                  m->t64,  m->s64, m->d32,  m->r32, m->p32, m->q32, m->partials, m->state,
                  m->partials_cells};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (m->state_host) cudaFreeHost(m->state_host);
  if (m->tev) {
    for (int i = 0; i < 3 * m->tev_cap; ++i) cudaEventDestroy(m->tev[i]);
    free(m->tev);
  }
  if (m->solve_stream) cudaStreamDestroy(m->solve_stream);
  if (m->ev) cudaEventDestroy(m->ev);
  for (cudaStream_t hs : m->hstream)
    if (hs) cudaStreamDestroy(hs);
  for (cudaEvent_t he : m->hev)
    if (he) cudaEventDestroy(he);
}

extern "C" int dg_create_mesh(int n_cells, int degree, dg_mesh** out) {
  if (out == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "dg_create_mesh: out is NULL");
  *out = nullptr;
  if (n_cells < 1 || n_cells > 1024)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_create_mesh: n_cells=%d outside [1, 1024]", n_cells);
  if (degree < 1 || degree > DG_MAXN - 1)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_create_mesh: degree=%d outside [1, %d]", degree,
                   DG_MAXN - 1);
  dg_mesh* m = (dg_mesh*)calloc(1, sizeof(dg_mesh));
  if (!m) return dg_fail(DG_ERR_OOM, "dg_create_mesh: host allocation failed");
  m->N = n_cells;
  m->k = degree;
  m->n = degree + 1;
  m->ncells = (long long)n_cells * n_cells * n_cells;
  const long long n3 = (long long)m->n * m->n * m->n;
  const long long n2 = (long long)m->n * m->n;
  m->ndofs = m->ncells * n3;
  m->h = 1.0 / n_cells;
  m->sigma = 2.0 * (degree + 1) * (degree + 1);
  m->dirichlet_mask = DG_BC_DIRICHLET;
  m->affine = false;
  m->geomDet = 1.0;
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 3; ++j) m->geomG[i][j] = i == j ? 1.0 : 0.0;
    m->geomKappa[i] = 1.0;
  }
  dg_build_tables(m->n, m->sigma, &m->tab64, &m->tab32);
  dg_build_nodal_tables(m->tab64, m->n, &m->tabN64, &m->tabN32);
  if (!dg_build_fixed_tables(m->n, m->h, &m->tabX, &m->tabXS, &m->tabXG)) {
    free(m);
    return dg_fail(DG_ERR_INVALID_ARG, "dg_create_mesh: fixed-point tables out of range");
  }
  cudaError_t e = cudaGetDevice(&m->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, m->device);
  const size_t nd = (size_t)m->ndofs, nc = (size_t)m->ncells, ntr = (size_t)(12 * n2) * nc;
  if (e == cudaSuccess) e = dmalloc(&m->kt64, nd);
  if (e == cudaSuccess) e = dmalloc(&m->kt32, nd);
  if (e == cudaSuccess) e = dmalloc(&m->gh64, 6 * nc);
  if (e == cudaSuccess) e = dmalloc(&m->gh32, 6 * nc);
  if (e == cudaSuccess) e = dmalloc(&m->gh32s, 6 * nc);
  if (e == cudaSuccess) e = dmalloc(&m->dgam, 6 * nc);
  if (e == cudaSuccess)
    e = dmalloc(&m->lineopX, (size_t)3 * n2 * (size_t)(m->n * (m->n + 1) / 2) * nc);
  if (e == cudaSuccess) e = dmalloc(&m->gamX, 6 * nc);
  if (e == cudaSuccess) e = dmalloc(&m->expM, nc);
  if (e == cudaSuccess) e = dmalloc(&m->expG, 6 * nc);
  if (e == cudaSuccess) e = dmalloc(&m->expU, nc);
  if (e == cudaSuccess) e = dmalloc(&m->expN, nc);
  if (e == cudaSuccess) e = dmalloc(&m->markU, nc);
  if (e == cudaSuccess) e = dmalloc(&m->kbar, nc);
  if (e == cudaSuccess) e = dmalloc(&m->dflag, 1);
  if (e == cudaSuccess) e = dmalloc(&m->U64, nd);
  if (e == cudaSuccess) e = dmalloc(&m->TR64, ntr);
  if (e == cudaSuccess) e = dmalloc(&m->TR32, ntr);
  if (e != cudaSuccess) {
    int rc = dg_cuda_fail(e, "dg_create_mesh: device allocation");
    free_all(m);
    free(m);
    return rc;
  }
  int rc = dg_prepare_fixed(m->n);
  if (rc == DG_OK) rc = dg_prepare_apply_f64(m->n);
  if (rc == DG_OK) rc = dg_prepare_apply_f32(m->n);
  if (rc == DG_OK) rc = dg_prepare_affine(m->n);
  if (rc == DG_OK) rc = dg_prepare_grad(m->n);
  if (rc != DG_OK) {
    free_all(m);
    free(m);
    return rc;
  }
  *out = m;
  return DG_OK;
}

extern "C" int dg_destroy_mesh(dg_mesh* m) {
  if (m == nullptr) return DG_OK;
  cudaError_t e = cudaDeviceSynchronize();
  free_all(m);
  free(m);
  if (e != cudaSuccess) return dg_cuda_fail(e, "dg_destroy_mesh: device synchronize");
  return DG_OK;
}

extern "C" int dg_mesh_info(const dg_mesh* m, long long* n_dofs, long long* n_cells_total,
                            int* n_points_1d, double* sigma) {
  if (m == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "dg_mesh_info: mesh is NULL");
  if (n_dofs) *n_dofs = m->ndofs;
  if (n_cells_total) *n_cells_total = m->ncells;
  if (n_points_1d) *n_points_1d = m->n;
  if (sigma) *sigma = m->sigma;
  return DG_OK;
}

extern "C" int dg_set_boundary(dg_mesh* m, int dirichlet_mask) {
  if (m == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "dg_set_boundary: mesh is NULL");
  if (dirichlet_mask < 0 || dirichlet_mask > 0x3F)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_set_boundary: mask 0x%x outside 0..0x3f",
                   dirichlet_mask);
  if (dirichlet_mask == 0)
    return dg_fail(DG_ERR_INVALID_ARG,
                   "dg_set_boundary: at least one side must be Dirichlet (the operator would "
                   "be singular)");
  m->dirichlet_mask = dirichlet_mask;
  m->has_coef = false;  // the face weights depend on it: set the coefficient again
  m->has_diag = false;
  m->has_block = false;
  m->has_kron = false;
  m->has_kron_x = m->has_kron_nx = false;
  m->has_nodal_diag = false;
  m->has_nodal32 = false;
  m->has_kron_nodal = false;
  return DG_OK;
}

int dg_require_cube(const dg_mesh* m, const char* who) {
  if (m != nullptr && (m->affine || m->multilinear))
    return dg_fail(DG_ERR_INVALID_ARG,
                   "%s: not available on an affine or multilinear geometry (FP64 dg_apply, "
                   "dg_apply_adjoint, dg_load_vector and the FP64 CG without preconditioner "
                   "are)", who);
  return DG_OK;
}

int dg_ensure_grad_ws(dg_mesh* m) {
  if (m->U64b) return DG_OK;
  const size_t nd = (size_t)m->ndofs;
  const size_t ntr = (size_t)(12 * m->n * m->n) * (size_t)m->ncells;
  DG_CUDA(dmalloc(&m->TR64b, ntr));
  DG_CUDA(dmalloc(&m->expUb, (size_t)m->ncells));
  DG_CUDA(dmalloc(&m->U64b, nd));
  return DG_OK;
}

int dg_ensure_solver_ws(dg_mesh* m) {
  if (m->state) return DG_OK;
  const size_t nd = (size_t)m->ndofs;
  DG_CUDA(dmalloc(&m->r64, nd));
  DG_CUDA(dmalloc(&m->p64, nd));
  DG_CUDA(dmalloc(&m->q64, nd));
  DG_CUDA(dmalloc(&m->t64, nd));
  DG_CUDA(dmalloc(&m->s64, nd));
  DG_CUDA(dmalloc(&m->d32, nd));
  DG_CUDA(dmalloc(&m->r32, nd));
  DG_CUDA(dmalloc(&m->p32, nd));
  DG_CUDA(dmalloc(&m->q32, nd));
  DG_CUDA(dmalloc(&m->partials, DG_RED_SUMS * DG_RED_BLOCKS));
  DG_CUDA(dmalloc(&m->partials_cells, (size_t)dg_mixed32_blocks(m->n, m->ncells)));
  DG_CUDA(cudaMallocHost((void**)&m->state_host, sizeof(DGCGState)));
  DG_CUDA(cudaStreamCreateWithFlags(&m->solve_stream, cudaStreamNonBlocking));
  DG_CUDA(cudaEventCreateWithFlags(&m->ev, cudaEventDisableTiming));
  DG_CUDA(dmalloc(&m->state, 1));
  DG_CUDA(cudaMemset(m->state, 0, sizeof(DGCGState)));
  return dg_prepare_mixed32(m);
}

// ---------------------------------------------------------------------------
// coefficient
// ---------------------------------------------------------------------------
extern "C" int dg_set_coefficient(dg_mesh* m, const double* K, void* stream) {
  if (m == nullptr || K == nullptr)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_set_coefficient: NULL mesh or K");
  cudaStream_t s = (cudaStream_t)stream;
  m->has_coef = false;
  m->has_diag = false;
  m->has_block = false;
  m->has_kron = false;
  m->has_kron_x = m->has_kron_nx = false;
  m->has_nodal_diag = false;
  m->has_nodal32 = false;
  m->has_kron_nodal = false;
  DG_CUDA(cudaMemsetAsync(m->dflag, 0, sizeof(int), s));
  DG_CUDA(dg_launch_coef_cells(K, m->kt64, m->kt32, m->kbar, m->ncells, m->n, m->h, m->dflag,
                               m->tab64, s));
  {
    const unsigned blocks = (unsigned)((m->ncells + 255) / 256);
    k_coef_faces<<<blocks, 256, 0, s>>>(m->kbar, m->gh64, m->gh32, m->gh32s, m->dgam, m->N, m->h,
                                        m->dirichlet_mask);
    DG_CUDA(cudaGetLastError());
    if (!m->affine)
      if (int rc = m->multilinear ? dg_setup_multilinear(m, s) : dg_setup_fixed(m, K, s)) return rc;
  }
  int flag = 0;
  DG_CUDA(cudaMemcpyAsync(&flag, m->dflag, sizeof(int), cudaMemcpyDeviceToHost, s));
  DG_CUDA(cudaStreamSynchronize(s));
  if (flag)
    return dg_fail(DG_ERR_INVALID_ARG,
                   "dg_set_coefficient: K has a value <= 0 or non-finite; coefficient not set");
  m->has_coef = true;
  return DG_OK;
}

// ---------------------------------------------------------------------------
// operator application
// ---------------------------------------------------------------------------
static int check_apply_args(const dg_mesh* m, const void* x, const void* y, int prec,
                            const char* who) {
  if (m == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "%s: mesh is NULL", who);
  if (!m->has_coef) return dg_fail(DG_ERR_INVALID_ARG, "%s: coefficient not set", who);
  if (x == nullptr || y == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "%s: NULL vector", who);
  if (x == y) return dg_fail(DG_ERR_INVALID_ARG, "%s: input and output alias", who);
  if (prec != DG_FP64 && prec != DG_FP32)
    return dg_fail(DG_ERR_INVALID_ARG, "%s: prec=%d is neither DG_FP64 nor DG_FP32", who, prec);
  return DG_OK;
}

extern "C" int dg_apply(const dg_mesh* m, const void* x, void* y, int prec, void* stream) {
  int rc = check_apply_args(m, x, y, prec, "dg_apply");
  if (rc) return rc;
  if (prec == DG_FP32 && (rc = dg_require_cube(m, "dg_apply(FP32)"))) return rc;
  if (prec == DG_FP64)
    return dg_launch_apply_f64(m, (const double*)x, (double*)y, nullptr, (cudaStream_t)stream);
  return dg_launch_apply_f32(m, (const float*)x, (float*)y, nullptr, (cudaStream_t)stream);
}

extern "C" int dg_apply_adjoint(const dg_mesh* m, const void* ybar, void* xbar, int prec,
                                void* stream) {
  int rc = check_apply_args(m, ybar, xbar, prec, "dg_apply_adjoint");
  if (rc) return rc;
  if (prec == DG_FP32 && (rc = dg_require_cube(m, "dg_apply_adjoint(FP32)"))) return rc;
  // a(u, v) = a(v, u): the transposed data flow performs the same contractions.
  if (prec == DG_FP64)
    return dg_launch_apply_f64(m, (const double*)ybar, (double*)xbar, nullptr,
                               (cudaStream_t)stream);
  return dg_launch_apply_f32(m, (const float*)ybar, (float*)xbar, nullptr, (cudaStream_t)stream);
}

// Host-buffer apply, pipelined over z-slabs of cells so that both copies
// overlap the kernels.  Four streams:
//   copy-in   H2D of x, slab by slab;
//   pass 1    pass 1 of slab s once its x has arrived (runs ahead of pass 2);
//   caller's  pass 2 of slab s once pass 1 has covered slab s+1 (the upper
//             neighbours of slab s are the first layer of slab s+1);
//   copy-out  D2H of y of slab s once pass 2 has written it.
// Pass 1 and pass 2 of different slabs may run at the same time, which fills
// the last partial wave of each launch.  Every event is recorded before any
// wait on it is enqueued.
static int ensure_host_pipeline(dg_mesh* m) {
  if (m->hx_dev == nullptr) {
    DG_CUDA(cudaMalloc(&m->hx_dev, (size_t)m->ndofs * sizeof(double)));
    DG_CUDA(cudaMalloc(&m->hy_dev, (size_t)m->ndofs * sizeof(double)));
  }
  for (cudaStream_t& hs : m->hstream)
    if (hs == nullptr) DG_CUDA(cudaStreamCreateWithFlags(&hs, cudaStreamNonBlocking));
  for (cudaEvent_t& he : m->hev)
    if (he == nullptr) DG_CUDA(cudaEventCreateWithFlags(&he, cudaEventDisableTiming));
  return DG_OK;
}

extern "C" int dg_apply_host(const dg_mesh* mc, const void* x_host, void* y_host, int prec,
                             void* stream) {
  int rc = check_apply_args(mc, x_host, y_host, prec, "dg_apply_host");
  if (rc) return rc;
  if ((rc = dg_require_cube(mc, "dg_apply_host"))) return rc;
  dg_mesh* m = const_cast<dg_mesh*>(mc);
  cudaStream_t s = (cudaStream_t)stream;
  rc = ensure_host_pipeline(m);
  if (rc) return rc;
  const size_t esz = prec == DG_FP64 ? sizeof(double) : sizeof(float);
  const long long layer = (long long)m->N * m->N;  // cells per z-layer
  // A slab costs about 10 us of launches and events, hidden only while the copies
  // take longer: one slab per 3 MB of a vector.  Measured (us; 1 / this rule /
  // always 16): 10^3 Q4 49 / 51 / 134, 18^3 Q3 71 / 72 / 120, 26^3 Q3
  // 153 / 146 / 202, 40^3 Q3 477 / 329 / 340; 64^3 Q3 one slab 1796, 16 1070,
  // 32 1138.
  const long long by_size = (long long)(m->ndofs * (long long)esz) / (3ll << 20);
  int nslab_max = by_size < 1 ? 1 : by_size > DG_HOST_SLABS ? DG_HOST_SLABS : (int)by_size;
  if (nslab_max > m->N) nslab_max = m->N;
  const int lps = (m->N + nslab_max - 1) / nslab_max;  // layers per slab
  const int nslab = (m->N + lps - 1) / lps;
  const long long n3 = (long long)m->n * m->n * m->n;
  auto cells = [&](int sl) { return (long long)(sl * lps < m->N ? sl * lps : m->N) * layer; };
  cudaStream_t cin = m->hstream[0], cout = m->hstream[1], p1 = m->hstream[2];
  cudaEvent_t* ev_in = m->hev;                       // H2D of slab s done
  cudaEvent_t* ev_p1 = m->hev + DG_HOST_SLABS;       // pass 1 of slab s done
  cudaEvent_t* ev_out = m->hev + 2 * DG_HOST_SLABS;  // pass 2 of slab s done
  cudaEvent_t ev_start = m->hev[3 * DG_HOST_SLABS];
  // order after the caller's earlier work on its stream
  DG_CUDA(cudaEventRecord(ev_start, s));
  DG_CUDA(cudaStreamWaitEvent(cin, ev_start, 0));
  DG_CUDA(cudaStreamWaitEvent(p1, ev_start, 0));
  DG_CUDA(cudaStreamWaitEvent(cout, ev_start, 0));
  char* xd = (char*)m->hx_dev;
  char* yd = (char*)m->hy_dev;
  auto span = [&](int sl, size_t* off, size_t* bytes) {
    *off = (size_t)(cells(sl) * n3) * esz;
    *bytes = (size_t)((cells(sl + 1) - cells(sl)) * n3) * esz;
  };
  auto pass = [&](int p, int sl, cudaStream_t st) {
    return prec == DG_FP64
               ? dg_launch_fixed_pass(m, true, p, (const double*)xd, (double*)yd, cells(sl),
                                      cells(sl + 1), nullptr, st)
               : dg_launch_pass_f32(m, p, (const float*)xd, (float*)yd, cells(sl),
                                    cells(sl + 1), nullptr, st);
  };
  for (int sl = 0; sl < nslab; ++sl) {
    size_t off, bytes;
    span(sl, &off, &bytes);
    DG_CUDA(cudaMemcpyAsync(xd + off, (const char*)x_host + off, bytes, cudaMemcpyHostToDevice,
                            cin));
    DG_CUDA(cudaEventRecord(ev_in[sl], cin));
  }
  for (int sl = 0; sl < nslab; ++sl) {
    DG_CUDA(cudaStreamWaitEvent(p1, ev_in[sl], 0));
    rc = pass(1, sl, p1);
    if (rc) return rc;
    DG_CUDA(cudaEventRecord(ev_p1[sl], p1));
  }
  for (int sl = 0; sl < nslab; ++sl) {
    // pass 1 of slabs sl - 1, sl, sl + 1 (in stream order on p1)
    DG_CUDA(cudaStreamWaitEvent(s, ev_p1[sl + 1 < nslab ? sl + 1 : sl], 0));
    rc = pass(2, sl, s);
    if (rc) return rc;
    DG_CUDA(cudaEventRecord(ev_out[sl], s));
  }
  for (int sl = 0; sl < nslab; ++sl) {
    size_t off, bytes;
    span(sl, &off, &bytes);
    DG_CUDA(cudaStreamWaitEvent(cout, ev_out[sl], 0));
    DG_CUDA(cudaMemcpyAsync((char*)y_host + off, yd + off, bytes, cudaMemcpyDeviceToHost, cout));
  }
  DG_CUDA(cudaStreamSynchronize(cout));
  DG_CUDA(cudaStreamSynchronize(s));
  return DG_OK;
}

// ---------------------------------------------------------------------------
// coefficient gradient
// ---------------------------------------------------------------------------
extern "C" int dg_coeff_grad(const dg_mesh* mc, const double* u, const double* v, double* g,
                             void* stream) {
  if (mc == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "dg_coeff_grad: mesh is NULL");
  if (!mc->has_coef) return dg_fail(DG_ERR_INVALID_ARG, "dg_coeff_grad: coefficient not set");
  if (u == nullptr || v == nullptr || g == nullptr)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_coeff_grad: NULL vector");
  if (g == u || g == v) return dg_fail(DG_ERR_INVALID_ARG, "dg_coeff_grad: g aliases u or v");
  if (int rc0 = dg_require_cube(mc, "dg_coeff_grad")) return rc0;
  dg_mesh* m = const_cast<dg_mesh*>(mc);
  int rc = dg_ensure_grad_ws(m);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  rc = dg_launch_fixed_trace(m, u, m->U64, m->TR64, m->expU, s);
  if (rc) return rc;
  rc = dg_launch_fixed_trace(m, v, m->U64b, m->TR64b, m->expUb, s);
  if (rc) return rc;
  return dg_launch_coeff_grad(m, g, s);
}

// ---------------------------------------------------------------------------
// per-pass kernel timing
// ---------------------------------------------------------------------------
void dg_timing_mark(const dg_mesh* mc, int slot, cudaStream_t s) {
  dg_mesh* m = const_cast<dg_mesh*>(mc);
  if (!m->timing || m->tev_used >= m->tev_cap) return;
  cudaEventRecord(m->tev[3 * m->tev_used + slot], s);
  if (slot == 2) m->tev_used += 1;
}

extern "C" int dg_timing_enable(dg_mesh* m, int max_applies) {
  if (m == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "dg_timing_enable: mesh is NULL");
  if (max_applies < 1 || max_applies > 65536)
    return dg_fail(DG_ERR_INVALID_ARG, "dg_timing_enable: max_applies=%d outside [1, 65536]",
                   max_applies);
  if (m->tev_cap < max_applies) {
    if (m->tev) {
      for (int i = 0; i < 3 * m->tev_cap; ++i) cudaEventDestroy(m->tev[i]);
      free(m->tev);
      m->tev = nullptr;
      m->tev_cap = 0;
    }
    m->tev = (cudaEvent_t*)calloc((size_t)3 * max_applies, sizeof(cudaEvent_t));
    if (!m->tev) return dg_fail(DG_ERR_OOM, "dg_timing_enable: host allocation failed");
    for (int i = 0; i < 3 * max_applies; ++i) DG_CUDA(cudaEventCreate(&m->tev[i]));
    m->tev_cap = max_applies;
  }
  m->tev_used = 0;
  m->timing = true;
  return DG_OK;
}

extern "C" int dg_timing_read(dg_mesh* m, int* n_applies, double* ms1, double* ms2) {
  if (m == nullptr) return dg_fail(DG_ERR_INVALID_ARG, "dg_timing_read: mesh is NULL");
  m->timing = false;
  double a = 0.0, b = 0.0;
  for (int i = 0; i < m->tev_used; ++i) {
    DG_CUDA(cudaEventSynchronize(m->tev[3 * i + 2]));
    float t1 = 0.f, t2 = 0.f;
    DG_CUDA(cudaEventElapsedTime(&t1, m->tev[3 * i], m->tev[3 * i + 1]));
    DG_CUDA(cudaEventElapsedTime(&t2, m->tev[3 * i + 1], m->tev[3 * i + 2]));
    a += t1;
    b += t2;
  }
  if (n_applies) *n_applies = m->tev_used;
  if (ms1) *ms1 = a;
  if (ms2) *ms2 = b;
  return DG_OK;
}
