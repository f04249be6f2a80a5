// FP64 operator application by geometry and basis.
#include "dg_apply_impl.cuh"

int dg_launch_apply_f64(const dg_mesh* m, const double* x, double* y, const int* skip,
                        cudaStream_t s) {
  // inside a solve in the scaled Gauss-point basis (DG_CG_NODAL): Q A Q^T
  if (m->nodal_op) return dg_launch_fixed_apply(m, false, x, y, skip, s);
  if (m->multilinear) return dg_launch_apply_multilinear(m, x, y, skip, s);
  if (m->affine) return dg_launch_apply_affine(m, x, y, skip, s);
  return dg_launch_fixed_apply(m, true, x, y, skip, s);
}

int dg_prepare_apply_f64(int n) {
  cudaError_t e = dgk::dispatch_n<double, dgk::PrepareF>(n);
  if (e != cudaSuccess) return dg_cuda_fail(e, "apply (fp64) kernel attributes");
  return DG_OK;
}
