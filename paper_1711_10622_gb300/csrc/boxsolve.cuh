// The solver's products by row boxes (solver_box.cu): launchers with the arguments of the row-by-row kernels of
// solver_impl.cuh. Blocks of width m with m = 4 or a multiple of 8 (float32: up to 16), 32-byte aligned.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "rowprod.cuh"

namespace ens {
namespace solver {

template <typename T>
struct Cols;

// Whether a block of width m (stride m) has box kernels in the solver.
template <typename T>
inline bool box_width(int m) {
  return m == 4 || m == 8 || (sizeof(T) == 8 ? m % 8 == 0 : m == 16);
}

// v = A ph, (rhat, v) and the step alpha
cudaError_t launch_box_v(const BoxPlan &B, const MatView &A, int32_t m, const double *ph, double *v, const double *rh, const Cols<double> &cs,
                         double *partials, unsigned *counter, int sms, cudaStream_t st);
cudaError_t launch_box_v(const BoxPlan &B, const MatView &A, int32_t m, const float *ph, float *v, const float *rh, const Cols<float> &cs,
                         float *partials, unsigned *counter, int sms, cudaStream_t st);
// t = A sh, (t, s), (t, t) and omega
cudaError_t launch_box_t(const BoxPlan &B, const MatView &A, int32_t m, const double *sh, double *t, const double *s, const Cols<double> &cs,
                         double *partials, unsigned *counter, int sms, cudaStream_t st);
cudaError_t launch_box_t(const BoxPlan &B, const MatView &A, int32_t m, const float *sh, float *t, const float *s, const Cols<float> &cs,
                         float *partials, unsigned *counter, int sms, cudaStream_t st);
// b - A x: its norms (and r, the outer residual of the mixed solver)
cudaError_t launch_box_resid(const BoxPlan &B, const MatView &A, int32_t m, const double *b, const double *x, double *r, int outer,
                             const Cols<double> &cs, double *partials, unsigned *counter, int sms, cudaStream_t st);
// z1 = (1 + c1) z - c1 zp + c2 D^-1 (src - A z) (zp = nullptr: 0); z1 may be zp
cudaError_t launch_box_cheb(const BoxPlan &B, const MatView &A, int32_t m, const double *z, const double *zp, const double *src, double *z1,
                            double c1, double c2, int sms, cudaStream_t st);
cudaError_t launch_box_cheb(const BoxPlan &B, const MatView &A, int32_t m, const float *z, const float *zp, const float *src, float *z1, float c1,
                            float c2, int sms, cudaStream_t st);
// res = r - A z
cudaError_t launch_box_amg_resid(const BoxPlan &B, const MatView &A, int32_t m, const double *z, const double *r, double *res, int sms,
                                 cudaStream_t st);
cudaError_t launch_box_amg_resid(const BoxPlan &B, const MatView &A, int32_t m, const float *z, const float *r, float *res, int sms,
                                 cudaStream_t st);
// both updates of a two-update smoothing from As = A D^-1 (boxes of As; dinv of A)
cudaError_t launch_box_smooth2(const BoxPlan &Bs, const MatView &As, const double *dinv, int32_t m, bool add, const double *src, double *z,
                               double inv_theta, double c1, double c2, int sms, cudaStream_t st);
cudaError_t launch_box_smooth2(const BoxPlan &Bs, const MatView &As, const float *dinv, int32_t m, bool add, const float *src, float *z,
                               float inv_theta, float c1, float c2, int sms, cudaStream_t st);

}  // namespace solver
}  // namespace ens
