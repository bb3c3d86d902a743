// Launchers for the small levels of the AMG V-cycle (amg_small.cu): levels with too few rows for one
// thread group per row to fill the GPU.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "rowprod.cuh"

namespace ens {
namespace solver {

constexpr int kMaxCoarseSteps = 64;
constexpr int kMaxTailLevels = 8;
// Levels that the one-cluster launch takes. The coarsest level always has at most kTailCoarseRows rows
// there; the levels above it at most kTailRows (float32) or kTailRowsF64: the cluster's eight SMs have 1/19
// of the GPU's FP64 rate, so float64 levels leave it earlier.
constexpr int64_t kTailCoarseRows = 4096;
// The coarsest level's updates as a dense matrix, up to this many rows (1 MB in float32, formed once at set-up).
constexpr int64_t kDenseRows = 512;
constexpr int64_t kTailRows = 4096;
constexpr int64_t kTailRowsF64 = 1024;

template <typename T>
struct TailLevel {
  const int32_t *rp, *ci;    // the level's matrix
  const T *va;
  const int32_t *srp, *sci;  // its column-scaled copy A D^-1 (smoothed levels)
  const T *sva;
  const T *dinv;
  const int32_t *agg, *ptr, *mem;
  T *r, *z, *res;
  int32_t n, nc;
};

template <typename T>
struct TailArgs {
  int32_t nl, m, lanes, steps;  // levels, block width, threads across a row's columns, coarsest updates
  T inv_theta, c1, c2;          // two-update smoothing
  const T *dense;               // matrix of the coarsest level's updates, n x n (nullptr: none)
  T *da, *db, *res;             // coarsest level's blocks (when its vectors do not fit shared memory)
  T k1[kMaxCoarseSteps], k2[kMaxCoarseSteps];
  TailLevel<T> lev[kMaxTailLevels];
};

// The dense matrix of `steps` updates on A (A.n <= kDenseRows): M and its float32 copy; k1, k2 [steps] on the device.
cudaError_t coarse_matrix(const MatView &A, int32_t steps, double inv_theta, const double *k1, const double *k2, double *M, float *M32,
                          cudaStream_t st);
// z of level 0 of `a` (its first level) from that level's r: the V-cycle from there down, in one cluster.
cudaError_t launch_amg_tail(const TailArgs<float> &a, int vec, cudaStream_t st);
cudaError_t launch_amg_tail(const TailArgs<double> &a, int vec, cudaStream_t st);

// res = r - A z, and both updates of a two-update smoothing from As = A D^-1 (add: z += ...), with the
// nonzeros of a row shared by several threads (native FMA).
template <typename T>
struct SmallLevel {
  const int32_t *rp, *ci;
  const T *va;
  const T *dinv;  // of A (smoothing)
  int32_t n, m, lanes;
};
cudaError_t launch_small_resid(const SmallLevel<float> &A, int vec, const float *z, const float *r, float *res, cudaStream_t st);
cudaError_t launch_small_resid(const SmallLevel<double> &A, int vec, const double *z, const double *r, double *res, cudaStream_t st);
cudaError_t launch_small_smooth2(const SmallLevel<float> &As, int vec, bool add, const float *src, float *z, float inv_theta, float c1,
                                 float c2, cudaStream_t st);
cudaError_t launch_small_smooth2(const SmallLevel<double> &As, int vec, bool add, const double *src, double *z, double inv_theta,
                                 double c1, double c2, cudaStream_t st);

// rc_I = sum of res over the rows of aggregate I (members mem[ptr[I]..ptr[I+1])).
cudaError_t launch_small_restrict(const int32_t *ptr, const int32_t *mem, int32_t nc, int32_t m, int32_t lanes, int vec, const float *res,
                                  float *rc, cudaStream_t st);
cudaError_t launch_small_restrict(const int32_t *ptr, const int32_t *mem, int32_t nc, int32_t m, int32_t lanes, int vec, const double *res,
                                  double *rc, cudaStream_t st);

}  // namespace solver
}  // namespace ens
