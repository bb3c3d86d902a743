// The whole iteration loop of a small plain float64 solve in one launch (solver_small.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "rowprod.cuh"

namespace ens {
namespace solver {

template <typename T>
struct Cols;

struct SmallSolve {
  MatView A;
  int32_t m, max_iter, tgrid, grid, sgrid;  // blocks of the product, x / r and s kernels of the loop it replaces
  uint32_t mask;
  double *x, *r, *p, *v, *s, *t;
  const double *rh;
  double *partials;  // two buffers of max(tgrid, grid, sgrid) * 2 m
  unsigned *bar;     // [0]: arrivals, [1]: a wait ran out of its limit; both zero at the launch
};

// Blocks of the launch, 0 where the form does not apply: widths of 2, 4, 6 and 8 columns, one row tile per block,
// every block resident at once and few enough for each to read all partial sums.
int small_solve_blocks(const SmallSolve &a, int64_t tiles, int num_sms);
cudaError_t launch_small_solve(const SmallSolve &a, const Cols<double> &cs, int blocks, cudaStream_t st);

}  // namespace solver
}  // namespace ens
