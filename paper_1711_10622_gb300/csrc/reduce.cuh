// Per-column block reductions with a deterministic cross-block pass.
//
// A kernel whose threads own (row, column-chunk) pairs accumulates ND per-column sums in
// registers; reduce_cols() combines them inside the block (warp shuffles in a fixed butterfly,
// then a fixed-order sum over warps), writes one partial per block and column, and the last
// block to finish (ticket from an atomic counter) sums the partials in block order and runs a
// per-column finalisation (the scalar step of the solver). No value is ever accumulated with an
// atomic, so results do not depend on block scheduling and are bitwise reproducible.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "ens_internal.cuh"

namespace ens {

constexpr int kMaxSolveM = 64;  // columns handled by the solver kernels (one chunk per lane)

template <typename T, int ND>
struct ColTotals {
  T v[ND][kMaxSolveM];
};

// acc[d][q]: this thread's sum for dot d and column lane*VEC + q (zero for idle lanes).
// partials: gridDim.x * ND * m scratch values; counter: zero before the launch, reset to zero by
// the last block. fin(l, totals) runs on threads l < m of the last block.
struct NoAfter {
  __device__ void operator()(bool) const {}
};

// The warp's sums of every value and column, to wsum[warp] (no barrier).
template <typename T, int ND, int VEC, int LANES>
__device__ __forceinline__ void warp_cols(const T (&acc)[ND][VEC], T (&wsum)[kThreads / 32][ND][LANES * VEC]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // Sums over the warp's row groups. While a lane holds several values it gives half of them to its partner and
  // adds the partner's share of the others, so ND * VEC values cost about that many additions instead of that many
  // per step: the FP64 pipe takes 16 clocks for a warp's addition, and whole butterflies of every value
  // were a third of the reductions' time (32^3 rows, m = 4).
  constexpr int kVals = ND * VEC, kPow = kVals <= 1 ? 1 : kVals <= 2 ? 2 : kVals <= 4 ? 4 : kVals <= 8 ? 8 : 16;
  static_assert(kVals <= 16, "at most 16 sums per thread");
  T v[kPow];
#pragma unroll
  for (int k = 0; k < kPow; ++k) v[k] = k < kVals ? acc[k / VEC][k % VEC] : T(0);
  int base = 0;
  {
    int cnt = kPow;  // folded: every step is unrolled
#pragma unroll
    for (int off = LANES; off < 32; off <<= 1) {
      if (cnt > 1) {
        const int half = cnt / 2;
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < kPow / 2; ++i)
          if (i < half) {
            const T send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        base += up ? half : 0;
        cnt = half;
      } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
      }
    }
#pragma unroll
    for (int i = 0; i < kPow; ++i)
      if (i < cnt) {
        const int k = base + i;
        if (k < kVals) wsum[warp][k / VEC][(lane % LANES) * VEC + k % VEC] = v[i];
      }
  }
}

// after(any): runs once, on thread 0 of the last block, when every column's fin() has finished; any: some fin()
// returned true (fin may return bool).
template <typename T, int ND, int VEC, int LANES, typename Fin, typename After = NoAfter>
__device__ __forceinline__ void reduce_cols(T (&acc)[ND][VEC], int32_t m, T *__restrict__ partials,
                                            unsigned *__restrict__ counter, Fin &&fin, After &&after = After()) {
  constexpr int kWarps = kThreads / 32;
  __shared__ T wsum[kWarps][ND][LANES * VEC];
  __shared__ ColTotals<T, ND> tot;
  __shared__ bool is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  warp_cols<T, ND, VEC, LANES>(acc, wsum);
  __syncthreads();
  for (int t = threadIdx.x; t < ND * m; t += kThreads) {  // block sums, warp by warp in a fixed order
    const int d = t / m, c = t - d * m;
    T b = wsum[0][d][c];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) b += wsum[w][d][c];
    partials[(size_t)blockIdx.x * ND * m + t] = b;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  for (int t = warp; t < ND * m; t += kWarps) {
    T s = T(0);
    for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(partials + (size_t)b * ND * m + t);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) tot.v[t / m][t % m] = s;
  }
  __syncthreads();
  bool go = false;
  if ((int)threadIdx.x < m) {
    if constexpr (std::is_same<decltype(fin(0, tot)), bool>::value)
      go = fin((int)threadIdx.x, tot);
    else
      fin((int)threadIdx.x, tot);
  }
  const int any = __syncthreads_or(go);
  if (threadIdx.x == 0) {
    after(any != 0);
    *counter = 0u;
  }
}

}  // namespace ens
