// The small levels of the AMG V-cycle. A level of a few thousand rows with one thread group per row and
// 256 rows per block ran on 3 to 54 blocks, each group walking rows of up to a hundred nonzeros one gather
// after the other: 25-30 us per launch, and 80-128 us for the coarsest level's updates in one block (float32,
// m = 8), more than the fine level's products. Two forms replace it:
//   * k_small_*: the nonzeros of a row are dealt to S threads (S as large as the row count leaves threads
//     for), whose sums are added by shuffles; each thread has four gathers in flight.
//   * k_amg_tail: every level below a few thousand rows, down and up again, in one launch of one
//     thread-block cluster. The stages are separated by the cluster's hardware barrier instead of kernel
//     boundaries; blocks exchange vectors through L2. The coarsest level's updates, one fixed linear operator,
//     are applied as its dense matrix, formed at set-up (levels of at most kDenseRows rows; otherwise update by
//     update in one block, on vectors in shared memory where they fit: 43 of a launch's 80-135 us).
// The bound is latency throughout (a stage is one or two dependent gathers); the sums are native FMA in the
// type of the cycle, rows summed in a fixed order of S interleaved parts.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "amg_small.cuh"
#include "ens_internal.cuh"

namespace ens {
namespace solver {
namespace {

constexpr int kTailBlocks = 8;  // portable cluster size; 16 gave 3 % on the mixed solve and lost 1 % on the batch
constexpr int kTailThreads = 1024;
constexpr size_t kTailSmem = 96 * 1024;

// This thread's part of row i's product with X, columns [c, c + VEC): nonzeros j0 + sub, j0 + sub + S, ...,
// four gathers at a time, then the sum over the S threads of the row (lanes of one warp, `lanes` apart). Every
// thread of a warp calls this the same number of times (valid = false: no row). (Dealing the rest of rows longer
// than 16 to the whole warp was tried for the few rows of a hundred nonzeros among rows of nine: the mixed AMG solve
// on 96^3 took 62.6 ms against 54.6.)
template <typename T, int VEC, bool SHARED>
__device__ __forceinline__ void row_part(bool valid, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                         const T *__restrict__ va, int32_t i, const T *X, int32_t m, int32_t c, int32_t sub,
                                         int32_t S, int32_t lanes, T (&w)[VEC]) {
  // float32: the rounding error of each thread's first product, which an FMA chain over the whole row would not make.
  // Without it rows dealt to many threads are further from float64 than one thread's (a cycle on 32^3 cells of the
  // channel, m = 1, 2 and 8: rms 1.13-1.16 times, with it 1.03-1.04); it costs a cycle 0 to 4 %.
  constexpr bool kErr = sizeof(T) == 4;
  T e[VEC];
#pragma unroll
  for (int q = 0; q < VEC; ++q) w[q] = e[q] = T(0);
  if (valid) {
    const int32_t j1 = __ldg(rp + i + 1);
    bool first = true;
    for (int32_t j = __ldg(rp + i) + sub; j < j1; j += 4 * S) {
      T a[4], x[4][VEC];
      int32_t k[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = j + u * S < j1;
        k[u] = in ? __ldg(ci + j + u * S) : -1;
        a[u] = in ? __ldg(va + j + u * S) : T(0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k[u] >= 0) {
          if constexpr (SHARED)
            load_vec_rw<T, VEC>(X + (int64_t)k[u] * m + c, x[u]);
          else
            load_l2<VEC>(X + (int64_t)k[u] * m + c, x[u]);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k[u] >= 0)
#pragma unroll
          for (int q = 0; q < VEC; ++q) {
            w[q] = fma(a[u], x[u][q], w[q]);
            if (kErr && u == 0 && first) e[q] = fma(a[u], x[u][q], -w[q]);
          }
      first = false;
    }
  }
  for (int32_t off = lanes; off < lanes * S; off <<= 1)
#pragma unroll
    for (int q = 0; q < VEC; ++q) {
      w[q] += __shfl_xor_sync(0xffffffffu, w[q], off);
      if (kErr) e[q] += __shfl_xor_sync(0xffffffffu, e[q], off);
    }
  if (kErr && S > 1)
#pragma unroll
    for (int q = 0; q < VEC; ++q)
      if (isfinite(w[q])) w[q] += e[q];
}

// Position of a thread: column offset c, part `sub` of S of a row, row group `grp` of `groups`.
struct Place {
  int32_t c, sub, grp, groups;
  bool col;
};
template <int VEC>
__device__ __forceinline__ Place place(int32_t tid, int32_t threads, int32_t m, int32_t lanes, int32_t S) {
  Place p;
  p.c = (tid & (lanes - 1)) * VEC;
  p.col = p.c < m;
  p.sub = (tid / lanes) & (S - 1);
  p.grp = tid / (lanes * S);
  p.groups = threads / (lanes * S);
  return p;
}

template <typename T, int VEC>
__device__ __forceinline__ void resid_rows(const Place &p, const int32_t *rp, const int32_t *ci, const T *va, int32_t n, int32_t m,
                                           int32_t lanes, int32_t S, const T *z, const T *r, T *res) {
  for (int32_t i0 = 0; i0 < n; i0 += p.groups) {
    const int32_t i = i0 + p.grp;
    const bool ok = i < n && p.col;
    T w[VEC];
    row_part<T, VEC, false>(ok, rp, ci, va, i, z, m, p.c, p.sub, S, lanes, w);
    if (ok && p.sub == 0) {
      T rv[VEC];
      load_l2<VEC>(r + (int64_t)i * m + p.c, rv);
#pragma unroll
      for (int q = 0; q < VEC; ++q) rv[q] -= w[q];
      store_vec<T, VEC>(res + (int64_t)i * m + p.c, rv);
    }
  }
}

// d0 = D^-1 src / theta, res1 = src - (As src) / theta, z (+)= d0 + c1 d0 + c2 D^-1 res1 (As = A D^-1).
template <typename T, int VEC>
__device__ __forceinline__ void smooth2_rows(const Place &p, const int32_t *rp, const int32_t *ci, const T *va, const T *dinv,
                                             int32_t n, int32_t m, int32_t lanes, int32_t S, bool add, const T *src, T *z,
                                             T inv_theta, T c1, T c2) {
  for (int32_t i0 = 0; i0 < n; i0 += p.groups) {
    const int32_t i = i0 + p.grp;
    const bool ok = i < n && p.col;
    T w[VEC];
    row_part<T, VEC, false>(ok, rp, ci, va, i, src, m, p.c, p.sub, S, lanes, w);
    if (ok && p.sub == 0) {
      T sv[VEC], zv[VEC];
      load_l2<VEC>(src + (int64_t)i * m + p.c, sv);
      if (add) load_l2<VEC>(z + (int64_t)i * m + p.c, zv);
      const T dv = __ldg(dinv + i);
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        const T d0 = dv * sv[q] * inv_theta;
        const T r1 = sv[q] - w[q] * inv_theta;
        const T d1 = c1 * d0 + c2 * (dv * r1);
        zv[q] = add ? zv[q] + (d0 + d1) : d0 + d1;
      }
      store_vec<T, VEC>(z + (int64_t)i * m + p.c, zv);
    }
  }
}

// rc_I = sum of res over the rows of aggregate I, the rows dealt to the S threads of the aggregate.
template <typename T, int VEC>
__device__ __forceinline__ void restrict_rows(const Place &p, const int32_t *__restrict__ ptr, const int32_t *__restrict__ mem, int32_t nc,
                                              int32_t m, int32_t lanes, int32_t S, const T *res, T *rc) {
  for (int32_t i0 = 0; i0 < nc; i0 += p.groups) {
    const int32_t I = i0 + p.grp;
    const bool ok = I < nc && p.col;
    T acc[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] = T(0);
    if (ok) {
      const int32_t t1 = __ldg(ptr + I + 1);
      for (int32_t t = __ldg(ptr + I) + p.sub; t < t1; t += 4 * S) {
        T v[4][VEC];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (t + u * S < t1) load_l2<VEC>(res + (int64_t)__ldg(mem + t + u * S) * m + p.c, v[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (t + u * S < t1)
#pragma unroll
            for (int q = 0; q < VEC; ++q) acc[q] += v[u][q];
      }
    }
    for (int32_t off = lanes; off < lanes * S; off <<= 1)
#pragma unroll
      for (int q = 0; q < VEC; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
    if (ok && p.sub == 0) store_vec<T, VEC>(rc + (int64_t)I * m + p.c, acc);
  }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(256)
    k_small_restrict(const int32_t *ptr, const int32_t *mem, int32_t nc, int32_t m, int32_t lanes, int32_t S, const T *res, T *rc) {
  const Place p = place<VEC>((int32_t)(blockIdx.x * 256 + threadIdx.x), (int32_t)gridDim.x * 256, m, lanes, S);
  restrict_rows<T, VEC>(p, ptr, mem, nc, m, lanes, S, res, rc);
}
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
    k_small_resid(SmallLevel<T> A, int32_t S, const T *z, const T *r, T *res) {
  const Place p = place<VEC>((int32_t)(blockIdx.x * 256 + threadIdx.x), (int32_t)gridDim.x * 256, A.m, A.lanes, S);
  resid_rows<T, VEC>(p, A.rp, A.ci, A.va, A.n, A.m, A.lanes, S, z, r, res);
}
template <typename T, int VEC>
__global__ void __launch_bounds__(256)
    k_small_smooth2(SmallLevel<T> A, int32_t S, int add, const T *src, T *z, T inv_theta, T c1, T c2) {
  const Place p = place<VEC>((int32_t)(blockIdx.x * 256 + threadIdx.x), (int32_t)gridDim.x * 256, A.m, A.lanes, S);
  smooth2_rows<T, VEC>(p, A.rp, A.ci, A.va, A.dinv, A.n, A.m, A.lanes, S, add != 0, src, z, inv_theta, c1, c2);
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The coarsest level's z = S_steps(r) in one block. The four vectors live in shared memory (in_smem) or in the
// level's global blocks; each row group keeps to its own rows except for the product's input d.
template <typename T, int VEC, bool SHARED>
__device__ __forceinline__ void coarse_updates(const TailArgs<T> &a, const TailLevel<T> &L, T *d0, T *d1, T *res, T *z, int32_t S) {
  const Place p = place<VEC>((int32_t)threadIdx.x, kTailThreads, a.m, a.lanes, S);
  const int32_t m = a.m;
  for (int32_t i = p.grp; i < L.n; i += p.groups)
    if (p.col && p.sub == 0) {
      T sv[VEC], dv[VEC];
      load_l2<VEC>(L.r + (int64_t)i * m + p.c, sv);
      const T sc = __ldg(L.dinv + i) * a.inv_theta;
#pragma unroll
      for (int q = 0; q < VEC; ++q) dv[q] = sv[q] * sc;
      store_vec<T, VEC>(res + (int64_t)i * m + p.c, sv);
      store_vec<T, VEC>(d0 + (int64_t)i * m + p.c, dv);
      store_vec<T, VEC>(z + (int64_t)i * m + p.c, dv);
    }
  __syncthreads();
  for (int k = 1; k < a.steps; ++k) {
    const T c1 = a.k1[k], c2 = a.k2[k];
    for (int32_t i0 = 0; i0 < L.n; i0 += p.groups) {
      const int32_t i = i0 + p.grp;
      const bool ok = i < L.n && p.col;
      T w[VEC];
      row_part<T, VEC, SHARED>(ok, L.rp, L.ci, L.va, i, d0, m, p.c, p.sub, S, a.lanes, w);
      if (ok && p.sub == 0) {
        T di[VEC], rs[VEC], zv[VEC];
        load_vec_rw<T, VEC>(d0 + (int64_t)i * m + p.c, di);
        load_vec_rw<T, VEC>(res + (int64_t)i * m + p.c, rs);
        load_vec_rw<T, VEC>(z + (int64_t)i * m + p.c, zv);
        const T dv = __ldg(L.dinv + i);
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          rs[q] -= w[q];
          di[q] = c1 * di[q] + c2 * (dv * rs[q]);
          zv[q] += di[q];
        }
        store_vec<T, VEC>(res + (int64_t)i * m + p.c, rs);
        store_vec<T, VEC>(d1 + (int64_t)i * m + p.c, di);
        store_vec<T, VEC>(z + (int64_t)i * m + p.c, zv);
      }
    }
    __syncthreads();
    T *t = d0;
    d0 = d1;
    d1 = t;
  }
}

// The coarsest level's z = M r, M the dense matrix of its updates: one warp per row and VEC columns, its lanes along
// the row; r from shared memory. Every block of the cluster takes a share of the rows.
template <typename T, int VEC>
__device__ __forceinline__ void coarse_dense(const TailArgs<T> &a, const TailLevel<T> &L, T *r) {
  const int32_t n = L.n, m = a.m, nv = m / VEC, lane = threadIdx.x & 31;
  for (int32_t t = threadIdx.x; t < n * nv; t += kTailThreads) {
    T v[VEC];
    load_l2<VEC>(L.r + (int64_t)t * VEC, v);
    store_vec<T, VEC>(r + (int64_t)t * VEC, v);
  }
  __syncthreads();
  for (int32_t t = blockIdx.x * (kTailThreads / 32) + threadIdx.x / 32; t < n * nv; t += kTailBlocks * (kTailThreads / 32)) {
    const int32_t i = t / nv, c = (t - i * nv) * VEC;
    const T *row = a.dense + (int64_t)i * n;
    T w[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) w[q] = T(0);
    for (int32_t j = lane; j < n; j += 128) {
      T f[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) f[u] = j + 32 * u < n ? __ldg(row + j + 32 * u) : T(0);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j + 32 * u < n) {
          T v[VEC];
          load_vec_rw<T, VEC>(r + (int64_t)(j + 32 * u) * m + c, v);
#pragma unroll
          for (int q = 0; q < VEC; ++q) w[q] = fma(f[u], v[q], w[q]);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int q = 0; q < VEC; ++q) w[q] += __shfl_xor_sync(0xffffffffu, w[q], off);
    if (lane == 0) store_vec<T, VEC>(L.z + (int64_t)i * m + c, w);
  }
}

// Column blockIdx.x of the dense matrix of z = S_steps(r), in float64: the updates applied to a unit vector.
__global__ void __launch_bounds__(256) k_coarse_matrix(MatView A, int32_t steps, double inv_theta, const double *__restrict__ k1,
                                                       const double *__restrict__ k2, double *__restrict__ M, float *__restrict__ M32) {
  extern __shared__ __align__(16) unsigned char raw[];
  const int32_t n = A.n, col = blockIdx.x;
  double *d0 = reinterpret_cast<double *>(raw), *d1 = d0 + n, *res = d1 + n, *z = res + n;
  for (int32_t i = threadIdx.x; i < n; i += 256) {
    res[i] = i == col ? 1.0 : 0.0;
    d0[i] = z[i] = res[i] * A.dinv[i] * inv_theta;
  }
  __syncthreads();
  for (int k = 1; k < steps; ++k) {
    for (int32_t i = threadIdx.x; i < n; i += 256) {
      double w = 0.0;
      for (int32_t j = A.rp[i]; j < A.rp[i + 1]; ++j) w = fma(A.val[j], d0[A.ci[j]], w);
      res[i] -= w;
      d1[i] = k1[k] * d0[i] + k2[k] * (A.dinv[i] * res[i]);
      z[i] += d1[i];
    }
    __syncthreads();
    double *t = d0;
    d0 = d1;
    d1 = t;
  }
  for (int32_t i = threadIdx.x; i < n; i += 256) {
    M[(int64_t)i * n + col] = z[i];
    M32[(int64_t)i * n + col] = (float)z[i];
  }
}

template <typename T, int VEC>
__global__ void __launch_bounds__(kTailThreads) k_amg_tail(const __grid_constant__ TailArgs<T> a, int32_t S, int in_smem) {
  extern __shared__ __align__(16) unsigned char raw[];
  const int32_t rank = (int32_t)blockIdx.x, m = a.m;
  const Place p = place<VEC>(rank * kTailThreads + (int32_t)threadIdx.x, kTailBlocks * kTailThreads, m, a.lanes, S);
  const Place e = place<VEC>(rank * kTailThreads + (int32_t)threadIdx.x, kTailBlocks * kTailThreads, m, a.lanes, 1);
  const int last = a.nl - 1;
  for (int l = 0; l < last; ++l) {
    const TailLevel<T> &L = a.lev[l], &C = a.lev[l + 1];
    smooth2_rows<T, VEC>(p, L.srp, L.sci, L.sva, L.dinv, L.n, m, a.lanes, S, false, L.r, L.z, a.inv_theta, a.c1, a.c2);
    cluster_barrier();
    resid_rows<T, VEC>(p, L.rp, L.ci, L.va, L.n, m, a.lanes, S, L.z, L.r, L.res);
    cluster_barrier();
    restrict_rows<T, VEC>(p, L.ptr, L.mem, L.nc, m, a.lanes, S, L.res, C.r);
    cluster_barrier();
  }
  if (a.dense) {
    coarse_dense<T, VEC>(a, a.lev[last], reinterpret_cast<T *>(raw));
  } else if (rank == 0) {
    const TailLevel<T> &L = a.lev[last];
    if (in_smem) {
      const int64_t blk = (int64_t)L.n * m;
      T *d0 = reinterpret_cast<T *>(raw), *d1 = d0 + blk, *res = d1 + blk, *z = res + blk;
      coarse_updates<T, VEC, true>(a, L, d0, d1, res, z, S);
      const Place g = place<VEC>((int32_t)threadIdx.x, kTailThreads, m, a.lanes, 1);
      for (int32_t i = g.grp; i < L.n && g.col; i += g.groups) {
        T zv[VEC];
        load_vec_rw<T, VEC>(z + (int64_t)i * m + g.c, zv);
        store_vec<T, VEC>(L.z + (int64_t)i * m + g.c, zv);
      }
    } else {
      coarse_updates<T, VEC, false>(a, L, a.da, a.db, a.res, L.z, S);
    }
  }
  cluster_barrier();
  for (int l = last - 1; l >= 0; --l) {
    const TailLevel<T> &L = a.lev[l], &C = a.lev[l + 1];
    for (int32_t i = e.grp; i < L.n && e.col; i += e.groups) {
      T zv[VEC], cv[VEC];
      load_l2<VEC>(L.z + (int64_t)i * m + e.c, zv);
      load_l2<VEC>(C.z + (int64_t)__ldg(L.agg + i) * m + e.c, cv);
#pragma unroll
      for (int q = 0; q < VEC; ++q) zv[q] += cv[q];
      store_vec<T, VEC>(L.z + (int64_t)i * m + e.c, zv);
    }
    cluster_barrier();
    resid_rows<T, VEC>(p, L.rp, L.ci, L.va, L.n, m, a.lanes, S, L.z, L.r, L.res);
    cluster_barrier();
    smooth2_rows<T, VEC>(p, L.srp, L.sci, L.sva, L.dinv, L.n, m, a.lanes, S, true, L.res, L.z, a.inv_theta, a.c1, a.c2);
    if (l > 0) cluster_barrier();
  }
}

template <typename T, int VEC>
cudaError_t run_tail(const TailArgs<T> &a, cudaStream_t st) {
  const TailLevel<T> &C = a.lev[a.nl - 1];
  const size_t need = 4 * (size_t)C.n * a.m * sizeof(T);
  const bool in_smem = need <= kTailSmem;
  const bool dense = a.dense != nullptr && need / 4 <= kTailSmem;
  auto k = k_amg_tail<T, VEC>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTailSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kTailBlocks);
  cfg.blockDim = dim3(kTailThreads);
  cfg.dynamicSmemBytes = dense ? need / 4 : in_smem ? need : 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kTailBlocks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // Four threads per row, on the coarsest level too (channel 96^3, m = 8, mixed solve: 59.5 ms; 8 threads
  // there 63.0, 16: 69.6; 8 or 16 on the other levels as well: 62.0 and 67.8).
  const int32_t S = std::min(4, 32 / a.lanes);
  if (dense || !a.dense) return cudaLaunchKernelEx(&cfg, k, a, S, in_smem ? 1 : 0);
  TailArgs<T> b = a;  // r does not fit: the updates themselves
  b.dense = nullptr;
  return cudaLaunchKernelEx(&cfg, k, b, S, in_smem ? 1 : 0);
}

// Threads per row: the rows of the level spread over the GPU's resident threads (152 SMs x 2048), at most 16
// and at most one warp per row.
int32_t parts(int32_t n, int32_t lanes) {
  int32_t S = 1;
  while (S < 16 && 2 * S * lanes <= 32 && (int64_t)n * lanes * S * 2 <= 152 * 2048) S <<= 1;
  return S;
}
int blocks_for(int32_t n, int32_t lanes, int32_t S) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)n * lanes * S + 255) / 256, 152 * 8));
}

template <typename T, typename F>
cudaError_t with_vec(int vec, F &&f) {
  if (vec == 1) return f(std::integral_constant<int, 1>{});
  if constexpr (sizeof(T) == 4)
    if (vec == 4) return f(std::integral_constant<int, 4>{});
  return f(std::integral_constant<int, 2>{});
}

template <typename T>
cudaError_t small_resid(const SmallLevel<T> &A, int vec, const T *z, const T *r, T *res, cudaStream_t st) {
  const int32_t S = parts(A.n, A.lanes);
  return with_vec<T>(vec, [&](auto V) {
    k_small_resid<T, decltype(V)::value><<<blocks_for(A.n, A.lanes, S), 256, 0, st>>>(A, S, z, r, res);
    return cudaGetLastError();
  });
}
template <typename T>
cudaError_t small_smooth2(const SmallLevel<T> &A, int vec, bool add, const T *src, T *z, T it, T c1, T c2, cudaStream_t st) {
  const int32_t S = parts(A.n, A.lanes);
  return with_vec<T>(vec, [&](auto V) {
    k_small_smooth2<T, decltype(V)::value><<<blocks_for(A.n, A.lanes, S), 256, 0, st>>>(A, S, add ? 1 : 0, src, z, it, c1, c2);
    return cudaGetLastError();
  });
}

template <typename T>
cudaError_t small_restrict(const int32_t *ptr, const int32_t *mem, int32_t nc, int32_t m, int32_t lanes, int vec, const T *res, T *rc,
                           cudaStream_t st) {
  const int32_t S = parts(nc, lanes);
  return with_vec<T>(vec, [&](auto V) {
    k_small_restrict<T, decltype(V)::value><<<blocks_for(nc, lanes, S), 256, 0, st>>>(ptr, mem, nc, m, lanes, S, res, rc);
    return cudaGetLastError();
  });
}

}  // namespace

cudaError_t launch_small_restrict(const int32_t *ptr, const int32_t *mem, int32_t nc, int32_t m, int32_t lanes, int vec, const float *res,
                                  float *rc, cudaStream_t st) {
  return small_restrict<float>(ptr, mem, nc, m, lanes, vec, res, rc, st);
}
cudaError_t launch_small_restrict(const int32_t *ptr, const int32_t *mem, int32_t nc, int32_t m, int32_t lanes, int vec, const double *res,
                                  double *rc, cudaStream_t st) {
  return small_restrict<double>(ptr, mem, nc, m, lanes, vec, res, rc, st);
}
cudaError_t coarse_matrix(const MatView &A, int32_t steps, double inv_theta, const double *k1, const double *k2, double *M, float *M32,
                          cudaStream_t st) {
  const size_t smem = 4 * (size_t)A.n * sizeof(double);
  k_coarse_matrix<<<A.n, 256, smem, st>>>(A, steps, inv_theta, k1, k2, M, M32);
  return cudaGetLastError();
}
cudaError_t launch_amg_tail(const TailArgs<float> &a, int vec, cudaStream_t st) {
  return with_vec<float>(vec, [&](auto V) { return run_tail<float, decltype(V)::value>(a, st); });
}
cudaError_t launch_amg_tail(const TailArgs<double> &a, int vec, cudaStream_t st) {
  return with_vec<double>(vec, [&](auto V) { return run_tail<double, decltype(V)::value>(a, st); });
}
cudaError_t launch_small_resid(const SmallLevel<float> &A, int vec, const float *z, const float *r, float *res, cudaStream_t st) {
  return small_resid<float>(A, vec, z, r, res, st);
}
cudaError_t launch_small_resid(const SmallLevel<double> &A, int vec, const double *z, const double *r, double *res, cudaStream_t st) {
  return small_resid<double>(A, vec, z, r, res, st);
}
cudaError_t launch_small_smooth2(const SmallLevel<float> &A, int vec, bool add, const float *src, float *z, float it, float c1, float c2,
                                 cudaStream_t st) {
  return small_smooth2<float>(A, vec, add, src, z, it, c1, c2, st);
}
cudaError_t launch_small_smooth2(const SmallLevel<double> &A, int vec, bool add, const double *src, double *z, double it, double c1,
                                 double c2, cudaStream_t st) {
  return small_smooth2<double>(A, vec, add, src, z, it, c1, c2, st);
}

}  // namespace solver
}  // namespace ens
