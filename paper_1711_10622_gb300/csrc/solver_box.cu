// The solver's products by row boxes (boxprod.cuh): the kernels of solver_impl.cuh whose body is a product, with
// the same epilogues. A thread owns one row and all columns of a chunk; the dot products of a row stay in its
// registers and are reduced once at the end of the kernel.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "boxprod.cuh"
#include "boxsolve.cuh"
#include "solver_impl.cuh"

namespace ens {
namespace solver {
namespace {

// Asks for the line of a row of another block that the epilogue will read, while the products are formed.
template <typename T>
__device__ __forceinline__ void ask(const T *p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// CW elements as 32-byte (float32 x 4: 16-byte) accesses.
template <typename T, int CW>
__device__ __forceinline__ void load_row(const T *p, T (&v)[CW]) {
  constexpr int W = CW * sizeof(T) >= 32 ? 32 / sizeof(T) : CW;
#pragma unroll
  for (int h = 0; h < CW; h += W) {
    if constexpr (sizeof(T) == 8)
      asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v[h]), "=d"(v[h + 1]), "=d"(v[h + 2]), "=d"(v[h + 3]) : "l"(p + h) : "memory");
    else if constexpr (W == 8)
      asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=f"(v[h]), "=f"(v[h + 1]), "=f"(v[h + 2]), "=f"(v[h + 3]), "=f"(v[h + 4]), "=f"(v[h + 5]), "=f"(v[h + 6]), "=f"(v[h + 7])
                   : "l"(p + h)
                   : "memory");
    else
      asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[h]), "=f"(v[h + 1]), "=f"(v[h + 2]), "=f"(v[h + 3]) : "l"(p + h) : "memory");
  }
}
template <typename T, int CW>
__device__ __forceinline__ void store_row(T *p, const T (&v)[CW]) {
  constexpr int W = CW * sizeof(T) >= 32 ? 32 / sizeof(T) : CW;
#pragma unroll
  for (int h = 0; h < CW; h += W) {
    if constexpr (sizeof(T) == 8)
      asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p + h), "d"(v[h]), "d"(v[h + 1]), "d"(v[h + 2]), "d"(v[h + 3]) : "memory");
    else if constexpr (W == 8)
      asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p + h), "f"(v[h]), "f"(v[h + 1]), "f"(v[h + 2]), "f"(v[h + 3]),
                   "f"(v[h + 4]), "f"(v[h + 5]), "f"(v[h + 6]), "f"(v[h + 7])
                   : "memory");
    else
      asm volatile("st.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p + h), "f"(v[h]), "f"(v[h + 1]), "f"(v[h + 2]), "f"(v[h + 3]) : "memory");
  }
}

// Per-column totals of ND sums kept by every thread for its chunk's CW columns (chunk blockIdx.x modulo the
// chunks), then fin(column, totals) in the last block. The block's staging memory carries the threads' sums:
// value v of thread t at v * 256 + t; each warp adds values v, v + 8, ... by eight rows per lane and a butterfly.
// Fixed order throughout, no atomics on values.
template <typename T, int ND, int CW, typename Fin>
__device__ __forceinline__ void box_reduce(const T (&acc)[ND][CW], int32_t m, T *__restrict__ partials, unsigned *__restrict__ counter, Fin &&fin) {
  extern __shared__ __align__(16) unsigned char box_sm[];
  T *const sm = reinterpret_cast<T *>(box_sm);
  __shared__ ColTotals<T, ND> tot;
  __shared__ bool is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
#pragma unroll
  for (int d = 0; d < ND; ++d)
#pragma unroll
    for (int q = 0; q < CW; ++q) sm[(d * CW + q) * kBoxRows + threadIdx.x] = acc[d][q];
  __syncthreads();
  for (int v = warp; v < ND * CW; v += kBoxRows / 32) {
    T s = sm[v * kBoxRows + lane];
#pragma unroll
    for (int j = 1; j < kBoxRows / 32; ++j) s += sm[v * kBoxRows + lane + 32 * j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) partials[(size_t)blockIdx.x * ND * CW + v] = s;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const int nch = m / CW;
  for (int t = warp; t < ND * m; t += kBoxRows / 32) {
    const int d = t / m, l = t - d * m, ch = l / CW, q = l - ch * CW;
    T s = T(0);
    for (int b = ch + lane * nch; b < (int)gridDim.x; b += 32 * nch) s += __ldcg(partials + (size_t)b * ND * CW + d * CW + q);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) tot.v[d][l] = s;
  }
  __syncthreads();
  if ((int)threadIdx.x < m) fin((int)threadIdx.x, tot);
  __syncthreads();
  if (threadIdx.x == 0) *counter = 0u;
}

template <typename T, int CW>
__device__ __forceinline__ void clear(T (&a)[CW]) {
#pragma unroll
  for (int q = 0; q < CW; ++q) a[q] = T(0);
}

#define ENS_BOX_KERNEL(T, CW) __global__ void __launch_bounds__(BoxShape<T, CW>::kThr, BoxShape<T, CW>::kBlocks)
template <typename T, int CW>
constexpr int wide() {
  return CW * sizeof(T) >= 32 ? 32 / (int)sizeof(T) : CW;
}

template <typename T, int CW, int K0>
ENS_BOX_KERNEL(T, CW)
    kb_v(BoxPlan B, MatView A, int32_t m, const T *__restrict__ ph, T *__restrict__ v, const T *__restrict__ rh, Cols<T> cs, T *partials,
         unsigned *counter) {
  T acc[1][CW];
  clear<T, CW>(acc[0]);
  box_rows<T, CW, wide<T, CW>(), true, K0, false, false>(B, A, m, ph, [&](int64_t i, int32_t c) { ask(rh + i * m + c); }, [&](int64_t i, int32_t c, const T (&y)[CW]) {
    T h[CW];
    load_row<T, CW>(rh + i * m + c, h);
    store_row<T, CW>(v + i * m + c, y);
#pragma unroll
    for (int q = 0; q < CW; ++q) acc[0][q] += h[q] * y[q];
  });
  box_reduce<T, 1, CW>(acc, m, partials, counter, [&](int l, const ColTotals<T, 1> &t) { step_alpha<T>(cs, l, t.v[0][l]); });
}

// (The two sums per column beside the product's own spill 84-96 bytes at eight float64 columns and 48-60 at four.)
template <typename T, int CW, int K0>
ENS_BOX_KERNEL(T, CW)
    kb_t(BoxPlan B, MatView A, int32_t m, const T *__restrict__ sh, T *__restrict__ t, const T *__restrict__ s, Cols<T> cs, T *partials,
         unsigned *counter) {
  T acc[2][CW];
  clear<T, CW>(acc[0]);
  clear<T, CW>(acc[1]);
  box_rows<T, CW, wide<T, CW>(), true, K0, false, false>(B, A, m, sh, [&](int64_t i, int32_t c) { ask(s + i * m + c); }, [&](int64_t i, int32_t c, const T (&y)[CW]) {
    T sv[CW];
    load_row<T, CW>(s + i * m + c, sv);
    store_row<T, CW>(t + i * m + c, y);
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      acc[0][q] += y[q] * sv[q];
      acc[1][q] += y[q] * y[q];
    }
  });
  box_reduce<T, 2, CW>(acc, m, partials, counter, [&](int l, const ColTotals<T, 2> &tt) { step_omega<T>(cs, l, tt.v[0][l], tt.v[1][l]); });
}

template <typename T, int CW, int K0>
ENS_BOX_KERNEL(T, CW)
    kb_resid(BoxPlan B, MatView A, int32_t m, const T *__restrict__ b, const T *__restrict__ x, T *__restrict__ r, int outer, Cols<T> cs,
             T *partials, unsigned *counter) {
  T acc[1][CW];
  clear<T, CW>(acc[0]);
  box_rows<T, CW, wide<T, CW>(), true, K0, false, false>(B, A, m, x, [&](int64_t i, int32_t c) { ask(b + i * m + c); }, [&](int64_t i, int32_t c, const T (&ax)[CW]) {
    T y[CW];
    load_row<T, CW>(b + i * m + c, y);
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      y[q] -= ax[q];
      acc[0][q] += y[q] * y[q];
    }
    if (r) store_row<T, CW>(r + i * m + c, y);
  });
  box_reduce<T, 1, CW>(acc, m, partials, counter, [&](int l, const ColTotals<T, 1> &t) { residual_norm<T>(cs, l, t.v[0][l], outer); });
}

// z1 = (1 + c1) z - c1 zp + c2 D^-1 (src - A z): four FP64 operations per element on a pipe of two per clock and SM (A z
// is widened in integer arithmetic), where the form with the updates d and the running residual took five and moved
// six streams instead of four.
template <typename T, int CW, int K0, bool FIRST>
ENS_BOX_KERNEL(T, CW)
    kb_cheb(BoxPlan B, MatView A, int32_t m, const T *__restrict__ z, const T *zp, const T *__restrict__ src, T *z1, T c1, T c2) {
  const T *const dinv = [&] {
    if constexpr (sizeof(T) == 8)
      return A.dinv;
    else
      return A.dinv32;
  }();
  auto ahead = [&](int64_t i, int32_t c) {
    ask(src + i * m + c);
    if (!FIRST) ask(zp + i * m + c);
  };
  box_rows<T, CW, wide<T, CW>(), true, K0, true, false>(B, A, m, z, ahead, [&](int64_t i, int32_t c, const T (&w)[CW]) {
    T zv[CW], pv[CW], sv[CW];
    load_row<T, CW>(src + i * m + c, sv);
    load_row<T, CW>(z + i * m + c, zv);
    if (!FIRST) load_row<T, CW>(zp + i * m + c, pv);
    const T g = c2 * __ldg(dinv + i), a = T(1) + c1;
#pragma unroll
    for (int q = 0; q < CW; ++q) {
      const T t = FIRST ? a * zv[q] : fma(a, zv[q], -(c1 * pv[q]));
      zv[q] = fma(g, sv[q] - w[q], t);
    }
    store_row<T, CW>(z1 + i * m + c, zv);
  });
}

template <typename T, int CW, int K0>
ENS_BOX_KERNEL(T, CW)
    kb_amg_resid(BoxPlan B, MatView A, int32_t m, const T *__restrict__ z, const T *__restrict__ r, T *__restrict__ res) {
  box_rows<T, CW, wide<T, CW>(), true, K0, true, false>(B, A, m, z, [&](int64_t i, int32_t c) { ask(r + i * m + c); }, [&](int64_t i, int32_t c, const T (&w)[CW]) {
    T rv[CW];
    load_row<T, CW>(r + i * m + c, rv);
#pragma unroll
    for (int q = 0; q < CW; ++q) rv[q] -= w[q];
    store_row<T, CW>(res + i * m + c, rv);
  });
}

template <typename T, int CW, int K0, bool ADD>
ENS_BOX_KERNEL(T, CW)
    kb_amg_smooth2(BoxPlan B, MatView As, const T *__restrict__ dinv, int32_t m, const T *__restrict__ src, T *z, T inv_theta, T c1, T c2) {
  auto ahead = [&](int64_t i, int32_t c) {
    if (ADD) ask(z + i * m + c);
  };
  box_rows<T, CW, wide<T, CW>(), true, K0, true, false>(B, As, m, src, ahead, [&](int64_t i, int32_t c, const T (&w)[CW]) {
    T sv[CW], zv[CW];
    load_row<T, CW>(src + i * m + c, sv);
    if (ADD) load_row<T, CW>(z + i * m + c, zv);
    // d0 + c1 d0 + c2 D^-1 (src - w / theta), d0 = D^-1 src / theta
    const T dv = __ldg(dinv + i);
    if constexpr (sizeof(T) == 4) {
      // term by term: the row's factors taken together and rounded once are off by the same amount in every row of
      // a uniform grid, and the whole float32 cycle was a third further from its float64 result
#pragma unroll
      for (int q = 0; q < CW; ++q) {
        const T d0 = dv * sv[q] * inv_theta, d1 = c1 * d0 + c2 * (dv * (sv[q] - w[q] * inv_theta));
        zv[q] = ADD ? zv[q] + (d0 + d1) : d0 + d1;
      }
    } else {  // together: three FP64 operations per element on a pipe of two per clock
      const T g = dv * (inv_theta * (T(1) + c1) + c2), h = dv * c2 * inv_theta;
#pragma unroll
      for (int q = 0; q < CW; ++q) {
        const T u = fma(g, sv[q], -(h * w[q]));
        zv[q] = ADD ? zv[q] + u : u;
      }
    }
    store_row<T, CW>(z + i * m + c, zv);
  });
}

// Chunk width as a compile-time constant, seven slots or B.K.
template <typename T, typename F>
cudaError_t with_shape(const BoxPlan &B, int m, F &&f) {
  using std::integral_constant;
  auto k = [&](auto CW) { return B.K == 7 ? f(CW, integral_constant<int, 7>{}) : f(CW, integral_constant<int, 0>{}); };
  if (m == 4) return k(integral_constant<int, 4>{});
  if constexpr (sizeof(T) == 4)
    if (m == 16) return k(integral_constant<int, 16>{});
  return k(integral_constant<int, 8>{});
}

// chunks > 1: one chunk per block (blocks a multiple of the chunks); else every chunk in turn.
template <typename T, int CW, typename Kern, typename... Args>
cudaError_t go(const BoxPlan &B, int chunks, int sms, cudaStream_t st, Kern k, Args... args) {
  using S = BoxShape<T, CW>;
  const size_t smem = S::smem(B.K);
  // for the longest rows: a size by row length could be lowered by another thread before this one launches
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem(kBoxMaxLen));
  if (e != cudaSuccess) return e;
  int64_t per = (int64_t)sms * S::kBlocks / chunks;
  per = std::max<int64_t>(1, std::min<int64_t>(per, B.boxes));
  k<<<(unsigned)(per * chunks), S::kThr, smem, st>>>(args...);
  return cudaGetLastError();
}

template <typename T>
cudaError_t box_v(const BoxPlan &B, const MatView &A, int32_t m, const T *ph, T *v, const T *rh, const Cols<T> &cs, T *partials,
                  unsigned *counter, int sms, cudaStream_t st) {
  return with_shape<T>(B, m, [&](auto CW, auto K) {
    return go<T, CW.value>(B, m / CW.value, sms, st, kb_v<T, CW.value, K.value>, B, A, m, ph, v, rh, cs, partials, counter);
  });
}
template <typename T>
cudaError_t box_t(const BoxPlan &B, const MatView &A, int32_t m, const T *sh, T *t, const T *s, const Cols<T> &cs, T *partials, unsigned *counter,
                  int sms, cudaStream_t st) {
  return with_shape<T>(B, m, [&](auto CW, auto K) {
    return go<T, CW.value>(B, m / CW.value, sms, st, kb_t<T, CW.value, K.value>, B, A, m, sh, t, s, cs, partials, counter);
  });
}
template <typename T>
cudaError_t box_cheb(const BoxPlan &B, const MatView &A, int32_t m, const T *z, const T *zp, const T *src, T *z1, T c1, T c2, int sms,
                     cudaStream_t st) {
  return with_shape<T>(B, m, [&](auto CW, auto K) {
    if (zp) return go<T, CW.value>(B, 1, sms, st, kb_cheb<T, CW.value, K.value, false>, B, A, m, z, zp, src, z1, c1, c2);
    return go<T, CW.value>(B, 1, sms, st, kb_cheb<T, CW.value, K.value, true>, B, A, m, z, zp, src, z1, c1, c2);
  });
}
template <typename T>
cudaError_t box_amg_resid(const BoxPlan &B, const MatView &A, int32_t m, const T *z, const T *r, T *res, int sms, cudaStream_t st) {
  return with_shape<T>(B, m, [&](auto CW, auto K) { return go<T, CW.value>(B, 1, sms, st, kb_amg_resid<T, CW.value, K.value>, B, A, m, z, r, res); });
}
template <typename T>
cudaError_t box_smooth2(const BoxPlan &B, const MatView &As, const T *dinv, int32_t m, bool add, const T *src, T *z, T it, T c1, T c2, int sms,
                        cudaStream_t st) {
  return with_shape<T>(B, m, [&](auto CW, auto K) {
    if (add) return go<T, CW.value>(B, 1, sms, st, kb_amg_smooth2<T, CW.value, K.value, true>, B, As, dinv, m, src, z, it, c1, c2);
    return go<T, CW.value>(B, 1, sms, st, kb_amg_smooth2<T, CW.value, K.value, false>, B, As, dinv, m, src, z, it, c1, c2);
  });
}

}  // namespace

#ifdef ENS_BOX_F32
using Real = float;
#else
using Real = double;
cudaError_t launch_box_resid(const BoxPlan &B, const MatView &A, int32_t m, const double *b, const double *x, double *r, int outer,
                             const Cols<double> &cs, double *partials, unsigned *counter, int sms, cudaStream_t st) {
  return with_shape<double>(B, m, [&](auto CW, auto K) {
    return go<double, CW.value>(B, m / CW.value, sms, st, kb_resid<double, CW.value, K.value>, B, A, m, b, x, r, outer, cs, partials, counter);
  });
}
#endif
cudaError_t launch_box_v(const BoxPlan &B, const MatView &A, int32_t m, const Real *ph, Real *v, const Real *rh, const Cols<Real> &cs,
                         Real *partials, unsigned *counter, int sms, cudaStream_t st) {
  return box_v<Real>(B, A, m, ph, v, rh, cs, partials, counter, sms, st);
}
cudaError_t launch_box_t(const BoxPlan &B, const MatView &A, int32_t m, const Real *sh, Real *t, const Real *s, const Cols<Real> &cs,
                         Real *partials, unsigned *counter, int sms, cudaStream_t st) {
  return box_t<Real>(B, A, m, sh, t, s, cs, partials, counter, sms, st);
}
cudaError_t launch_box_cheb(const BoxPlan &B, const MatView &A, int32_t m, const Real *z, const Real *zp, const Real *src, Real *z1, Real c1,
                            Real c2, int sms, cudaStream_t st) {
  return box_cheb<Real>(B, A, m, z, zp, src, z1, c1, c2, sms, st);
}
cudaError_t launch_box_amg_resid(const BoxPlan &B, const MatView &A, int32_t m, const Real *z, const Real *r, Real *res, int sms,
                                 cudaStream_t st) {
  return box_amg_resid<Real>(B, A, m, z, r, res, sms, st);
}
cudaError_t launch_box_smooth2(const BoxPlan &Bs, const MatView &As, const Real *dinv, int32_t m, bool add, const Real *src, Real *z,
                               Real inv_theta, Real c1, Real c2, int sms, cudaStream_t st) {
  return box_smooth2<Real>(Bs, As, dinv, m, add, src, z, inv_theta, c1, c2, sms, st);
}

}  // namespace solver
}  // namespace ens
