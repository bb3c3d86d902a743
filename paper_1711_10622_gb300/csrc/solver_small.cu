// A plain (unpreconditioned) float64 split solve of a small system as one cooperative launch.
//
// At 32^3 rows an iteration is five launches of 4 to 13 us, each a chain of dependent round trips: row pointers, row
// entries, gathers, partial sums, the ticket, the last block's sums. Here every block keeps its row tile in shared
// memory for the whole solve, the kernels become phases between barriers of the grid, and every block forms the
// totals and the per-column scalars for itself from the partial sums (in shared memory), so nothing is passed on by a
// last block. The phases visit rows and add sums in exactly the order of k_p, k_v, k_s, k_t and k_xr with their grids:
// both forms give the same bits.
//
// What bounds it is the chain of each phase: gathers, the sums of the warps and blocks (an FP64 addition has the latency
// of a shuffle), arrival, partial sums, totals, a division; 4 to 7 us, most of it independent of the rows. Plain
// Dirichlet solve, tol 1e-12, 32^3 rows, m = 4: 6.27 ms as a graph, 5.55 ms here; per 100 iterations, graph / here:
// 8^3 rows m = 4 3.96 / 2.53 ms, m = 8 4.01 / 2.88; 24^3 m = 4 4.31 / 2.76, m = 6 4.85 / 4.29.
// Every block reads every partial sum, so the form loses where there are many: 24^3, m = 8 (216 blocks of 16 sums)
// 5.02 / 5.22; 32^3, m = 8, with four blocks per SM at 64 registers 6.2 / 11.5. Four blocks per SM also left
// eight loads of a lane in flight no registers (32^3, m = 4: 4.04 ms against 3.60).
//
// What other blocks wrote in the launch is read from L2 or after an acquire that drops older lines from L1. A block's
// arrival at the barrier is released after its writes; the waits are bounded: a block that gives up sets bar[1] and
// every block leaves.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "solver_small.cuh"
#include "solver_impl.cuh"

namespace ens {
namespace solver {
namespace {

using T = double;
using Arith = ArithF64Split;
constexpr int kMaxCols = 8;
constexpr unsigned kPolls = 1u << 23;  // of one barrier: seconds
constexpr int kBatch = 8;              // partial sums of a lane on their way together

struct SharedCols {
  T rho[kMaxCols], beta[kMaxCols], alpha[kMaxCols], omega[kMaxCols], thr2[kMaxCols], rh2[kMaxCols], rn2[kMaxCols];
  int32_t state[kMaxCols], iters[kMaxCols], status[kMaxCols], flags[kMaxCols], it[2];
};

template <int LANES, int SVEC, int SLANES>
__global__ void __launch_bounds__(kThreads, 2) k_small_solve(const __grid_constant__ SmallSolve a, const __grid_constant__ Cols<T> g) {
  constexpr int VEC = 2, W = LANES * VEC, G = kThreads / LANES, kWarps = kThreads / 32;
  static_assert(SLANES * SVEC == W && W <= kMaxCols, "one shared buffer for both mappings");
  __shared__ __align__(16) Arith::Tile sm;
  __shared__ __align__(16) int32_t rp[kTileRows + 4];
  __shared__ T wsum[kWarps * 2 * W];
  __shared__ ColTotals<T, 2> tot;
  __shared__ SharedCols sc;
  __shared__ bool dead;
  const int32_t m = a.m;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Cols<T> cs = g;
  cs.rho = sc.rho, cs.beta = sc.beta, cs.alpha = sc.alpha, cs.omega = sc.omega, cs.thr2 = sc.thr2, cs.rh2 = sc.rh2, cs.rn2 = sc.rn2;
  cs.state = sc.state, cs.iters = sc.iters, cs.status = sc.status, cs.flags = sc.flags, cs.it = sc.it;
  if ((int)threadIdx.x < m) {
    const int l = threadIdx.x;
    sc.rho[l] = g.rho[l], sc.beta[l] = g.beta[l], sc.alpha[l] = g.alpha[l], sc.omega[l] = g.omega[l];
    sc.thr2[l] = g.thr2[l], sc.rh2[l] = g.rh2[l], sc.rn2[l] = g.rn2[l];
    sc.state[l] = g.state[l], sc.iters[l] = g.iters[l], sc.status[l] = g.status[l], sc.flags[l] = g.flags[l];
  }
  if (threadIdx.x == 0) {
    sc.it[0] = g.it[0], sc.it[1] = g.it[1];
    dead = false;
  }
  // this block's rows, staged once
  const int R = tile_rows_for(a.A.n, LANES), RPG = R / G;
  const int64_t r0 = (int64_t)blockIdx.x * R;
  const int rows = (int)blockIdx.x < a.tgrid && r0 < a.A.n ? (int)min((int64_t)R, a.A.n - r0) : 0;
  if (rows) stage16<int32_t>(rp, a.A.rp + r0, (rows + 1 + 3) & ~3);
  __syncthreads();
  const int32_t ab = rows ? rp[0] & ~3 : 0, ae = rows ? (rp[rows] + 3) & ~3 : 0;
  const bool staged = ae - ab <= kTileNnz;
  if (rows && staged) Arith::stage(sm, a.A, ab, ae);
  __syncthreads();
  const uint32_t sweep0 = (uint32_t)(r0 / R) * RPG + (threadIdx.x >> 5) * 5u + blockIdx.x;  // as tile_rows
  auto product = [&](const T *X, auto &&epi) {
    const int grp = threadIdx.x / LANES;
    const int32_t c = (threadIdx.x % LANES) * VEC;
#pragma unroll 1
    for (int rr = 0; rr < RPG; ++rr) {
      const int lr = rr * G + grp;
      if (lr >= rows) break;
      const bool nat = (a.mask >> ((sweep0 + rr) & 31)) & 1u;
      if (c < m) {
        T y[VEC];
        if (staged)
          Arith::template row_s<VEC, Coherent>(sm, a.A, ab, rp[lr] - ab, rp[lr + 1] - ab, m, c, X, y, nat);
        else
          Arith::template row_g<VEC, Coherent>(a.A, ab, rp[lr] - ab, rp[lr + 1] - ab, m, c, X, y, nat);
        epi((r0 + lr) * m + c, y);
      }
    }
  };

  unsigned goal = 0;
  auto barrier = [&] {  // of the grid; false: some wait ran out
    __syncthreads();
    if (threadIdx.x == 0) {
      goal += gridDim.x;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
      unsigned at = 0, gone = 0, polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(at) : "l"(a.bar) : "memory");
        if ((++polls & 1023u) == 0) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(gone) : "l"(a.bar + 1) : "memory");
      } while ((int)(at - goal) < 0 && !gone && polls < kPolls);
      if ((int)(at - goal) < 0) {
        atomicExch(a.bar + 1, 1u);
        dead = true;
      }
    }
    __syncthreads();
    return !dead;
  };
  // Totals of the phase's first nb blocks' sums, in every block (reduce_cols' sums in its order). The partial sums of
  // two phases in turn: a block reaches the phase after next only when all have read this one's.
  const size_t half = (size_t)gridDim.x * 2 * m;
  int buf = 0;
  auto totals = [&](auto &acc, auto lanes, int nb) {
    constexpr int ND = sizeof(acc) / sizeof(acc[0]), V = sizeof(acc[0]) / sizeof(T), L = decltype(lanes)::value;
    T *const part = a.partials + buf * half;
    buf ^= 1;
    if ((int)blockIdx.x < nb) {
      T(&ws)[kWarps][ND][L * V] = reinterpret_cast<T(&)[kWarps][ND][L * V]>(wsum);
      warp_cols<T, ND, V, L>(acc, ws);
      __syncthreads();
      if ((int)threadIdx.x < ND * m) {
        const int d = threadIdx.x / m, c = threadIdx.x - d * m;
        T b = ws[0][d][c];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) b += ws[w][d][c];
        part[(size_t)blockIdx.x * ND * m + threadIdx.x] = b;
      }
    }
    if (!barrier()) return false;
    for (int t = warp; t < ND * m; t += kWarps) {
      T s = T(0);
      for (int b0 = lane; b0 < nb; b0 += 32 * kBatch) {
        T v[kBatch][1];
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
          if (b0 + 32 * k < nb) load_l2<1>(part + (size_t)(b0 + 32 * k) * ND * m + t, v[k]);
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
          if (b0 + 32 * k < nb) s += v[k][0];
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) tot.v[t / m][t % m] = s;
    }
    __syncthreads();
    return true;
  };
  using PL = std::integral_constant<int, LANES>;
  using SL = std::integral_constant<int, SLANES>;
  // rows of the vector updates: ENS_ROWS of k_p, k_s (four columns per thread) and k_xr
  const int32_t cs_ = (threadIdx.x % SLANES) * SVEC, cx = (threadIdx.x % LANES) * VEC;
  auto stream_rows = [&](auto lanes, int nb, auto &&fn) {
    constexpr int L = decltype(lanes)::value;
    if ((int)blockIdx.x < nb)
      for (int64_t i = (int64_t)blockIdx.x * (kThreads / L) + threadIdx.x / L; i < a.A.n; i += (int64_t)nb * (kThreads / L)) fn(i);
  };

  while (sc.it[1]) {
    {  // k_p
      T beta[SVEC], om[SVEC];
      bool act[SVEC];
#pragma unroll
      for (int q = 0; q < SVEC; ++q) {
        act[q] = cs_ + q < m && sc.state[min(cs_ + q, kMaxCols - 1)] == ST_ACTIVE;
        beta[q] = act[q] ? sc.beta[cs_ + q] : T(0);
        om[q] = act[q] ? sc.omega[cs_ + q] : T(0);
      }
      if (cs_ < m)
        stream_rows(SL{}, a.sgrid, [&](int64_t i) {
          T rv[SVEC], pv[SVEC], vv[SVEC];
          load_l2<SVEC>(a.r + i * m + cs_, rv);
          load_l2<SVEC>(a.p + i * m + cs_, pv);
          load_l2<SVEC>(a.v + i * m + cs_, vv);
#pragma unroll
          for (int q = 0; q < SVEC; ++q) pv[q] = act[q] ? rv[q] + beta[q] * (pv[q] - om[q] * vv[q]) : pv[q];
          store_vec<T, SVEC>(a.p + i * m + cs_, pv);
        });
      if (!barrier()) return;
    }
    {  // k_v
      T acc[1][VEC] = {};
      product(a.p, [&](int64_t at, const T(&y)[VEC]) {
        T h[VEC];
        store_vec<T, VEC>(a.v + at, y);
        load_vec<T, VEC>(a.rh + at, h);
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[0][q] += h[q] * y[q];
      });
      if (!totals(acc, PL{}, a.tgrid)) return;
      if ((int)threadIdx.x < m) step_alpha<T>(cs, threadIdx.x, tot.v[0][threadIdx.x]);
      __syncthreads();
    }
    {  // k_s
      T acc[1][SVEC] = {}, al[SVEC];
      int32_t on[SVEC];
#pragma unroll
      for (int q = 0; q < SVEC; ++q) {
        al[q] = cs_ + q < m && sc.state[min(cs_ + q, kMaxCols - 1)] == ST_ACTIVE ? sc.alpha[cs_ + q] : T(0);
        on[q] = al[q] != T(0) ? 1 : 0;
      }
      if (cs_ < m)
        stream_rows(SL{}, a.sgrid, [&](int64_t i) {
          T rv[SVEC], vv[SVEC];
          load_l2<SVEC>(a.r + i * m + cs_, rv);
          load_l2<SVEC>(a.v + i * m + cs_, vv);
#pragma unroll
          for (int q = 0; q < SVEC; ++q) {
            rv[q] = on[q] ? rv[q] - al[q] * vv[q] : rv[q];
            acc[0][q] += rv[q] * rv[q];
          }
          store_vec<T, SVEC>(a.s + i * m + cs_, rv);
        });
      if (!totals(acc, SL{}, a.sgrid)) return;
      if ((int)threadIdx.x < m) step_half<T>(cs, threadIdx.x, tot.v[0][threadIdx.x]);
      __syncthreads();
    }
    {  // k_t
      T acc[2][VEC] = {};
      product(a.s, [&](int64_t at, const T(&y)[VEC]) {
        T sv[VEC];
        store_vec<T, VEC>(a.t + at, y);
        load_l2<VEC>(a.s + at, sv);
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          acc[0][q] += y[q] * sv[q];
          acc[1][q] += y[q] * y[q];
        }
      });
      if (!totals(acc, PL{}, a.tgrid)) return;
      if ((int)threadIdx.x < m) step_omega<T>(cs, threadIdx.x, tot.v[0][threadIdx.x], tot.v[1][threadIdx.x]);
      __syncthreads();
    }
    {  // k_xr
      T acc[2][VEC] = {}, al[VEC], om[VEC];
      int st[VEC];
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        st[q] = cx + q < m ? sc.state[min(cx + q, kMaxCols - 1)] : ST_DONE;
        al[q] = st[q] == ST_DONE ? T(0) : sc.alpha[cx + q];
        om[q] = st[q] == ST_ACTIVE ? sc.omega[cx + q] : T(0);
      }
      if (cx < m)
        stream_rows(PL{}, a.grid, [&](int64_t i) {
          T xv[VEC], pv[VEC], sv[VEC], tv[VEC], hv[VEC];
          load_l2<VEC>(a.x + i * m + cx, xv);
          load_l2<VEC>(a.p + i * m + cx, pv);
          load_l2<VEC>(a.s + i * m + cx, sv);
          load_l2<VEC>(a.t + i * m + cx, tv);
          load_vec<T, VEC>(a.rh + i * m + cx, hv);
#pragma unroll
          for (int q = 0; q < VEC; ++q) {
            const T xa = xv[q] + al[q] * pv[q];
            xv[q] = st[q] == ST_ACTIVE ? xa + om[q] * sv[q] : st[q] == ST_HALF ? xa : xv[q];
            sv[q] = st[q] == ST_ACTIVE ? sv[q] - om[q] * tv[q] : sv[q];
            acc[0][q] += sv[q] * sv[q];
            acc[1][q] += hv[q] * sv[q];
          }
          store_vec<T, VEC>(a.x + i * m + cx, xv);
          store_vec<T, VEC>(a.r + i * m + cx, sv);
        });
      const int32_t it = sc.it[0] + 1;
      if (!totals(acc, PL{}, a.grid)) return;
      bool go = false;
      if ((int)threadIdx.x < m) go = step_end<T>(cs, threadIdx.x, tot.v[0][threadIdx.x], tot.v[1][threadIdx.x], it, a.max_iter);
      const int any = __syncthreads_or(go);
      if (threadIdx.x == 0) {
        sc.it[0] = it;
        sc.it[1] = any && it < a.max_iter;
      }
      __syncthreads();
    }
  }
  if (blockIdx.x == 0 && (int)threadIdx.x < m) {
    const int l = threadIdx.x;
    g.rho[l] = sc.rho[l], g.beta[l] = sc.beta[l], g.alpha[l] = sc.alpha[l], g.omega[l] = sc.omega[l], g.rn2[l] = sc.rn2[l];
    g.state[l] = sc.state[l], g.iters[l] = sc.iters[l], g.status[l] = sc.status[l], g.flags[l] = sc.flags[l];
    if (l == 0) g.it[0] = sc.it[0], g.it[1] = sc.it[1];
  }
}

template <typename F>
cudaError_t with_kernel(int m, F &&f) {
  switch (m) {
    case 2: return f(k_small_solve<1, 2, 1>);
    case 4: return f(k_small_solve<2, 4, 1>);
    case 6: return f(k_small_solve<4, 2, 4>);
    case 8: return f(k_small_solve<4, 4, 2>);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

constexpr int kMaxSums = 1536;  // blocks times columns, between 24^3 rows with m = 6 (1296) and m = 8 (1728)

int small_solve_blocks(const SmallSolve &a, int64_t tiles, int num_sms) {
  if (a.m < 2 || a.m > kMaxCols || a.m % 2 || a.tgrid != tiles) return 0;
  const int blocks = std::max(a.tgrid, std::max(a.grid, a.sgrid));
  if (blocks * a.m > kMaxSums) return 0;
  int per_sm = 0;
  const cudaError_t e = with_kernel(a.m, [&](auto *k) { return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kThreads, 0); });
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e == cudaSuccess && blocks <= per_sm * num_sms ? blocks : 0;
}

cudaError_t launch_small_solve(const SmallSolve &a, const Cols<double> &cs, int blocks, cudaStream_t st) {
  SmallSolve arg = a;
  Cols<double> c = cs;
  void *args[] = {&arg, &c};
  return with_kernel(a.m, [&](auto *k) { return cudaLaunchCooperativeKernel((const void *)k, dim3(blocks), dim3(kThreads), args, 0, st); });
}

}  // namespace solver
}  // namespace ens
