// GSpMV Y = A X for a CSR matrix and an n x m row-interleaved block (Section 2.3, Fig. GSpMV).
//
// Work mapping: a "row group" of LANES consecutive threads owns one row at a time; each lane
// owns VEC consecutive columns of that row and reads them from X with 16-byte loads (one double2
// or float4; four doubles as two double2), so a row of X (m contiguous values) is read by the
// group as one contiguous segment. Every val[j] and col_idx[j] is loaded once per lane group and
// reused for all the lane's columns; with LANES = m / VEC there is exactly one pass per row. The
// grid is sized to fill the GPU once and strides over tiles of rows; a launch may also cover a
// row range only (the pipelined host-buffer product).
//
// Three arithmetic variants:
//   * float32 (ENS_F32): float products and sums (inner solver of the mixed-precision mode).
//   * native float64: one DFMA per product.
//   * split float64: FP64-accurate products on the FP32 pipe. GB300's FP64 rate is a small
//     fraction of its FP32 rate, so native DFMA makes the FP64 product ALU-bound for m >= 2;
//     here each value is carried as an unevaluated sum hi + lo of two floats (about 47
//     significant bits) and each row sum is accumulated error-free in (hi, lo) form. Segments
//     whose X values fall outside the split range are recomputed with native DFMA.
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include <cstdint>
#include <vector>

#include "boxprod.cuh"
#include "ens_internal.cuh"
#include "rowprod.cuh"

namespace ens {
namespace {

MatView view_of(const ens_matrix *A) {
  return MatView{(int32_t)A->n, A->row, A->col, A->val, A->val32, A->valsplit, A->dinv, A->dinv32};
}

// Tiled GSpMV: CSR segments staged in shared memory (tile_rows), Y written with streaming stores.
template <typename Arith, int VEC, int LANES, int R0 = 0>
__device__ __forceinline__ void gspmv_body(const MatView &A, int32_t m, const typename Arith::T *__restrict__ X,
                                           typename Arith::T *__restrict__ Y, uint32_t native_mask) {
  using T = typename Arith::T;
  tile_rows<Arith, VEC, LANES, R0>(A, m, X, native_mask,
                                   [&](int64_t i, int32_t c, const T (&y)[VEC]) { store_vec_cs<T, VEC>(Y + i * m + c, y); });
}

template <typename Arith, int VEC, int LANES>
__global__ void __launch_bounds__(kThreads)
    gspmv_kernel(MatView A, int32_t m, const typename Arith::T *__restrict__ X, typename Arith::T *__restrict__ Y,
                 uint32_t native_mask) {
  gspmv_body<Arith, VEC, LANES>(A, m, X, Y, native_mask);
}

// Register caps (minimum resident blocks per SM) for the gather-latency-bound kernels, which need
// resident warps more than registers. Measured on GB300, channel 256 x 128 x 128:
//   * split float64, two columns per lane: 6 blocks, 40 registers (6 beat 5 by 1-10 % over
//     m = 2..32; 7 or 8 blocks spill and lose 1-10 %);
//   * split float64, four columns per lane: 5 blocks, 48 registers (6 spill 164-212 bytes; 4 blocks
//     with 64 registers lose 2-12 %);
//   * float32: 8 blocks, 32 registers (10-12 % faster than the compiler's own 40 registers over
//     m = 8..32).
// Native float64 keeps the compiler's own choice (no minimum): a minimum of one block, which asks
// for no occupancy at all, let the compiler take far more registers and halved the launches (split
// kernels: 125-140 registers; native m = 32: 3.3 ms against 1.7 ms).
template <typename Arith, int VEC>
struct MinBlocks {
  static constexpr int value = std::is_same<Arith, ArithF32>::value ? 8 : VEC == 4 ? 5 : 6;
};
// R0: rows of a tile where they are known at compile time (0: by the rows of the product, tile_rows_for). At 32 registers
// the float32 kernels spill 40-72 bytes with a tile height of their own (two columns per lane, and four with two lanes
// per row: m = 8 6.4 us against 5.5 on 127872 rows), so whole tiles have instances of theirs.
template <typename Arith, int VEC, int LANES, int R0 = 0>
__global__ void __launch_bounds__(kThreads, MinBlocks<Arith, VEC>::value)
    gspmv_kernel_capped(MatView A, int32_t m, const typename Arith::T *__restrict__ X,
                        typename Arith::T *__restrict__ Y, uint32_t native_mask) {
  gspmv_body<Arith, VEC, LANES, R0>(A, m, X, Y, native_mask);
}

// Untiled variant (direct_rows): an autotuner candidate beside the tiled kernels.
template <typename Arith, int VEC, int LANES>
__global__ void __launch_bounds__(kThreads, MinBlocks<Arith, VEC>::value)
    gspmv_kernel_direct(MatView A, int32_t m, const typename Arith::T *__restrict__ X,
                        typename Arith::T *__restrict__ Y, uint32_t native_mask) {
  using T = typename Arith::T;
  direct_rows<Arith, VEC, LANES>(A, m, X, native_mask,
                                 [&](int64_t i, int32_t c, const T (&y)[VEC]) { store_vec_cs<T, VEC>(Y + i * m + c, y); });
}
template <typename Arith, int VEC, int LANES>
__global__ void __launch_bounds__(kThreads)
    gspmv_kernel_direct_free(MatView A, int32_t m, const typename Arith::T *__restrict__ X,
                             typename Arith::T *__restrict__ Y, uint32_t native_mask) {
  using T = typename Arith::T;
  direct_rows<Arith, VEC, LANES>(A, m, X, native_mask,
                                 [&](int64_t i, int32_t c, const T (&y)[VEC]) { store_vec_cs<T, VEC>(Y + i * m + c, y); });
}

// Resident blocks per SM of a kernel (threads, dynamic shared memory), asked for once per kernel instance and kept in
// its caller's `known` (0: not yet): the query costs a microsecond or two of every small product's launch. All GPUs
// this library is built for are the same part.
int resident(std::atomic<int> &known, const void *kernel, int threads, size_t smem) {
  int n = known.load(std::memory_order_relaxed);
  if (n > 0) return n;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess) {
    (void)cudaGetLastError();
    return 1;
  }
  n = n < 1 ? 1 : n;
  known.store(n, std::memory_order_relaxed);
  return n;
}

// Product by row boxes (boxprod.cuh).
template <typename T, int CW, int ACC, bool FULL, int K0>
__global__ void __launch_bounds__(BoxShape<T, CW>::kThr, BoxShape<T, CW>::kBlocks)
    gspmv_kernel_box(BoxPlan B, MatView A, int32_t m, const T *__restrict__ X, T *__restrict__ Y) {
  box_rows<T, CW, ACC, FULL, K0, true, true>(B, A, m, X, [](int64_t, int32_t) {}, [&](int64_t i, int32_t c, const T (&y)[CW]) {
    store_cols_cs<T, CW, ACC>(Y + i * m + c, FULL ? CW : m - c, y);
  });
}

template <typename T, int CW, int ACC, bool FULL, int K0>
cudaError_t run_box(const ens_matrix *A, int m, const void *X, void *Y, cudaStream_t s) {
  using S = BoxShape<T, CW>;
  auto k = gspmv_kernel_box<T, CW, ACC, FULL, K0>;
  const size_t smem = S::smem(A->box.K);
  // Once per kernel instance and device, for the longest rows: the call costs a tenth of a small product's launch, and
  // a size by row length could be lowered by another thread before this one launches.
  static std::atomic<uint64_t> allowed{0};
  const uint64_t bit = A->device < 64 ? 1ull << A->device : 0;
  if (!(allowed.load(std::memory_order_acquire) & bit)) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem(kBoxMaxLen));
    if (e != cudaSuccess) return e;
    allowed.fetch_or(bit, std::memory_order_release);
  }
  static std::atomic<int> known[kBoxMaxLen + 1];  // by row length: the shared memory depends on it
  const int64_t full = (int64_t)A->num_sms * resident(known[A->box.K], (const void *)k, S::kThr, smem);
  k<<<(unsigned)(full < A->box.boxes ? full : (int64_t)A->box.boxes), S::kThr, smem, s>>>(A->box, view_of(A), m, (const T *)X, (T *)Y);
  return cudaGetLastError();
}
template <typename T, int CW, int ACC, bool FULL>
cudaError_t launch_box_acc(const ens_matrix *A, int m, const void *X, void *Y, cudaStream_t s) {
  // seven slots: the three-dimensional seven-point stencil
  return A->box.K == 7 ? run_box<T, CW, ACC, FULL, 7>(A, m, X, Y, s) : run_box<T, CW, ACC, FULL, 0>(A, m, X, Y, s);
}
// The widest access that every row of X and Y is aligned to, up to 32 bytes.
template <typename T, int CW>
cudaError_t launch_box_cw(const ens_matrix *A, int m, const void *X, void *Y, cudaStream_t s) {
  const uint64_t p = (uint64_t)(uintptr_t)X | (uint64_t)(uintptr_t)Y | (uint64_t)m * sizeof(T);
  constexpr int kWide = CW * sizeof(T) >= 32 ? 32 / sizeof(T) : CW;
  if (p % (kWide * sizeof(T)) == 0) {
    if constexpr (CW == 16)  // for m = 16 alone
      return launch_box_acc<T, CW, kWide, true>(A, m, X, Y, s);
    else
      return m % CW == 0 ? launch_box_acc<T, CW, kWide, true>(A, m, X, Y, s) : launch_box_acc<T, CW, kWide, false>(A, m, X, Y, s);
  }
  if constexpr (kWide * sizeof(T) == 32 && CW != 16)  // (sixteen columns aligned to 8 or 16 bytes go row by row: box_pays)
    if (p % 16 == 0) return launch_box_acc<T, CW, kWide / 2, false>(A, m, X, Y, s);
  return launch_box_acc<T, CW, 1, false>(A, m, X, Y, s);
}
int pow2_at_least(int v, int cap) {
  int p = 1;
  while (p < v && p < cap) p <<= 1;
  return p;
}

// Whether this product of a width that may take row boxes (use_box) is faster by them than row by row. It is wherever
// the row-by-row launch leaves lanes without columns; where its lanes are (nearly) full, boxes lose
//   * with rows that are not 32-byte aligned, whose X then comes in smaller pieces (128^3 channel: float64, rows aligned to
//     16 bytes, m = 16 284 us against 248, 32 567 against 481, 64 1140 against 903, but 20 0.76, 24 0.87 and 8 0.87 times;
//     float32, aligned to 8 bytes, m = 14 1.03 (rows of nine entries 0.83), 16 217 against 157, 24 345 against 295, but
//     12 0.91 and 20 0.90 times;
//     float32, aligned to 16, m = 16 1.03, 24 1.12);
//   * in float64 from m = 16 on where the rounds of boxes per resident block take 1.3 times the rows there are (bricks cut
//     off by the grid, a last round that is nearly empty; back to back 112640 rows in 440 boxes m = 16 1.12 times, 32 1.13,
//     64 1.14; 155648 rows in 1024 boxes 1.17, 1.21, 1.21; 221184 rows at 1.4 times 1.00; at 1.06 times 0.93-0.96). Below 400
//     row tiles the row-by-row launch's last round is as empty (92160 rows in 360 boxes 0.93, 0.95, 0.98): there only where
//     cut bricks alone make it 1.35 times (85140 rows in 495 boxes 1.15, 1.18, 1.21; 81807 in 400 0.92-0.96). Not asked where
//     the autotuner has timed both.
// float32, m = 14 on seven-point rows: 1.03 times on 2.1 million rows, 1.08 to 1.27 with cut bricks, else 0.9.
bool box_pays(const ens_matrix *A, int m, int dtype, const void *X, const void *Y) {
  const bool f32 = dtype == ENS_F32;
  const uint64_t p = (uint64_t)(uintptr_t)X | (uint64_t)(uintptr_t)Y | (uint64_t)m * (f32 ? 4 : 8);
  const int tile = pow2_at_least(m, 32);  // columns of a row-by-row tile
  const double full = (double)m / ((m + tile - 1) / tile * tile), rows = (double)A->n;
  const int64_t boxes = A->box.boxes;
  if (f32) {
    if (p % 32 == 0 || p % 8 != 0 || m < 14 || full < 0.75) return true;
    return m == 14 && (A->box.K != 7 || (A->n < (1 << 20) && boxes * kBoxRows <= 1.05 * rows));
  }
  if (m < 16 || m % 4 != 0 || full < 0.875) return true;
  if (p % 32 != 0 && p % 16 == 0) return false;
  const bool timed = m <= kTuneMaxM && A->tuned_lanes[0][m] > 0;
  if (timed || p % 16 != 0) return true;
  const int64_t round = A->num_sms * (int64_t)BoxShape<double, 8>::kBlocks, slots = (boxes + round - 1) / round * round;
  return slots * kBoxRows < 1.3 * rows || (A->n < 400 * kTileRows && boxes * kBoxRows < 1.35 * rows);
}

cudaError_t launch_box(const ens_matrix *A, int m, int dtype, const void *X, void *Y, cudaStream_t s) {
  if (dtype == ENS_F32) {
    if (m <= 4) return launch_box_cw<float, 4>(A, m, X, Y, s);
    return m == 16 ? launch_box_cw<float, 16>(A, m, X, Y, s) : launch_box_cw<float, 8>(A, m, X, Y, s);
  }
  return m <= 4 ? launch_box_cw<double, 4>(A, m, X, Y, s) : launch_box_cw<double, 8>(A, m, X, Y, s);
}

// A contiguous range of rows [r0, r1) of the product (r0 a multiple of kTileRows, so the shifted
// row-pointer array keeps its 16-byte alignment).
struct Rows {
  int64_t r0, r1;
};
static_assert(kPipeAlignRows % kTileRows == 0, "row chunks must be whole tiles");

int grid_for(const ens_matrix *A, int64_t rows, int per_sm, int64_t rows_per_block) {
  const int64_t need = (rows + rows_per_block - 1) / rows_per_block;
  const int64_t full = (int64_t)A->num_sms * per_sm;
  return (int)(need < full ? need : full);
}

template <typename Arith, int VEC, int LANES>
cudaError_t run(const ens_matrix *A, int m, const void *X, void *Y, uint32_t mask, const Rows &rows, cudaStream_t s,
                bool direct) {
  using T = typename Arith::T;
  MatView v = view_of(A);
  v.n = (int32_t)(rows.r1 - rows.r0);
  v.rp = A->row + rows.r0;
  T *y = (T *)Y + rows.r0 * m;
  constexpr bool capped = std::is_same<Arith, ArithF64Split>::value || std::is_same<Arith, ArithF32>::value;
  if constexpr (!std::is_same<Arith, ArithF64Hybrid>::value) {
    if (direct) {
      auto k = capped ? gspmv_kernel_direct<Arith, VEC, LANES> : gspmv_kernel_direct_free<Arith, VEC, LANES>;
      static std::atomic<int> known{0};
      k<<<grid_for(A, v.n, resident(known, (const void *)k, kThreads, 0), kThreads / LANES), kThreads, 0, s>>>(v, m, (const T *)X, y, mask);
      return cudaGetLastError();
    }
  }
  if constexpr (std::is_same<Arith, ArithF32>::value && LANES > 1 && (VEC == 2 || (VEC == 4 && LANES == 2)))
    if (tile_rows_for(v.n, LANES) == kTileRows) {
      auto k = gspmv_kernel_capped<Arith, VEC, LANES, kTileRows>;
      static std::atomic<int> known{0};
      k<<<grid_for(A, v.n, resident(known, (const void *)k, kThreads, 0), kTileRows), kThreads, 0, s>>>(v, m, (const T *)X, y, mask);
      return cudaGetLastError();
    }
  if constexpr (capped) {
    auto k = gspmv_kernel_capped<Arith, VEC, LANES>;
    static std::atomic<int> known{0};
    k<<<grid_for(A, v.n, resident(known, (const void *)k, kThreads, 0), tile_rows_for(v.n, LANES)), kThreads, 0, s>>>(v, m, (const T *)X, y, mask);
  } else {
    auto k = gspmv_kernel<Arith, VEC, LANES>;
    static std::atomic<int> known{0};
    k<<<grid_for(A, v.n, resident(known, (const void *)k, kThreads, 0), tile_rows_for(v.n, LANES)), kThreads, 0, s>>>(v, m, (const T *)X, y, mask);
  }
  return cudaGetLastError();
}

bool aligned(const void *p, size_t a) { return ((uintptr_t)p % a) == 0; }

// Dispatch on LANES, a power of two in [1, 32].
template <typename Arith, int VEC>
cudaError_t dispatch(const ens_matrix *A, int m, const void *X, void *Y, int lanes, uint32_t mask, const Rows &rows,
                     cudaStream_t s, bool direct = false) {
  switch (lanes) {
    case 1: return run<Arith, VEC, 1>(A, m, X, Y, mask, rows, s, direct);
    case 2: return run<Arith, VEC, 2>(A, m, X, Y, mask, rows, s, direct);
    case 4: return run<Arith, VEC, 4>(A, m, X, Y, mask, rows, s, direct);
    case 8: return run<Arith, VEC, 8>(A, m, X, Y, mask, rows, s, direct);
    case 16: return run<Arith, VEC, 16>(A, m, X, Y, mask, rows, s, direct);
    default: return run<Arith, VEC, 32>(A, m, X, Y, mask, rows, s, direct);
  }
}

}  // namespace

bool use_split(const ens_matrix *A) {
  return A->f64_mode != ENS_F64_NATIVE && A->split_ok && A->max_row_len <= kSplitMaxRow;
}

bool use_box(const ens_matrix *A, int m, int dtype) {
  // m <= 2 is at the memory's speed row by row. float32 blocks of 28 columns and more read a quarter of each line
  // per chunk (28: 441 us against 302 row by row, 32: 303 against 303); at 24 boxes still win (258 against 299).
  if (A->box.boxes == 0 || m < 3 || (dtype == ENS_F32 && m > 24)) return false;
  if (dtype != ENS_F32 && (A->f64_mode != ENS_F64_AUTO || A->native_share >= 0 || !use_split(A))) return false;
  if (A->untiled >= 0) return false;
  return m > kTuneMaxM || A->tuned_box[dtype == ENS_F32 ? 1 : 0][m];
}

// Share (in 32nds) of row sweeps given to native DFMA in split mode, by block width m: the FP64
// pipe is otherwise idle, so hybrid tiles add its throughput to that of the split path. A value
// set with ens_set_native_share overrides the table.
int native_share(const ens_matrix *A, int m) {
  if (A->f64_mode == ENS_F64_HYBRID) return kShareHybrid;
  if (A->native_share >= 0) return A->native_share;
  if (A->f64_mode == ENS_F64_SPLIT) return 0;
  if (m >= 1 && m <= kTuneMaxM && A->tuned_share[m] >= 0) return A->tuned_share[m];
  // Measured on GB300 (channel 256 x 128 x 128): native DFMA is fastest up to m = 2; at m = 4 nearly
  // all split (4/32: 180 us, against 195 us with 12/32); from m = 8 about 12/32 of the row sweeps
  // on the FP64 pipe and the rest split (m = 32: 928 us against 1077 us all split and 1695 us all
  // native).
  if (m <= 2) return 32;
  if (m < 8) return 4;
  return 12;
}

// Bit s set for about share/32 of the sweep indices s = 0..31, spread evenly.
uint32_t share_mask(int share) {
  uint32_t mask = 0;
  for (int s = 0; s < 32; ++s)
    if (((s + 1) * share) / 32 > (s * share) / 32) mask |= 1u << s;
  return mask;
}

namespace {

// Launch configuration of one product: VEC from m and alignment; lanes per row (rows per warp =
// 32 / lanes, column tile = VEC * lanes); share of native-DFMA sweeps (FP64 only).
struct Cfg {
  int vec, lanes, share;
  bool direct = false;  // untiled rows (direct_rows) instead of shared-memory tiles
};

// VEC and full-width lanes of a float64 launch with native share `share`: split-float products take
// four columns per lane when m allows (two packed float pairs share each nonzero's index and
// matrix pair; measured on GB300, channel 256 x 128 x 128, m = 8..32: 9-11 % faster than two),
// native DFMA and the column hybrid two.
void f64_shape(int m, int share, bool al16, int &vec, int &lanes) {
  if (share < 32 && m % 4 == 0 && al16) {
    vec = 4;
    lanes = pow2_at_least(m / 4, 8);
  } else if (m % 2 == 0 && al16) {
    vec = 2;
    lanes = pow2_at_least(m / 2, 16);
  } else {
    vec = 1;
    lanes = pow2_at_least(m, 32);
  }
}

Cfg default_cfg(const ens_matrix *A, int m, int dtype, const void *X, const void *Y) {
  Cfg c{};
  if (dtype == ENS_F32) {
    if (m % 4 == 0 && aligned(X, 16) && aligned(Y, 16)) {
      c.vec = 4;
      c.lanes = pow2_at_least(m / 4, 8);
    } else if (m % 2 == 0 && aligned(X, 8) && aligned(Y, 8)) {
      c.vec = 2;
      c.lanes = pow2_at_least(m / 2, 16);
    } else {
      c.vec = 1;
      c.lanes = pow2_at_least(m, 32);
    }
    c.share = 0;
  } else {
    c.share = use_split(A) ? native_share(A, m) : 32;
    f64_shape(m, c.share, aligned(X, 16) && aligned(Y, 16), c.vec, c.lanes);
  }
  if (m >= 1 && m <= kTuneMaxM) {
    const int tl = A->tuned_lanes[dtype == ENS_F32 ? 1 : 0][m];
    if (tl > 0 && tl <= c.lanes) c.lanes = tl;  // tuned for the same share, hence VEC (alignment permitting)
    c.direct = A->tuned_direct[dtype == ENS_F32 ? 1 : 0][m] == 1 && c.share != kShareHybrid;
  }
  if (A->untiled >= 0) c.direct = A->untiled == 1 && c.share != kShareHybrid;
  return c;
}

cudaError_t launch_cfg(const ens_matrix *A, int m, int dtype, const void *X, void *Y, const Cfg &c, const Rows &rows,
                       cudaStream_t s) {
  const bool d = c.direct;
  if (dtype == ENS_F32) {
    if (c.vec == 4) return dispatch<ArithF32, 4>(A, m, X, Y, c.lanes, 0u, rows, s, d);
    if (c.vec == 2) return dispatch<ArithF32, 2>(A, m, X, Y, c.lanes, 0u, rows, s, d);
    return dispatch<ArithF32, 1>(A, m, X, Y, c.lanes, 0u, rows, s, d);
  }
  if (c.share == kShareHybrid) {  // column hybrid needs two columns per lane
    return c.vec == 2 ? dispatch<ArithF64Hybrid, 2>(A, m, X, Y, c.lanes, 0u, rows, s)
                      : dispatch<ArithF64Native, 1>(A, m, X, Y, c.lanes, 0u, rows, s);
  }
  if (c.share < 32) {
    const uint32_t mask = share_mask(c.share);
    if (c.vec == 4) return dispatch<ArithF64Split, 4>(A, m, X, Y, c.lanes, mask, rows, s, d);
    return c.vec == 2 ? dispatch<ArithF64Split, 2>(A, m, X, Y, c.lanes, mask, rows, s, d)
                      : dispatch<ArithF64Split, 1>(A, m, X, Y, c.lanes, mask, rows, s, d);
  }
  return c.vec == 2 ? dispatch<ArithF64Native, 2>(A, m, X, Y, c.lanes, 0u, rows, s, d)
                    : dispatch<ArithF64Native, 1>(A, m, X, Y, c.lanes, 0u, rows, s, d);
}

// Deterministic N(0,1)-like fill of the tuning block (values in the split range, no zeros).
__global__ void k_tune_fill(int64_t count, double *x, float *x32) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x) {
    uint32_t h = (uint32_t)(e * 2654435761ull) ^ 0x9E3779B9u;
    h ^= h >> 15;
    h *= 0x2C1B3C6Du;
    h ^= h >> 12;
    const float v = 0.25f + (float)(h & 0xFFFFFF) * (1.0f / 16777216.0f);  // [0.25, 1.25)
    const float sgn = (h & 0x80000000u) ? -1.f : 1.f;
    if (x) x[e] = (double)(sgn * v);
    if (x32) x32[e] = sgn * v;
  }
}

}  // namespace

ens_status launch_gspmv(const ens_matrix *A, int m, int dtype, const void *X, void *Y, cudaStream_t s) {
  if (A->n == 0) return ENS_OK;
  cudaError_t e = use_box(A, m, dtype) && box_pays(A, m, dtype, X, Y) ? launch_box(A, m, dtype, X, Y, s)
                                       : launch_cfg(A, m, dtype, X, Y, default_cfg(A, m, dtype, X, Y), Rows{0, A->n}, s);
  if (e != cudaSuccess) return cuda_fail(e, "gspmv launch");
  return ENS_OK;
}

ens_status launch_gspmv_rows(const ens_matrix *A, int m, int dtype, const void *X, void *Y, int64_t r0, int64_t r1,
                             cudaStream_t s) {
  if (r1 <= r0) return ENS_OK;
  const Cfg c = default_cfg(A, m, dtype, X, Y);
  cudaError_t e = launch_cfg(A, m, dtype, X, Y, c, Rows{r0, r1}, s);
  if (e != cudaSuccess) return cuda_fail(e, "gspmv launch");
  return ENS_OK;
}

// Autotuner: time every candidate (FP64 arithmetic: native DFMA, split with native shares 0, 8, 12,
// 16, 24 and the column hybrid; for each, lanes per row giving the full, half and quarter column
// tile of its VEC) on this matrix for block width m with CUDA events, keep the fastest in the
// matrix's table.
ens_status autotune(ens_matrix *A, int m, int dtype, cudaStream_t s, int32_t *lanes_out, int32_t *share_out,
                    double *best_us_out) {
  const size_t count = (size_t)A->n * m, xcount = (size_t)A->ncols * m;  // Y rows, X rows (= n if square)
  void *X = nullptr, *Y = nullptr;
  const size_t es = dtype == ENS_F32 ? 4 : 8;
  cudaError_t e = cudaMallocAsync(&X, xcount * es, s);
  if (e == cudaSuccess) e = cudaMallocAsync(&Y, count * es, s);
  if (e == cudaSuccess) {
    const int grid = A->num_sms * 8;
    k_tune_fill<<<grid, 256, 0, s>>>((int64_t)xcount, dtype == ENS_F32 ? nullptr : (double *)X,
                                     dtype == ENS_F32 ? (float *)X : nullptr);
    e = cudaGetLastError();
  }
  // the defaults without any previous tuning
  const int di = dtype == ENS_F32 ? 1 : 0;
  const int keep_lanes = A->tuned_lanes[di][m], keep_share = A->tuned_share[m], keep_direct = A->tuned_direct[di][m];
  A->tuned_lanes[di][m] = -1;
  A->tuned_direct[di][m] = -1;
  if (dtype != ENS_F32) A->tuned_share[m] = -1;
  const Cfg base = default_cfg(A, m, dtype, X, Y);
  std::vector<Cfg> cand;
  auto add_widths = [&](int vec, int full, int share) {
    for (int div = 1; div <= 4 && full / div >= 1; div *= 2) {
      cand.push_back(Cfg{vec, full / div, share, false});
      if (share != kShareHybrid) cand.push_back(Cfg{vec, full / div, share, true});
    }
  };
  if (dtype == ENS_F32) {
    add_widths(base.vec, base.lanes, 0);
  } else {
    std::vector<int> shares{32};
    if (use_split(A)) shares.insert(shares.end(), {0, 8, 12, 16, 24, kShareHybrid});
    for (int sh : shares) {
      int vec = 1, full = 1;
      f64_shape(m, sh, true, vec, full);  // the tuning blocks are 256-byte aligned
      if (sh == kShareHybrid && vec != 2) continue;
      add_widths(vec, full, sh);
    }
  }
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&t0);
  if (e == cudaSuccess) e = cudaEventCreate(&t1);
  float best = 1e30f;
  Cfg bestc = base;
  for (const Cfg &c : cand) {
    if (e != cudaSuccess) break;
    for (int w = 0; w < 2 && e == cudaSuccess; ++w) e = launch_cfg(A, m, dtype, X, Y, c, Rows{0, A->n}, s);
    if (e == cudaSuccess) e = cudaEventRecord(t0, s);
    for (int r = 0; r < 5 && e == cudaSuccess; ++r) e = launch_cfg(A, m, dtype, X, Y, c, Rows{0, A->n}, s);
    if (e == cudaSuccess) e = cudaEventRecord(t1, s);
    if (e == cudaSuccess) e = cudaEventSynchronize(t1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, t0, t1);
    if (e == cudaSuccess && ms < best) {
      best = ms;
      bestc = c;
    }
  }
  // row boxes, where the matrix has them and the arithmetic is left to the library
  const bool keep_box = A->tuned_box[di][m];
  A->tuned_box[di][m] = true;
  bool box = false;
  if (e == cudaSuccess && use_box(A, m, dtype)) {
    for (int w = 0; w < 2 && e == cudaSuccess; ++w) e = launch_box(A, m, dtype, X, Y, s);
    if (e == cudaSuccess) e = cudaEventRecord(t0, s);
    for (int r = 0; r < 5 && e == cudaSuccess; ++r) e = launch_box(A, m, dtype, X, Y, s);
    if (e == cudaSuccess) e = cudaEventRecord(t1, s);
    if (e == cudaSuccess) e = cudaEventSynchronize(t1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, t0, t1);
    box = e == cudaSuccess && ms < best;
    if (box) best = ms;
  }
  A->tuned_box[di][m] = e == cudaSuccess ? box : keep_box;
  if (t0) cudaEventDestroy(t0);
  if (t1) cudaEventDestroy(t1);
  if (X) cudaFreeAsync(X, s);
  if (Y) cudaFreeAsync(Y, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    A->tuned_lanes[di][m] = keep_lanes;
    A->tuned_share[m] = keep_share;
    A->tuned_direct[di][m] = keep_direct;
    return cuda_fail(e, "autotune");
  }
  A->tuned_lanes[di][m] = bestc.lanes;
  A->tuned_direct[di][m] = bestc.direct ? 1 : 0;
  if (dtype != ENS_F32) A->tuned_share[m] = bestc.share;
  if (lanes_out) *lanes_out = bestc.lanes;
  if (share_out) *share_out = box ? 0 : bestc.share;
  if (best_us_out) *best_us_out = best * 1e3 / 5.0;
  return ENS_OK;
}

}  // namespace ens
