// Products by row boxes: Y = A X with the X rows that a box of matrix rows needs staged in shared memory
// once (boxplan.cu builds the boxes).
//
// What bounded the row-by-row products (rowprod.cuh) was the work around each nonzero, not HBM: every X
// value was fetched through L1 and, in split float64, converted from double to two floats once per nonzero
// that used it, seven times for a seven-point stencil: 21 thread instructions per float64 product and 9 per
// float32 product. A brick of 16 x 4 x 4 cells reads 544 distinct X rows for its 1792 nonzeros, so here each
// of them is fetched and converted once per box (2.1 times per X row instead of 7). One thread owns one row
// and all columns of a chunk, so a nonzero costs one 16-bit index, one value and conflict-free 16-byte shared
// loads for up to sixteen columns. The matrix is stored by slots (entry k of every row together, missing
// entries pointing at a row of zeros): no bounds, predicates or row pointers in the inner loop, and 10 bytes
// per nonzero instead of 12.
//
// The work is pipelined by hand. An item is a box and a chunk of columns. While a block computes one item from
// shared memory, the X rows of the next are on their way to registers, the next box's matrix entries to the other
// half of a shared-memory buffer (cp.async) and the column list of the box after that to registers. The other
// block of the SM covers the staging pass (conversion, two barriers) with its products.
//
// Measured on the 256 x 128 x 128 channel against the default row-by-row launch: float64 m = 3 112 us (296), 4 116
// (183), 5 210 (562), 8 196 (267), 12 408 (454), 16 450 (457), 24 590 (909), 32 871 (923); float32 m = 3 58 (153),
// 4 58 (77), 8 86 (129), 12 154 (173), 16 149 (179). What bounds m = 8 float64 now is issue: 16.6 thread instructions
// per product at 50 %, FP32 pipe 42 %, L1 / shared wavefronts 56 %. Wider blocks lose line efficiency: a chunk of
// eight columns touches half of each 128-byte line of a 128-byte row.
// Tried and slower: staging and computing in turn without prefetch (m = 8 313 us); X rows by cp.async into a raw
// buffer, four columns per thread and twice the warps (243); two staged buffers with one barrier (232-248);
// sixteen columns per chunk in 512-thread blocks (m = 32 856-931); columns in the order of the rows that read them
// instead of ascending (217: bank conflicts and split lines).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "rowprod.cuh"

namespace ens {

// 16 x 4 x 4 cells have 16*4*4 + 2*(4*4 + 16*4 + 16*4) = 544 columns; 32 more for irregular boxes.
constexpr int kBoxRows = 256, kBoxCols = 576, kBoxLineX = 16, kBoxLinesY = 4, kBoxLinesZ = 4;
constexpr int kBoxMaxLen = 16;       // longest row with a plan
constexpr int64_t kBoxMinRows = 65536;  // fewer than 256 boxes leave SMs idle

// X values of the split form: |x| in [2^-40, 2^88), as in split_range, or 0. Matrix values are at least 2^-40, so a
// product is at least 2^-80 and what is lost below the smallest normal float (2^-126) stays below 2^-46 of it.
constexpr uint32_t kBoxELo = kSplitELo, kBoxEHi = kSplitELo + 128u;  // biased exponents of 2^-40 and 2^88

// x -> hi + lo: hi = x rounded to 24 bits (half up on the 29 bits below), lo = the remainder rounded to 24
// bits: |x - hi - lo| <= 2^-49 |x|, a quarter of split_f64's truncation. The remainder is the low 29 bits as a
// signed number, one integer conversion (per distinct X value, not per product). x inside the window.
__device__ __forceinline__ void box_split(double x, float &hi, float &lo) {
  const uint32_t hw = (uint32_t)__double2hiint(x), lw = (uint32_t)__double2loint(x);
  const uint32_t t = split_hi_bits(hw, lw), rem = lw << 3;
  const float scale = __uint_as_float(t & 0xFF800000u) * 0x1p-55f;
  lo = __int2float_rn((int32_t)rem) * scale;
  hi = __uint_as_float(t + (rem >> 31));
}
// Below the window's width exactly for values inside it.
__device__ __forceinline__ uint32_t box_range(double x) { return (uint32_t)__double2hiint(x) * 2u - (kBoxELo << 21); }
constexpr uint32_t kBoxWindow = (kBoxEHi - kBoxELo) << 21;

// Four values at once; zeros stay zeros, and values outside the window poison the sums that use them
// (NaN), which are then recomputed natively.
__device__ __forceinline__ void box_split4(const double (&x)[4], float4 &hi, float4 &lo) {
  float h[4], l[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) box_split(x[q], h[q], l[q]);
  if (max(max(box_range(x[0]), box_range(x[1])), max(box_range(x[2]), box_range(x[3]))) >= kBoxWindow) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (box_range(x[q]) >= kBoxWindow) {
        h[q] = x[q] == 0.0 ? 0.f : __uint_as_float(0x7FC00000u);
        l[q] = 0.f;
      }
  }
  hi = make_float4(h[0], h[1], h[2], h[3]);
  lo = make_float4(l[0], l[1], l[2], l[3]);
}

// hi + lo as a double, with integer widening of both and one addition. A zero hi or lo would widen to 2^-127:
// harmless for lo beside a hi of at least 2^-70, so the caller sends smaller sums (and zeros, infinities and
// NaN) to split_to_double.
__device__ __forceinline__ double box_widen(float f) {
  const uint32_t b = __float_as_uint(f);
  return __hiloint2double((int32_t)(((uint32_t)((int32_t)b >> 3) & 0x8FFFFFFFu) + (896u << 20)), (int32_t)(b << 29));
}
__device__ __forceinline__ uint32_t box_sum_range(float hi) { return (__float_as_uint(hi) << 1) - (57u << 24); }
constexpr uint32_t kBoxSumWindow = (255u - 57u) << 24;  // |hi| in [2^-70, inf)

// (sh, sl) += (ah + al) (xh + xl) for a pair of columns: 10 packed operations. The rounded high product goes
// through TwoSum; its own rounding error comes with TwoSum's second error term in one FMA against the exact
// product, so neither a separate error FMA nor a negation is needed.
// The product is rounded as an FMA with `zero`, a zero the compiler cannot see: as mul.rn.f32x2 it was
// contracted with the addition that follows, and TwoSum of an unrounded product loses 2^-25 of it.
__device__ __forceinline__ void box_acc2(uint64_t ah, uint64_t al, uint64_t xh, uint64_t xl, uint64_t zero, uint64_t &sh, uint64_t &sl) {
  const uint64_t ph = f2_fma(ah, xh, zero);
  const uint64_t s = f2_add(sh, ph);
  const uint64_t nb = f2_sub(sh, s);
  const uint64_t t = f2_add(s, nb);
  uint64_t e = f2_add(f2_sub(sh, t), f2_fma(ah, xh, nb));
  e = f2_fma(ah, xl, e);
  e = f2_fma(al, xh, e);
  sl = f2_add(sl, e);
  sh = s;
}

// hi + lo as a double without the FP64 pipe: TwoSum makes |lo| at most half an ulp of hi, which in units of the
// double's last place is an integer below 2^29; it is added to the widened hi as an integer. Rounds like the FP64
// addition. Not for hi outside box_sum_range's window, and not for a power of two, where a negative lo would
// borrow from the exponent (box_mantissa 0): the caller sends those to split_to_double.
__device__ __forceinline__ double box_add(float &hi, float lo) {
  float s, e;
  two_sum(hi, lo, s, e);
  hi = s;
  const uint32_t b = __float_as_uint(s);
  // e / 2^(E - 52) with the sign of s, E the exponent of s
  const float scale = __uint_as_float((((52u + 254u) << 23) - (b & 0x7F800000u)) | (b & 0x80000000u));
  const int32_t r = __float2int_rn(e * scale);
  const int64_t w = __double_as_longlong(box_widen(s));
  return __longlong_as_double(w + (int64_t)r);
}
__device__ __forceinline__ uint32_t box_mantissa(float hi) { return __float_as_uint(hi) << 9; }

// N consecutive elements, of which those at column offsets below `left` exist (the others keep what they held);
// ACC elements per access, aligned to it: one 32-byte access for four doubles or eight floats. Volatile: these
// are prefetches, and the compiler would otherwise sink them to the first use of their values.
template <typename T, int N, int ACC>
__device__ __forceinline__ void load_cols(const T *p, int32_t left, T (&v)[N]) {
#pragma unroll
  for (int h = 0; h < N; h += ACC) {
    if (h < left) {
      if constexpr (sizeof(T) == 8 && ACC == 4)
        asm volatile("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v[h]), "=d"(v[h + 1]), "=d"(v[h + 2]), "=d"(v[h + 3]) : "l"(p + h));
      else if constexpr (sizeof(T) == 8 && ACC == 2)
        asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v[h]), "=d"(v[h + 1]) : "l"(p + h));
      else if constexpr (sizeof(T) == 8)
        asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v[h]) : "l"(p + h));
      else if constexpr (ACC == 8)
        asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(v[h]), "=f"(v[h + 1]), "=f"(v[h + 2]), "=f"(v[h + 3]), "=f"(v[h + 4]), "=f"(v[h + 5]), "=f"(v[h + 6]), "=f"(v[h + 7])
                     : "l"(p + h));
      else if constexpr (ACC == 4)
        asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[h]), "=f"(v[h + 1]), "=f"(v[h + 2]), "=f"(v[h + 3]) : "l"(p + h));
      else
        asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v[h]) : "l"(p + h));
    } else if constexpr (sizeof(T) == 8) {
      // never read; without these zeros the compiler's schedule of the float64 kernels is 6 % slower (m = 8: 207 us
      // against 196)
#pragma unroll
      for (int q = 0; q < ACC; ++q) v[h + q] = T(0);
    }
  }
}
// Streaming stores of the same shape.
template <typename T, int N, int ACC>
__device__ __forceinline__ void store_cols_cs(T *p, int32_t left, const T (&v)[N]) {
#pragma unroll
  for (int h = 0; h < N; h += ACC)
    if (h < left) {
      if constexpr (sizeof(T) == 8 && ACC == 4)
        asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p + h), "d"(v[h]), "d"(v[h + 1]), "d"(v[h + 2]), "d"(v[h + 3]) : "memory");
      else if constexpr (sizeof(T) == 8 && ACC == 2)
        asm volatile("st.global.cs.v2.f64 [%0], {%1, %2};" ::"l"(p + h), "d"(v[h]), "d"(v[h + 1]) : "memory");
      else if constexpr (sizeof(T) == 8)
        asm volatile("st.global.cs.f64 [%0], %1;" ::"l"(p + h), "d"(v[h]) : "memory");
      else if constexpr (ACC == 8)
        asm volatile("st.global.cs.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p + h), "f"(v[h]), "f"(v[h + 1]), "f"(v[h + 2]), "f"(v[h + 3]),
                     "f"(v[h + 4]), "f"(v[h + 5]), "f"(v[h + 6]), "f"(v[h + 7])
                     : "memory");
      else if constexpr (ACC == 4)
        asm volatile("st.global.cs.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p + h), "f"(v[h]), "f"(v[h + 1]), "f"(v[h + 2]), "f"(v[h + 3]) : "memory");
      else
        asm volatile("st.global.cs.f32 [%0], %1;" ::"l"(p + h), "f"(v[h]) : "memory");
    }
}

// A thread owns one row of a box and a chunk of CW columns (float64: 4 or 8; float32: 4, 8 or 16). kBlocks: resident blocks per SM the kernels are
// compiled for (the shared memory of seven-entry rows allows as many).
template <typename T, int CW>
struct BoxShape {
  static constexpr bool kF64 = sizeof(T) == 8;
  static constexpr int kThr = kBoxRows, kBlocks = kF64 ? (CW == 4 ? 3 : 2) : CW == 16 ? 2 : 4;
  // The staged X rows lie in planes of four columns (16 bytes per row; float64: hi planes, then lo planes), the
  // last row zeros; four extra rows per plane shift neighbouring planes by half the banks.
  static constexpr int kPlanes = CW / 4, kPlane = kBoxCols + 4;
  static constexpr size_t kXBytes = (size_t)kPlane * 16 * kPlanes * (kF64 ? 2 : 1);
  static constexpr size_t ent_bytes(int K) { return (size_t)kBoxRows * ((kF64 ? 10 : 6) * (size_t)K + 4); }
  static constexpr size_t smem(int K) { return kXBytes + 2 * ent_bytes(K); }
};

// Every row of the product, all of a chunk's columns in one thread: epi(row, first column, y). INNER: a block
// takes every chunk of its boxes in turn (matrix entries read once); otherwise one chunk, blockIdx.x modulo the
// chunks, so that a thread keeps its columns. ACC: elements per global access of X, to which its rows are
// aligned. FULL: m is a multiple of CW (checks of the last chunk cost 8-11 % where they are not needed). K0: slots
// per row where it is known at compile time (0: B.K). ADD64: a float64 sum is widened with one FP64 addition; else
// in integer arithmetic, which frees the FP64 pipe for an epilogue that needs it (the solver's Chebyshev step 235 ->
// 212 us on cubes 192 x 128 x 96, m = 8) but costs the plain product 5 %. (The solver's other kernels take the integer form
// too; it was not measured for each of them.) ahead(row, first column) runs before the
// products: the epilogue's own reads can be asked for there.
template <typename T, int CW, int ACC, bool FULL, int K0, bool INNER, bool ADD64, typename Pre, typename Epi>
__device__ __forceinline__ void box_rows(const BoxPlan &B, const MatView &A, int32_t m, const T *__restrict__ X, Pre &&ahead, Epi &&epi) {
  using S = BoxShape<T, CW>;
  constexpr bool kF64 = S::kF64;
  constexpr int NT = S::kThr, NP = S::kPlanes, PL = S::kPlane;
  constexpr int N = CW * sizeof(T) >= 32 ? 32 / sizeof(T) : CW;  // columns of one staged unit (32 bytes of X)
  constexpr int UPR = CW / N, SR = NT / UPR, U = (kBoxCols + SR - 1) / SR;
  using V = typename std::conditional<kF64, float2, float>::type;
  extern __shared__ __align__(16) unsigned char box_sm[];
  float4 *const sx = reinterpret_cast<float4 *>(box_sm);
  unsigned char *const ent = box_sm + S::kXBytes;
  const int32_t K = K0 ? K0 : B.K;
  const int32_t ent_bytes = kBoxRows * ((int32_t)(sizeof(V) + 2) * K + 4);
  const int32_t nch = (m + CW - 1) / CW;
  const int32_t unit = threadIdx.x % UPR, srow = threadIdx.x / UPR;
  const int32_t step = INNER ? (int32_t)gridDim.x : (int32_t)gridDim.x / nch;
  int32_t b = INNER ? (int32_t)blockIdx.x : (int32_t)blockIdx.x / nch, ch = INNER ? 0 : (int32_t)blockIdx.x % nch;
  if (b >= B.boxes) return;
  const uint64_t zero = (uint64_t)(uint32_t)(B.K >> 31);  // 0: B.K is positive
  if (threadIdx.x < NP * (kF64 ? 2 : 1)) sx[threadIdx.x * PL + kBoxCols] = make_float4(0.f, 0.f, 0.f, 0.f);

  // matrix entries of box bb into buffer w
  auto fetch_entries = [&](int32_t bb, int32_t w) {
    unsigned char *d = ent + w * ent_bytes;
    const char *va;
    if constexpr (kF64)
      va = reinterpret_cast<const char *>(B.vs) + (int64_t)bb * K * kBoxRows * 8;
    else
      va = reinterpret_cast<const char *>(B.v32) + (int64_t)bb * K * kBoxRows * 4;
    const char *lc = reinterpret_cast<const char *>(B.loc) + (int64_t)bb * K * kBoxRows * 2;
    for (int32_t t = threadIdx.x * 16; t < kBoxRows * K * (int32_t)sizeof(V); t += NT * 16) cp_async16(d + t, va + t);
    d += kBoxRows * K * (int32_t)sizeof(V);
    for (int32_t t = threadIdx.x * 16; t < kBoxRows * K * 2; t += NT * 16) cp_async16(d + t, lc + t);
    d += kBoxRows * K * 2;
    if (threadIdx.x < kBoxRows / 4) cp_async16(d + threadIdx.x * 16, B.row + (int64_t)bb * kBoxRows + threadIdx.x * 4);
    cp_async_commit();
  };
  int32_t at[U], at_next[U];  // X rows of this thread's staged units: of the item in flight, of the box after it
  auto fetch_columns = [&](int32_t bb, int32_t (&o)[U], int2 &cnt) {
    asm volatile("ld.global.nc.v2.s32 {%0, %1}, [%2];" : "=r"(cnt.x), "=r"(cnt.y) : "l"(B.cnt + bb));
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (srow + u * SR < kBoxCols)
        asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(o[u]) : "l"(B.col + (int64_t)bb * kBoxCols + srow + u * SR));
  };
  T x[U][N];
  auto fetch_x = [&](int32_t cc, int32_t ncols) {
    const int32_t c = cc * CW + unit * N;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (srow + u * SR < ncols && (FULL || c < m)) load_cols<T, N, ACC>(X + (int64_t)at[u] * m + c, m - c, x[u]);
  };

  int2 cnt, cnt_next = make_int2(0, 0);
  int32_t buf = 0;
  fetch_columns(b, at, cnt);
  fetch_entries(b, 0);
  if (b + step < B.boxes) fetch_columns(b + step, at_next, cnt_next);
  fetch_x(ch, cnt.y);
  for (;;) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (srow + u * SR < cnt.y && (FULL || ch * CW + unit * N < m)) {
        float4 *d = sx + srow + u * SR;
        if constexpr (kF64) {
          float4 h, l;
          if (!FULL)  // columns beyond the block repeat the first one: a value the conversion takes as it comes
#pragma unroll
            for (int q = 1; q < N; ++q)
              if (ch * CW + unit * N + q >= m) x[u][q] = x[u][0];
          box_split4(x[u], h, l);
          d[unit * PL] = h;
          d[(NP + unit) * PL] = l;
        } else {
#pragma unroll
          for (int p = 0; p < N / 4; ++p)
            d[(unit * (N / 4) + p) * PL] = make_float4(x[u][4 * p], x[u][4 * p + 1], x[u][4 * p + 2], x[u][4 * p + 3]);
        }
      }
    cp_async_wait_all();
    __syncthreads();
    // start the next item: the next chunk of this box, or the block's next box
    const bool same = INNER && ch + 1 < nch;
    const int32_t bn = same ? b : b + step, chn = same ? ch + 1 : INNER ? 0 : ch, bufn = same ? buf : buf ^ 1;
    const bool more = bn < B.boxes;
    int2 cn = cnt;
    if (more) {
      if (!same) {
        cn = cnt_next;
#pragma unroll
        for (int u = 0; u < U; ++u) at[u] = at_next[u];
        fetch_entries(bn, bufn);
        if (bn + step < B.boxes) fetch_columns(bn + step, at_next, cnt_next);
      }
      fetch_x(chn, cn.y);
    }
    const int32_t r = threadIdx.x, c = ch * CW;
    if (r < cnt.x) {
      const unsigned char *const en = ent + buf * ent_bytes;
      const V *const va = reinterpret_cast<const V *>(en) + r;
      const uint16_t *const loc = reinterpret_cast<const uint16_t *>(en + kBoxRows * K * sizeof(V)) + r;
      const int64_t i = reinterpret_cast<const int32_t *>(en + kBoxRows * K * (sizeof(V) + 2))[r];
      ahead(i, c);
      T y[CW];
      if constexpr (kF64) {
        uint64_t sh[2 * NP], sl[2 * NP];
#pragma unroll
        for (int p = 0; p < 2 * NP; ++p) sh[p] = sl[p] = 0ull;
        auto one = [&](int32_t k, auto planes) {
          const float4 *xr = sx + loc[k * kBoxRows];
          const float2 a = va[k * kBoxRows];
          const uint64_t ah = f2_pack(a.x, a.x), al = f2_pack(a.y, a.y);
#pragma unroll
          for (int p = 0; p < decltype(planes)::value; ++p) {
            const ulonglong2 xh = *reinterpret_cast<const ulonglong2 *>(xr + p * PL);
            const ulonglong2 xl = *reinterpret_cast<const ulonglong2 *>(xr + (NP + p) * PL);
            box_acc2(ah, al, xh.x, xl.x, zero, sh[2 * p], sl[2 * p]);
            box_acc2(ah, al, xh.y, xl.y, zero, sh[2 * p + 1], sl[2 * p + 1]);
          }
        };
        auto all = [&](auto planes) {
          if constexpr (K0 > 0) {
#pragma unroll
            for (int k = 0; k < K0; ++k) one(k, planes);
          } else {
            for (int32_t k = 0; k < K; ++k) one(k, planes);
          }
        };
        if (NP == 2 && !FULL && m - c <= 4)  // a last chunk of one plane
          all(std::integral_constant<int, 1>{});
        else
          all(std::integral_constant<int, NP>{});
        float h[CW], w[CW];
        uint32_t worst = 0u;
#pragma unroll
        for (int p = 0; p < 2 * NP; ++p) {
          f2_unpack(sh[p], h[2 * p], h[2 * p + 1]);
          f2_unpack(sl[p], w[2 * p], w[2 * p + 1]);
          if (FULL || c + 4 * (p / 2) < m) worst = max(worst, max(box_sum_range(h[2 * p]), box_sum_range(h[2 * p + 1])));
        }
        if constexpr (ADD64) {
#pragma unroll
          for (int q = 0; q < CW; ++q) y[q] = box_widen(h[q]) + box_widen(w[q]);
        } else {
          uint32_t least = 0xFFFFFFFFu;
          float g[CW];
#pragma unroll
          for (int q = 0; q < CW; ++q) {
            g[q] = h[q];
            y[q] = box_add(g[q], w[q]);
            least = min(least, box_mantissa(g[q]));
            worst = max(worst, box_sum_range(g[q]));
          }
          if (least == 0u) worst = kBoxSumWindow;
        }
        if (worst >= kBoxSumWindow) {
          // Tiny and zero sums; values outside the split range or sums beyond float: native DFMA, two columns at a time
          // (one by one, a block of small values took up to twice as long). The unrolling is the one that leaves the
          // split products' schedule alone: m = 6 148 us instead of 120 with two, m = 8 118 instead of 112 with four;
          // a function of its own, or four columns at a time, costs them 5 to 70 %.
          constexpr int kGathers = FULL ? 2 : 4;
          const int32_t j0 = __ldg(A.rp + i), j1 = __ldg(A.rp + i + 1);
#pragma unroll
          for (int u = 0; u < CW; u += 2) {
            const bool ok0 = split_finite(h[u]) && split_finite(w[u]), ok1 = split_finite(h[u + 1]) && split_finite(w[u + 1]);
            if (ok0) y[u] = split_to_double(h[u], w[u]);
            if (ok1) y[u + 1] = split_to_double(h[u + 1], w[u + 1]);
            if (!(ok0 && ok1) && (FULL || c + u < m)) {
              double z0 = 0.0, z1 = 0.0;
#pragma unroll kGathers
              for (int32_t j = j0; j < j1; ++j) {
                const double a = __ldg(A.val + j);
                const T *xr = X + (int64_t)__ldg(A.ci + j) * m + c + u;
                if constexpr (ACC >= 2) {
                  const double2 t = __ldg(reinterpret_cast<const double2 *>(xr));
                  z0 = fma(a, t.x, z0);
                  z1 = fma(a, t.y, z1);
                } else {
                  z0 = fma(a, __ldg(xr), z0);
                  if (FULL || c + u + 1 < m) z1 = fma(a, __ldg(xr + 1), z1);
                }
              }
              if (!ok0) y[u] = z0;
              if (!ok1) y[u + 1] = z1;
            }
          }
        }
      } else {
        uint64_t s[2 * NP];
#pragma unroll
        for (int p = 0; p < 2 * NP; ++p) s[p] = 0ull;
        auto one = [&](int32_t k) {
          const float4 *xr = sx + loc[k * kBoxRows];
          const float a = va[k * kBoxRows];
          const uint64_t aa = f2_pack(a, a);
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(xr + p * PL);
            s[2 * p] = f2_fma(aa, xv.x, s[2 * p]);
            s[2 * p + 1] = f2_fma(aa, xv.y, s[2 * p + 1]);
          }
        };
        if constexpr (K0 > 0) {
#pragma unroll
          for (int k = 0; k < K0; ++k) one(k);
        } else {
          for (int32_t k = 0; k < K; ++k) one(k);
        }
#pragma unroll
        for (int p = 0; p < 2 * NP; ++p) f2_unpack(s[p], y[2 * p], y[2 * p + 1]);
      }
      epi(i, c, y);
    }
    if (!more) break;
    __syncthreads();
    b = bn, ch = chn, buf = bufn, cnt = cn;
  }
}

}  // namespace ens
