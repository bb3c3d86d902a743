// The projection step around the pressure solve for m flow states (Section 2.2, Eqs. eq2/eq3):
// the divergence of m staggered velocity fields (the Poisson right-hand sides) and the pressure-
// gradient correction u -= tau G p. Both are streaming passes over the fluid cells with the m
// states of a face contiguous in memory (row-interleaved), one thread per (cell, group of 1, 2 or 4
// states).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <new>
#include <vector>

#include "boxprod.cuh"
#include "ens_internal.cuh"
#include "ensemble_project.h"
#include "rowprod.cuh"

struct ens_grid {
  int32_t N[3] = {0, 0, 0};
  int32_t F[3] = {0, 0, 0};  // faces per direction in each velocity component array
  int32_t bc[3] = {0, 0, 0};
  int32_t n = 0;  // fluid cells (rows)
  int64_t ncell = 0;
  int64_t nfaces[3] = {0, 0, 0};
  bool all_fluid = true;
  int device = 0;
  int num_sms = 0;
  int32_t *cell_of_row = nullptr;  // [n] (NULL when every cell is fluid: row = cell)
  int32_t *row_of_cell = nullptr;  // [ncell] (-1: solid; NULL when every cell is fluid)
  uint8_t *open = nullptr;         // [n] bit 2d: low face along d open, bit 2d+1: high face open
  double *width[3] = {nullptr, nullptr, nullptr};     // [N_d] cell widths
  double *inv_dist[3] = {nullptr, nullptr, nullptr};  // [N_d + 1] per face position (see below)
  double *area[3] = {nullptr, nullptr, nullptr};      // face areas normal to d, indexed by the other two
                                                      // coordinates (lower one fastest)
  bool split_area = false;  // every area lies in the split-float product range [2^-40, 2^60)
};

namespace ens {
namespace {

// Kernel view of a grid. inv_dist[d][i] belongs to the faces at position i along d: 1 / (distance
// between the centres of cells i-1 and i) inside, across the wrap for i = 0 of a periodic
// direction, 2 / width of the boundary cell on a Dirichlet boundary face (p = 0 half a cell out).
struct GridView {
  int32_t N[3], F[3], bc[3];
  int32_t n;
  bool all_fluid;
  const int32_t *__restrict__ cell_of_row;
  const int32_t *__restrict__ row_of_cell;
  const uint8_t *__restrict__ open;
  const double *__restrict__ width[3];
  const double *__restrict__ inv_dist[3];
  const double *__restrict__ area[3];
};

GridView view_of(const ens_grid *G) {
  GridView v;
  for (int d = 0; d < 3; ++d) {
    v.N[d] = G->N[d];
    v.F[d] = G->F[d];
    v.bc[d] = G->bc[d];
    v.width[d] = G->width[d];
    v.area[d] = G->area[d];
    v.inv_dist[d] = G->inv_dist[d];
  }
  v.n = G->n;
  v.all_fluid = G->all_fluid;
  v.cell_of_row = G->cell_of_row;
  v.row_of_cell = G->row_of_cell;
  v.open = G->open;
  return v;
}

// VEC consecutive doubles (VEC = 1, 2 or 4; 16-byte aligned for 2 and 4).
template <int VEC>
__device__ __forceinline__ void ldv(const double *p, double (&v)[VEC]) {
  if constexpr (VEC == 1) {
    v[0] = __ldg(p);
  } else {
#pragma unroll
    for (int h = 0; h < VEC / 2; ++h) {
      const double2 t = __ldg(reinterpret_cast<const double2 *>(p) + h);
      v[2 * h] = t.x;
      v[2 * h + 1] = t.y;
    }
  }
}
template <int VEC>
__device__ __forceinline__ void ldv_rw(const double *p, double (&v)[VEC]) {
  if constexpr (VEC == 1) {
    v[0] = *p;
  } else {
#pragma unroll
    for (int h = 0; h < VEC / 2; ++h) {
      const double2 t = reinterpret_cast<const double2 *>(p)[h];
      v[2 * h] = t.x;
      v[2 * h + 1] = t.y;
    }
  }
}
template <int VEC>
__device__ __forceinline__ void stv(double *p, const double (&v)[VEC]) {
  if constexpr (VEC == 1) {
    *p = v[0];
  } else {
#pragma unroll
    for (int h = 0; h < VEC / 2; ++h) reinterpret_cast<double2 *>(p)[h] = make_double2(v[2 * h], v[2 * h + 1]);
  }
}

// Face array index of the face at position (c0, c1, c2) along d (c_d is the face number).
__device__ __forceinline__ int64_t face_at(const GridView &g, int d, int32_t c0, int32_t c1, int32_t c2) {
  const int32_t s0 = d == 0 ? g.F[0] : g.N[0];
  const int32_t s1 = d == 1 ? g.F[1] : g.N[1];
  return (int64_t)c0 + (int64_t)s0 * ((int64_t)c1 + (int64_t)s1 * c2);
}

// D[r*m + c + q] = scale * sum_d area_d (u_hi - u_lo) over the open faces of the row's cell.
template <int VEC>
__global__ void __launch_bounds__(kThreads)
    k_divergence(GridView g, int32_t m, double scale, const double *__restrict__ U, const double *__restrict__ V,
                 const double *__restrict__ W, double *__restrict__ D) {
  const int32_t groups = m / VEC;
  const int64_t total = (int64_t)g.n * groups;
  const double *comp[3] = {U, V, W};
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = (int32_t)(t / groups);
    const int32_t c = (int32_t)(t - (int64_t)r * groups) * VEC;
    const int32_t cell = g.all_fluid ? r : g.cell_of_row[r];
    const int32_t p[3] = {cell % g.N[0], (cell / g.N[0]) % g.N[1], cell / (g.N[0] * g.N[1])};
    const uint32_t op = g.open[r];
    // face areas of the cell (tables of the products of the other two widths)
    const double ar[3] = {g.area[0][p[1] + (int64_t)g.N[1] * p[2]], g.area[1][p[0] + (int64_t)g.N[0] * p[2]],
                          g.area[2][p[0] + (int64_t)g.N[0] * p[1]]};
    double acc[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double area = ar[d];
      int32_t lo[3] = {p[0], p[1], p[2]}, hi[3] = {p[0], p[1], p[2]};
      hi[d] = (g.bc[d] == ENS_BC_PERIODIC && p[d] + 1 == g.N[d]) ? 0 : p[d] + 1;
      if (op & (2u << (2 * d))) {
        double u[VEC];
        ldv<VEC>(comp[d] + face_at(g, d, hi[0], hi[1], hi[2]) * m + c, u);
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[q] = fma(area, u[q], acc[q]);
      }
      if (op & (1u << (2 * d))) {
        double u[VEC];
        ldv<VEC>(comp[d] + face_at(g, d, lo[0], lo[1], lo[2]) * m + c, u);
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[q] = fma(-area, u[q], acc[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] *= scale;
    stv<VEC>(D + (int64_t)r * m + c, acc);
  }
}

// The same divergence with split-float products (the GSpMV's arithmetic, rowprod.cuh): the FP64 pipe
// of GB300 is narrow, and the native form spends 7 FP64 operations per cell and state; here the six
// face products and their sum run on the FP32 pipe as packed pairs of states (split_acc2: each area and
// face value carried as hi + lo floats, the sum accumulated error-free), and each output costs one
// FP64 addition (the widening of hi + lo) and the scale multiply. A state whose face values leave the
// split range (zero among them) is recomputed with native DFMA. VEC = 2 or 4 states per thread.
template <int VEC>
__global__ void __launch_bounds__(kThreads, 4)
    k_divergence_split(GridView g, int32_t m, double scale, const double *__restrict__ U, const double *__restrict__ V,
                       const double *__restrict__ W, double *__restrict__ D) {
  constexpr int NP = VEC / 2;
  constexpr uint64_t kSign2 = 0x8000000080000000ull;
  const int32_t groups = m / VEC;
  const int64_t total = (int64_t)g.n * groups;
  const double *comp[3] = {U, V, W};
  const uint64_t g23 = f2_pack(__uint_as_float(kSplitG), __uint_as_float(kSplitG));
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = (int32_t)(t / groups);
    const int32_t c = (int32_t)(t - (int64_t)r * groups) * VEC;
    const int32_t cell = g.all_fluid ? r : g.cell_of_row[r];
    const int32_t p[3] = {cell % g.N[0], (cell / g.N[0]) % g.N[1], cell / (g.N[0] * g.N[1])};
    const uint32_t op = g.open[r];
    const double ar[3] = {g.area[0][p[1] + (int64_t)g.N[1] * p[2]], g.area[1][p[0] + (int64_t)g.N[0] * p[2]],
                          g.area[2][p[0] + (int64_t)g.N[0] * p[1]]};
    uint64_t sh[NP], sl[NP];
    uint32_t rng[VEC];
#pragma unroll
    for (int q = 0; q < NP; ++q) sh[q] = sl[q] = 0ull;
#pragma unroll
    for (int q = 0; q < VEC; ++q) rng[q] = 0u;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float ah, al;
      split_f64(ar[d], ah, al);
      const SplitPair a = split_pair(make_float2(ah, al));
      int32_t lo[3] = {p[0], p[1], p[2]}, hi[3] = {p[0], p[1], p[2]};
      hi[d] = (g.bc[d] == ENS_BC_PERIODIC && p[d] + 1 == g.N[d]) ? 0 : p[d] + 1;
      if (op & (2u << (2 * d))) {
        double u[VEC];
        ldv<VEC>(comp[d] + face_at(g, d, hi[0], hi[1], hi[2]) * m + c, u);
#pragma unroll
        for (int q = 0; q < NP; ++q) split_acc2(a, u[2 * q], u[2 * q + 1], g23, sh[q], sl[q], rng[2 * q], rng[2 * q + 1]);
      }
      if (op & (1u << (2 * d))) {
        double u[VEC];
        ldv<VEC>(comp[d] + face_at(g, d, lo[0], lo[1], lo[2]) * m + c, u);
        const SplitPair na{a.ah ^ kSign2, a.al ^ kSign2};  // -area, exactly
#pragma unroll
        for (int q = 0; q < NP; ++q) split_acc2(na, u[2 * q], u[2 * q + 1], g23, sh[q], sl[q], rng[2 * q], rng[2 * q + 1]);
      }
    }
    double y[VEC];
    bool all_ok = true, ok[VEC];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      float h0, h1, l0, l1;
      f2_unpack(sh[q], h0, h1);
      f2_unpack(sl[q], l0, l1);
      ok[2 * q] = split_ok(rng[2 * q], h0, l0);
      ok[2 * q + 1] = split_ok(rng[2 * q + 1], h1, l1);
      y[2 * q] = split_to_double(h0, l0);
      y[2 * q + 1] = split_to_double(h1, l1);
      all_ok &= ok[2 * q] && ok[2 * q + 1];
    }
    if (!all_ok) {  // native products for the states the split form cannot carry
      double acc[VEC];
#pragma unroll
      for (int q = 0; q < VEC; ++q) acc[q] = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        int32_t lo[3] = {p[0], p[1], p[2]}, hi[3] = {p[0], p[1], p[2]};
        hi[d] = (g.bc[d] == ENS_BC_PERIODIC && p[d] + 1 == g.N[d]) ? 0 : p[d] + 1;
        if (op & (2u << (2 * d))) {
          double u[VEC];
          ldv<VEC>(comp[d] + face_at(g, d, hi[0], hi[1], hi[2]) * m + c, u);
#pragma unroll
          for (int q = 0; q < VEC; ++q) acc[q] = fma(ar[d], u[q], acc[q]);
        }
        if (op & (1u << (2 * d))) {
          double u[VEC];
          ldv<VEC>(comp[d] + face_at(g, d, lo[0], lo[1], lo[2]) * m + c, u);
#pragma unroll
          for (int q = 0; q < VEC; ++q) acc[q] = fma(-ar[d], u[q], acc[q]);
        }
      }
#pragma unroll
      for (int q = 0; q < VEC; ++q) y[q] = ok[q] ? y[q] : acc[q];
    }
#pragma unroll
    for (int q = 0; q < VEC; ++q) y[q] *= scale;
    stv<VEC>(D + (int64_t)r * m + c, y);
  }
}

// u -= tau (p_hi - p_lo) inv_dist on the open faces. Each fluid cell owns its low face in every
// direction (the cell is that face's high side) and, in a Dirichlet direction, the high boundary
// face when it is the last cell; together these are all open faces, each written once.
template <int VEC>
__global__ void __launch_bounds__(kThreads)
    k_grad_correct(GridView g, int32_t m, double tau, const double *__restrict__ P, double *U, double *V, double *W) {
  const int32_t groups = m / VEC;
  const int64_t total = (int64_t)g.n * groups;
  double *comp[3] = {U, V, W};
  const int32_t stride[3] = {1, g.N[0], g.N[0] * g.N[1]};
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = (int32_t)(t / groups);
    const int32_t c = (int32_t)(t - (int64_t)r * groups) * VEC;
    const int32_t cell = g.all_fluid ? r : g.cell_of_row[r];
    const int32_t p[3] = {cell % g.N[0], (cell / g.N[0]) % g.N[1], cell / (g.N[0] * g.N[1])};
    const uint32_t op = g.open[r];
    double pc[VEC];
    ldv<VEC>(P + (int64_t)r * m + c, pc);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (op & (1u << (2 * d))) {  // low face open: a fluid neighbour or a Dirichlet boundary
        double pn[VEC];
        const bool boundary = p[d] == 0 && g.bc[d] != ENS_BC_PERIODIC;
        if (boundary) {
#pragma unroll
          for (int q = 0; q < VEC; ++q) pn[q] = 0.0;
        } else {
          const int32_t nb_cell = p[d] == 0 ? cell + (g.N[d] - 1) * stride[d] : cell - stride[d];
          const int32_t nb = g.all_fluid ? nb_cell : g.row_of_cell[nb_cell];
          ldv<VEC>(P + (int64_t)nb * m + c, pn);
        }
        const double coef = tau * g.inv_dist[d][p[d]];
        double *u = comp[d] + face_at(g, d, p[0], p[1], p[2]) * m + c;
        double v[VEC];
        ldv_rw<VEC>(u, v);
#pragma unroll
        for (int q = 0; q < VEC; ++q) v[q] = fma(-coef, pc[q] - pn[q], v[q]);
        stv<VEC>(u, v);
      }
      if (g.bc[d] == ENS_BC_DIRICHLET && p[d] == g.N[d] - 1 && (op & (2u << (2 * d)))) {
        const double coef = tau * g.inv_dist[d][g.N[d]];
        int32_t f[3] = {p[0], p[1], p[2]};
        f[d] = g.N[d];
        double *u = comp[d] + face_at(g, d, f[0], f[1], f[2]) * m + c;
        double v[VEC];
        ldv_rw<VEC>(u, v);
#pragma unroll
        for (int q = 0; q < VEC; ++q) v[q] = fma(-coef, 0.0 - pc[q], v[q]);
        stv<VEC>(u, v);
      }
    }
  }
}

// Grids without solid cells: the place of a thread is its cell x and states c on a line, and the lines y0 .. y1 of plane
// z that it takes; a cell costs no index divisions and which faces are open follows from the position. One block:
// up to 256 (x, states) pairs.
struct March {
  int32_t x, c, y0, y1, z;
  bool on;
};
template <int VEC, int MARCH>
__device__ __forceinline__ March march_place(const GridView &g, int32_t m) {
  const int32_t groups = m / VEC, width = g.N[0] * groups;
  const int32_t xb = (width + (int32_t)blockDim.x - 1) / (int32_t)blockDim.x, yc = (g.N[1] + MARCH - 1) / MARCH;
  const int32_t bx = blockIdx.x % xb, rest = blockIdx.x / xb;
  const int32_t e = bx * (int32_t)blockDim.x + (int32_t)threadIdx.x;
  March p;
  p.on = e < width;
  p.x = e / groups;
  p.c = (e - p.x * groups) * VEC;
  p.y0 = (rest % yc) * MARCH;
  p.y1 = min(p.y0 + MARCH, g.N[1]);
  p.z = rest / yc;
  return p;
}

// Four (VEC = 2: two) values as hi and lo floats; values outside the split range come out as NaN.
template <int VEC>
__device__ __forceinline__ void split_states(const double (&u)[VEC], float (&h)[VEC], float (&l)[VEC]) {
  const double x[4] = {u[0], u[1], u[VEC - 2], u[VEC - 1]};
  float4 a, b;
  box_split4(x, a, b);
  h[0] = a.x, h[1] = a.y, l[0] = b.x, l[1] = b.y;
  if constexpr (VEC == 4) h[2] = a.z, h[3] = a.w, l[2] = b.z, l[3] = b.w;
}

// The divergence with split-float products (box_acc2), marching along y: five face values are read and converted per
// cell, the sixth is the previous line's. Bound by issue (about 110 instructions per cell and state) and, beside it,
// HBM. Lines per thread on the 128^3 channel, m = 8: 1 181 us, 2 154, 4 137, 8 130. With two states per thread it spills
// 28 bytes at its 64 registers and is still 0.58-0.67 times k_divergence_split's time there (m = 2, 6, 10).
constexpr int kDivMarch = 8;
template <int VEC, int MARCH>
__global__ void __launch_bounds__(256, VEC == 4 ? 2 : 4)
    k_divergence_march(GridView g, int32_t m, double scale, const double *__restrict__ U, const double *__restrict__ V,
                       const double *__restrict__ W, double *__restrict__ D) {
  constexpr int NP = VEC / 2;
  constexpr uint64_t kSign2 = 0x8000000080000000ull;
  const March p = march_place<VEC, MARCH>(g, m);
  if (!p.on) return;
  const int32_t nx = g.N[0], ny = g.N[1], nz = g.N[2];
  const bool wx = g.bc[0] == ENS_BC_WALL, wy = g.bc[1] == ENS_BC_WALL, wz = g.bc[2] == ENS_BC_WALL;
  const bool lx = !(wx && p.x == 0), hx = !(wx && p.x == nx - 1), lz = !(wz && p.z == 0), hz = !(wz && p.z == nz - 1);
  const int32_t xh = g.bc[0] == ENS_BC_PERIODIC && p.x + 1 == nx ? 0 : p.x + 1, zh = g.bc[2] == ENS_BC_PERIODIC && p.z + 1 == nz ? 0 : p.z + 1;
  const double *pu = U + (p.x + (int64_t)g.F[0] * (p.y0 + (int64_t)ny * p.z)) * m + p.c;
  const double *pv = V + (p.x + (int64_t)nx * ((int64_t)g.F[1] * p.z)) * m + p.c;  // line 0
  const double *pw = W + (p.x + (int64_t)nx * (p.y0 + (int64_t)ny * p.z)) * m + p.c;
  double *pd = D + (p.x + (int64_t)nx * (p.y0 + (int64_t)ny * p.z)) * m + p.c;
  const int64_t du = (int64_t)(xh - p.x) * m, dw = (int64_t)(zh - p.z) * nx * ny * m, sv = (int64_t)nx * m, su = (int64_t)g.F[0] * m;
  const uint64_t zero = (uint64_t)(uint32_t)(m >> 31);
  const double ay = g.area[1][p.x + (int64_t)nx * p.z];
  float ayh, ayl;
  box_split(ay, ayh, ayl);
  const uint64_t YH = f2_pack(ayh, ayh), YL = f2_pack(ayl, ayl);
  float vh[VEC], vl[VEC];  // the low face of the current line
  const bool ly0 = !(wy && p.y0 == 0);
  if (ly0) {
    double v[VEC];
    ldv<VEC>(pv + p.y0 * sv, v);
    split_states<VEC>(v, vh, vl);
  }
  for (int32_t y = p.y0; y < p.y1; ++y, pu += su, pw += sv, pd += sv) {
    const bool ly = !(wy && y == 0), hy = !(wy && y == ny - 1);
    const int32_t yh = g.bc[1] == ENS_BC_PERIODIC && y + 1 == ny ? 0 : y + 1;
    const double ax = g.area[0][y + (int64_t)ny * p.z], az = g.area[2][p.x + (int64_t)nx * y];
    double u0[VEC], u1[VEC], v1[VEC], w0[VEC], w1[VEC];
    if (hx) ldv<VEC>(pu + du, u1);
    if (lx) ldv<VEC>(pu, u0);
    if (hy) ldv<VEC>(pv + yh * sv, v1);
    if (hz) ldv<VEC>(pw + dw, w1);
    if (lz) ldv<VEC>(pw, w0);
    uint64_t sh[NP], sl[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) sh[q] = sl[q] = 0ull;
    auto add = [&](uint64_t ah, uint64_t al, const float (&h)[VEC], const float (&l)[VEC]) {
#pragma unroll
      for (int q = 0; q < NP; ++q) box_acc2(ah, al, f2_pack(h[2 * q], h[2 * q + 1]), f2_pack(l[2 * q], l[2 * q + 1]), zero, sh[q], sl[q]);
    };
    float h[VEC], l[VEC], a0, a1;
    box_split(ax, a0, a1);
    uint64_t AH = f2_pack(a0, a0), AL = f2_pack(a1, a1);
    if (hx) {
      split_states<VEC>(u1, h, l);
      add(AH, AL, h, l);
    }
    if (lx) {
      split_states<VEC>(u0, h, l);
      add(AH ^ kSign2, AL ^ kSign2, h, l);
    }
    float nh[VEC], nl[VEC];
    if (hy) {
      split_states<VEC>(v1, nh, nl);
      add(YH, YL, nh, nl);
    }
    if (ly) add(YH ^ kSign2, YL ^ kSign2, vh, vl);
    box_split(az, a0, a1);
    AH = f2_pack(a0, a0), AL = f2_pack(a1, a1);
    if (hz) {
      split_states<VEC>(w1, h, l);
      add(AH, AL, h, l);
    }
    if (lz) {
      split_states<VEC>(w0, h, l);
      add(AH ^ kSign2, AL ^ kSign2, h, l);
    }
    float s[VEC], t[VEC];
    double out[VEC];
    uint32_t worst = 0u, least = 0xFFFFFFFFu;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      f2_unpack(sh[q], s[2 * q], s[2 * q + 1]);
      f2_unpack(sl[q], t[2 * q], t[2 * q + 1]);
    }
#pragma unroll
    for (int q = 0; q < VEC; ++q) {
      float sum = s[q];
      out[q] = box_add(sum, t[q]);
      worst = max(worst, max(box_sum_range(s[q]), box_sum_range(sum)));
      least = min(least, box_mantissa(sum));
    }
    if (worst >= kBoxSumWindow || least == 0u) {
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        if (split_finite(s[q]) && split_finite(t[q])) {
          out[q] = split_to_double(s[q], t[q]);
        } else {  // a face value outside the split range: native products for this state
          double acc = 0.0;
          if (hx) acc = fma(ax, __ldg(pu + du + q), acc);
          if (lx) acc = fma(-ax, __ldg(pu + q), acc);
          if (hy) acc = fma(ay, __ldg(pv + yh * sv + q), acc);
          if (ly) acc = fma(-ay, __ldg(pv + y * sv + q), acc);
          if (hz) acc = fma(az, __ldg(pw + dw + q), acc);
          if (lz) acc = fma(-az, __ldg(pw + q), acc);
          out[q] = acc;
        }
      }
    }
#pragma unroll
    for (int q = 0; q < VEC; ++q) {
      out[q] *= scale;
      vh[q] = nh[q];
      vl[q] = nl[q];
    }
    stv<VEC>(pd, out);
  }
}

// The correction, one line per block and four states per thread: a difference and an update per face and state, six FP64
// operations on a pipe of two per clock and SM, and 0.75 more for the coefficients (186 us for 128^3 cells, m = 8;
// measured 209, 220 with the index divisions of k_grad_correct). Slower: coefficients shared by the block (226: a
// barrier before the first load), marching along y as the divergence does (345: the next line's loads wait for
// this line's stores), one or two states per thread (128^3, m = 1 75 us, 2 115, 6 307, 7 426 against 60, 80, 224, 344
// of k_grad_correct, which takes these widths).
__global__ void __launch_bounds__(256)
    k_grad_correct_lines(GridView g, int32_t m, double tau, const double *__restrict__ P, double *U, double *V, double *W) {
  constexpr int VEC = 4;
  const March p = march_place<VEC, 1>(g, m);
  const int32_t nx = g.N[0], ny = g.N[1], nz = g.N[2], y = p.y0;
  if (!p.on) return;
  const bool lx = !(g.bc[0] == ENS_BC_WALL && p.x == 0), ly = !(g.bc[1] == ENS_BC_WALL && y == 0), lz = !(g.bc[2] == ENS_BC_WALL && p.z == 0);
  const bool zx = g.bc[0] == ENS_BC_DIRICHLET && p.x == 0, zy = g.bc[1] == ENS_BC_DIRICHLET && y == 0,
             zz = g.bc[2] == ENS_BC_DIRICHLET && p.z == 0;  // p = 0 beyond
  const double cx = tau * g.inv_dist[0][p.x], cy = tau * g.inv_dist[1][y], cz = tau * g.inv_dist[2][p.z];
  const int64_t sp = (int64_t)nx * m, line = (int64_t)ny * p.z + y;
  const double *pp = P + (p.x + nx * line) * m + p.c;
  double *pu = U + (p.x + g.F[0] * line) * m + p.c;
  double *pv = V + (p.x + nx * (y + (int64_t)g.F[1] * p.z)) * m + p.c;
  double *pw = W + (p.x + nx * line) * m + p.c;
  double pc[VEC], px[VEC], py[VEC], pz[VEC], u[VEC], v[VEC], w[VEC];
  ldv<VEC>(pp, pc);
  auto low = [&](bool has, int64_t off, double (&q)[VEC]) {
    if (has)
      ldv<VEC>(pp + off, q);
    else
#pragma unroll
      for (int k = 0; k < VEC; ++k) q[k] = 0.0;
  };
  low(lx && !zx, (int64_t)(p.x == 0 ? nx - 1 : -1) * m, px);
  low(ly && !zy, (y == 0 ? ny - 1 : -1) * sp, py);
  low(lz && !zz, (p.z == 0 ? nz - 1 : -1) * sp * ny, pz);
  if (lx) ldv_rw<VEC>(pu, u);
  if (ly) ldv_rw<VEC>(pv, v);
  if (lz) ldv_rw<VEC>(pw, w);
  auto update = [&](double *f, double coef, const double (&q)[VEC], double (&a)[VEC]) {
#pragma unroll
    for (int k = 0; k < VEC; ++k) a[k] = fma(-coef, pc[k] - q[k], a[k]);
    stv<VEC>(f, a);
  };
  if (lx) update(pu, cx, px, u);
  if (ly) update(pv, cy, py, v);
  if (lz) update(pw, cz, pz, w);
  auto edge = [&](double *f, double coef) {  // a Dirichlet boundary face on the high side
    double a[VEC];
    ldv_rw<VEC>(f, a);
#pragma unroll
    for (int k = 0; k < VEC; ++k) a[k] = fma(-coef, 0.0 - pc[k], a[k]);
    stv<VEC>(f, a);
  };
  if (g.bc[0] == ENS_BC_DIRICHLET && p.x == nx - 1) edge(pu + m, tau * g.inv_dist[0][nx]);
  if (g.bc[1] == ENS_BC_DIRICHLET && y == ny - 1) edge(pv + sp, tau * g.inv_dist[1][ny]);
  if (g.bc[2] == ENS_BC_DIRICHLET && p.z == nz - 1) edge(pw + sp * ny, tau * g.inv_dist[2][nz]);
}

// Threads and blocks of a marching launch over lines of MARCH (0 blocks: more than a grid dimension holds).
struct MarchLaunch {
  int threads;
  int64_t blocks;
};
template <int VEC, int MARCH>
MarchLaunch march_launch(const ens_grid *G, int m) {
  const int64_t width = (int64_t)G->N[0] * (m / VEC), xb = (width + 255) / 256;
  const int threads = (int)(((width + xb - 1) / xb + 31) / 32 * 32);
  const int64_t blocks = (width + threads - 1) / threads * ((G->N[1] + MARCH - 1) / MARCH) * G->N[2];
  return MarchLaunch{threads, width <= INT32_MAX && blocks <= INT32_MAX ? blocks : 0};
}
// Both return false (nothing launched) where the general kernel runs: a grid too large for one launch, or (the
// divergence) one whose lines of kDivMarch cells are too few for the chip. A thread's cells follow one another, so the
// launch pays only while its waves of resident threads (by the kernels' registers) are mostly full: against the general
// kernel, fill 0.14-0.47 with four states per thread 1.02-1.3 times its time (24^3 cells, m = 8 25 us against 20), 0.63
// 0.95-1.02, 0.71 0.95, 0.84 0.84, 0.96 0.81; with two states per thread 0.1-0.2 1.1-1.2, 0.3 0.96, 0.6 0.8.
template <int VEC>
bool divergence_march(const ens_grid *G, const GridView &g, int m, double scale, const double *U, const double *V, const double *W, double *D,
                      cudaStream_t s) {
  constexpr int64_t kRoom = VEC == 4 ? 512 : 1024;
  constexpr double kFill = VEC == 4 ? 0.65 : 0.3;
  const MarchLaunch l = march_launch<VEC, kDivMarch>(G, m);
  const int64_t wave = G->num_sms * (kRoom / l.threads), waves = (l.blocks + wave - 1) / wave;
  if ((double)l.blocks * l.threads < kFill * (double)(waves * G->num_sms * kRoom)) return false;
  if (l.blocks > 0) k_divergence_march<VEC, kDivMarch><<<(unsigned)l.blocks, l.threads, 0, s>>>(g, m, scale, U, V, W, D);
  return l.blocks > 0;
}
bool grad_correct_lines(const ens_grid *G, const GridView &g, int m, double tau, const double *P, double *U, double *V, double *W,
                        cudaStream_t s) {
  const MarchLaunch l = march_launch<4, 1>(G, m);
  if (l.blocks > 0) k_grad_correct_lines<<<(unsigned)l.blocks, l.threads, 0, s>>>(g, m, tau, P, U, V, W);
  return l.blocks > 0;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int grid_blocks(const ens_grid *G, int64_t work) {
  const int64_t want = (work + kThreads - 1) / kThreads;
  const int64_t cap = (int64_t)G->num_sms * 8;
  return (int)std::max<int64_t>(1, std::min(want, cap));
}

bool overlaps(const void *a, size_t na, const void *b, size_t nb) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return x < y + nb && y < x + na;
}

void free_grid(ens_grid *G) {
  if (!G) return;
  cudaFree(G->cell_of_row);
  cudaFree(G->row_of_cell);
  cudaFree(G->open);
  for (int d = 0; d < 3; ++d) {
    cudaFree(G->width[d]);
    cudaFree(G->inv_dist[d]);
    cudaFree(G->area[d]);
  }
  delete G;
}

template <typename T>
cudaError_t upload(T **dst, const std::vector<T> &src, cudaStream_t s) {
  cudaError_t e = cudaMalloc(reinterpret_cast<void **>(dst), src.size() * sizeof(T));
  if (e != cudaSuccess) return e;
  return cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, s);
}

}  // namespace
}  // namespace ens

using namespace ens;

static ens_status create_grid_impl(int32_t nx, int32_t ny, int32_t nz, const double *xn, const double *yn,
                                   const double *zn, const int32_t *bc, const uint8_t *solid, void *stream,
                                   ens_grid **out);

extern "C" ens_status ens_create_grid(int32_t nx, int32_t ny, int32_t nz, const double *xn, const double *yn,
                                      const double *zn, const int32_t *bc, const uint8_t *solid, void *stream,
                                      ens_grid **out) {
  clear_error();
  try {
    return create_grid_impl(nx, ny, nz, xn, yn, zn, bc, solid, stream, out);
  } catch (const std::bad_alloc &) {
    return fail(ENS_ERR_OOM, "create_grid: host allocation failed");
  }
}

static ens_status create_grid_impl(int32_t nx, int32_t ny, int32_t nz, const double *xn, const double *yn,
                                   const double *zn, const int32_t *bc, const uint8_t *solid, void *stream,
                                   ens_grid **out) {
  if (!out) return fail(ENS_ERR_INVALID, "create_grid: out is NULL");
  *out = nullptr;
  if (nx < 1 || ny < 1 || nz < 1) return fail(ENS_ERR_INVALID, "create_grid: dimensions must be >= 1");
  if (!xn || !yn || !zn || !bc) return fail(ENS_ERR_INVALID, "create_grid: NULL coordinates or boundary codes");
  const int32_t N[3] = {nx, ny, nz};
  const double *nodes[3] = {xn, yn, zn};
  const int64_t ncell = (int64_t)nx * ny * nz;
  if (ncell > INT32_MAX) return fail(ENS_ERR_INVALID, "create_grid: %lld cells exceed int32 indexing", (long long)ncell);
  for (int d = 0; d < 3; ++d) {
    if (bc[d] != ENS_BC_WALL && bc[d] != ENS_BC_PERIODIC && bc[d] != ENS_BC_DIRICHLET)
      return fail(ENS_ERR_INVALID, "create_grid: unknown boundary code %d in direction %d", bc[d], d);
    if (bc[d] == ENS_BC_PERIODIC && N[d] < 3)
      return fail(ENS_ERR_INVALID, "create_grid: periodic direction %d needs at least 3 cells", d);
    for (int32_t i = 0; i <= N[d]; ++i)
      if (!std::isfinite(nodes[d][i]) || (i > 0 && !(nodes[d][i] > nodes[d][i - 1])))
        return fail(ENS_ERR_INVALID, "create_grid: node coordinates of direction %d not finite and increasing", d);
  }
  // cell <-> row maps and open-face masks (host)
  std::vector<int32_t> row_of_cell(ncell);
  std::vector<int32_t> cell_of_row;
  cell_of_row.reserve(ncell);
  for (int64_t cidx = 0; cidx < ncell; ++cidx) {
    if (solid && solid[cidx]) {
      row_of_cell[cidx] = -1;
    } else {
      row_of_cell[cidx] = (int32_t)cell_of_row.size();
      cell_of_row.push_back((int32_t)cidx);
    }
  }
  const int32_t n = (int32_t)cell_of_row.size();
  if (n == 0) return fail(ENS_ERR_INVALID, "create_grid: every cell is solid");
  const int64_t stride[3] = {1, nx, (int64_t)nx * ny};
  std::vector<uint8_t> open(n);
  for (int32_t r = 0; r < n; ++r) {
    const int64_t cell = cell_of_row[r];
    const int64_t p[3] = {cell % nx, (cell / nx) % ny, cell / ((int64_t)nx * ny)};
    uint8_t bits = 0;
    for (int d = 0; d < 3; ++d) {
      // low side
      if (p[d] > 0) {
        if (row_of_cell[cell - stride[d]] >= 0) bits |= (uint8_t)(1u << (2 * d));
      } else if (bc[d] == ENS_BC_PERIODIC) {
        if (row_of_cell[cell + (N[d] - 1) * stride[d]] >= 0) bits |= (uint8_t)(1u << (2 * d));
      } else if (bc[d] == ENS_BC_DIRICHLET) {
        bits |= (uint8_t)(1u << (2 * d));
      }
      // high side
      if (p[d] < N[d] - 1) {
        if (row_of_cell[cell + stride[d]] >= 0) bits |= (uint8_t)(2u << (2 * d));
      } else if (bc[d] == ENS_BC_PERIODIC) {
        if (row_of_cell[cell - (N[d] - 1) * stride[d]] >= 0) bits |= (uint8_t)(2u << (2 * d));
      } else if (bc[d] == ENS_BC_DIRICHLET) {
        bits |= (uint8_t)(2u << (2 * d));
      }
    }
    open[r] = bits;
  }
  std::vector<double> width[3], inv_dist[3];
  for (int d = 0; d < 3; ++d) {
    const int32_t Nd = N[d];
    width[d].resize(Nd);
    std::vector<double> centre(Nd);
    for (int32_t i = 0; i < Nd; ++i) {
      width[d][i] = nodes[d][i + 1] - nodes[d][i];
      centre[i] = 0.5 * (nodes[d][i] + nodes[d][i + 1]);
    }
    inv_dist[d].assign(Nd + 1, 0.0);
    for (int32_t i = 1; i < Nd; ++i) inv_dist[d][i] = 1.0 / (centre[i] - centre[i - 1]);
    if (bc[d] == ENS_BC_PERIODIC) {
      const double L = nodes[d][Nd] - nodes[d][0];
      inv_dist[d][0] = 1.0 / (centre[0] + L - centre[Nd - 1]);
    } else if (bc[d] == ENS_BC_DIRICHLET) {
      inv_dist[d][0] = 2.0 / width[d][0];
      inv_dist[d][Nd] = 2.0 / width[d][Nd - 1];
    }
  }

  // area of the faces normal to d: the product of the cell widths in the other two directions
  // (ascending direction order), tabulated over those two coordinates
  std::vector<double> area[3];
  for (int d = 0; d < 3; ++d) {
    const int a = d == 0 ? 1 : 0, b = d == 2 ? 1 : 2;  // the other two directions, a < b
    area[d].resize((size_t)N[a] * N[b]);
    for (int32_t jb = 0; jb < N[b]; ++jb)
      for (int32_t ja = 0; ja < N[a]; ++ja) area[d][ja + (size_t)N[a] * jb] = width[a][ja] * width[b][jb];
  }

  bool split_area = true;
  for (int d = 0; d < 3; ++d)
    for (double a : area[d]) split_area = split_area && a >= 0x1p-40 && a < 0x1p60;

  ens_grid *G = new ens_grid();
  G->split_area = split_area;
  for (int d = 0; d < 3; ++d) {
    G->N[d] = N[d];
    G->bc[d] = bc[d];
    G->F[d] = bc[d] == ENS_BC_PERIODIC ? N[d] : N[d] + 1;
  }
  G->n = n;
  G->ncell = ncell;
  G->all_fluid = n == ncell;
  for (int d = 0; d < 3; ++d) {
    int64_t f = 1;
    for (int e = 0; e < 3; ++e) f *= e == d ? G->F[e] : G->N[e];
    G->nfaces[d] = f;
  }
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaGetDevice(&G->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&G->num_sms, cudaDevAttrMultiProcessorCount, G->device);
  if (e == cudaSuccess && !G->all_fluid) e = upload(&G->cell_of_row, cell_of_row, s);
  if (e == cudaSuccess && !G->all_fluid) e = upload(&G->row_of_cell, row_of_cell, s);
  if (e == cudaSuccess) e = upload(&G->open, open, s);
  for (int d = 0; d < 3 && e == cudaSuccess; ++d) {
    e = upload(&G->width[d], width[d], s);
    if (e == cudaSuccess) e = upload(&G->inv_dist[d], inv_dist[d], s);
    if (e == cudaSuccess) e = upload(&G->area[d], area[d], s);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    free_grid(G);
    return cuda_fail(e, "create_grid");
  }
  *out = G;
  return ENS_OK;
}

extern "C" ens_status ens_destroy_grid(ens_grid *G) {
  clear_error();
  if (!G) return ENS_OK;
  cudaError_t e = cudaDeviceSynchronize();
  free_grid(G);
  if (e != cudaSuccess) return cuda_fail(e, "destroy_grid");
  return ENS_OK;
}

extern "C" ens_status ens_grid_info(const ens_grid *G, int64_t *n_rows, int64_t n_faces[3]) {
  clear_error();
  if (!G) return fail(ENS_ERR_INVALID, "grid_info: grid is NULL");
  if (n_rows) *n_rows = G->n;
  if (n_faces)
    for (int d = 0; d < 3; ++d) n_faces[d] = G->nfaces[d];
  return ENS_OK;
}

namespace {
ens_status check_common(const ens_grid *G, int32_t m, const char *who) {
  if (!G) return fail(ENS_ERR_INVALID, "%s: grid is NULL", who);
  if (m < 1) return fail(ENS_ERR_INVALID, "%s: m must be >= 1 (got %d)", who, m);
  int dev = 0;
  ENS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != G->device) return fail(ENS_ERR_INVALID, "%s: current device %d is not the grid's device %d", who, dev, G->device);
  return ENS_OK;
}
}  // namespace

extern "C" ens_status ens_divergence(const ens_grid *G, int32_t m, double scale, const double *U, const double *V,
                                     const double *W, double *D, void *stream) {
  clear_error();
  ens_status st = check_common(G, m, "divergence");
  if (st != ENS_OK) return st;
  if (!U || !V || !W || !D) return fail(ENS_ERR_INVALID, "divergence: NULL array");
  if (!std::isfinite(scale)) return fail(ENS_ERR_INVALID, "divergence: scale is not finite");
  const size_t nd = (size_t)G->n * m * sizeof(double);
  const double *comp[3] = {U, V, W};
  for (int d = 0; d < 3; ++d)
    if (overlaps(D, nd, comp[d], (size_t)G->nfaces[d] * m * sizeof(double)))
      return fail(ENS_ERR_INVALID, "divergence: D overlaps a velocity component");
  // four or two states per thread when the rows allow 16-byte accesses: the per-cell work (coordinates,
  // open faces, areas) is shared by those states
  const bool al = aligned16(U) && aligned16(V) && aligned16(W) && aligned16(D);
  const int vec = al && m % 4 == 0 ? 4 : (al && m % 2 == 0 ? 2 : 1);
  const GridView g = view_of(G);
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t work = (int64_t)G->n * (m / vec);
  if (vec > 1 && G->all_fluid && G->split_area &&
      (vec == 4 ? divergence_march<4>(G, g, m, scale, U, V, W, D, s) : divergence_march<2>(G, g, m, scale, U, V, W, D, s))) {
    ENS_CUDA_TRY(cudaGetLastError());
    return ENS_OK;
  }
  // split-float products on the FP32 pipe for two or four states per thread (native for one)
  if (vec == 4 && G->split_area)
    k_divergence_split<4><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, scale, U, V, W, D);
  else if (vec == 2 && G->split_area)
    k_divergence_split<2><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, scale, U, V, W, D);
  else if (vec == 4)
    k_divergence<4><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, scale, U, V, W, D);
  else if (vec == 2)
    k_divergence<2><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, scale, U, V, W, D);
  else
    k_divergence<1><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, scale, U, V, W, D);
  ENS_CUDA_TRY(cudaGetLastError());
  return ENS_OK;
}

extern "C" ens_status ens_grad_correct(const ens_grid *G, int32_t m, double tau, const double *P, double *U, double *V,
                                       double *W, void *stream) {
  clear_error();
  ens_status st = check_common(G, m, "grad_correct");
  if (st != ENS_OK) return st;
  if (!P || !U || !V || !W) return fail(ENS_ERR_INVALID, "grad_correct: NULL array");
  if (!std::isfinite(tau)) return fail(ENS_ERR_INVALID, "grad_correct: tau is not finite");
  const size_t np = (size_t)G->n * m * sizeof(double);
  double *comp[3] = {U, V, W};
  for (int d = 0; d < 3; ++d) {
    const size_t nb = (size_t)G->nfaces[d] * m * sizeof(double);
    if (overlaps(P, np, comp[d], nb)) return fail(ENS_ERR_INVALID, "grad_correct: P overlaps a velocity component");
    for (int e = d + 1; e < 3; ++e)
      if (overlaps(comp[d], nb, comp[e], (size_t)G->nfaces[e] * m * sizeof(double)))
        return fail(ENS_ERR_INVALID, "grad_correct: velocity components overlap");
  }
  const bool al = aligned16(P) && aligned16(U) && aligned16(V) && aligned16(W);
  const int vec = al && m % 4 == 0 ? 4 : (al && m % 2 == 0 ? 2 : 1);
  const GridView g = view_of(G);
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t work = (int64_t)G->n * (m / vec);
  if (vec == 4 && G->all_fluid && grad_correct_lines(G, g, m, tau, P, U, V, W, s)) {
    ENS_CUDA_TRY(cudaGetLastError());
    return ENS_OK;
  }
  if (vec == 4)
    k_grad_correct<4><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, tau, P, U, V, W);
  else if (vec == 2)
    k_grad_correct<2><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, tau, P, U, V, W);
  else
    k_grad_correct<1><<<grid_blocks(G, work), kThreads, 0, s>>>(g, m, tau, P, U, V, W);
  ENS_CUDA_TRY(cudaGetLastError());
  return ENS_OK;
}
