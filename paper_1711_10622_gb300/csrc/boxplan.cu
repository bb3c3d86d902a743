// Row boxes of a sparse matrix (see boxprod.cuh for the product that uses them): built on the host when
// the matrix is created, by several threads, and uploaded; the values are laid out on the device.
//
// A box is up to kBoxRows rows whose columns overlap as much as possible. For the stencils of grid
// operators these are bricks of grid cells, found from the matrix alone: `short_step` and `long_step` are
// the two commonest distances between a row and a later column (one line and one plane of the grid), and a
// brick starts at the first free row and follows, line by line, the actual columns nearest to those
// distances, so removed cells that shift the numbering do not matter. A box ends early when its columns
// would exceed kBoxCols. Any matrix gets a correct plan; it is kept only where the columns are read few
// enough times to pay (columns of all boxes <= 0.45 nnz) and the boxes are mostly full.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <memory>
#include <new>
#include <thread>
#include <unordered_map>
#include <vector>

#include "boxprod.cuh"
#include "ens_internal.cuh"

namespace ens {
namespace {

// The two commonest distances d = col - row > 1 over a sample of rows: the commonest, and the commonest of
// those at least twice as far or half as near. 0 where there is none.
void common_steps(int64_t n, const int32_t *rp, const int32_t *ci, int64_t &short_step, int64_t &long_step) {
  std::unordered_map<int64_t, int64_t> count;
  const int64_t samples = std::min<int64_t>(n, 4096);
  for (int64_t s = 0; s < samples; ++s) {
    const int64_t i = (int64_t)((uint64_t)s * 2654435761u % (uint64_t)n);  // not in step with the grid's lines
    for (int32_t j = rp[i]; j < rp[i + 1]; ++j)
      if ((int64_t)ci[j] - i > 1) ++count[(int64_t)ci[j] - i];
  }
  int64_t a = 0, na = 0, b = 0, nb = 0;
  for (auto &e : count)
    if (e.second > na || (e.second == na && e.first < a)) a = e.first, na = e.second;
  for (auto &e : count)
    if ((e.first >= 2 * a || 2 * e.first <= a) && (e.second > nb || (e.second == nb && e.first < b))) b = e.first, nb = e.second;
  if (nb * 8 < na) b = 0;
  short_step = b == 0 ? a : std::min(a, b);
  long_step = b == 0 ? 0 : std::max(a, b);
}

struct Part {  // boxes of one range of rows, in the layout of BoxPlan
  std::vector<int32_t> rows, cols;
  std::vector<uint16_t> loc;
  std::vector<int2> cnt;
  int64_t ucols = 0;
};

// Columns of the box that is being filled -> position in the order of their first entry, by open addressing; cleared
// by a new stamp.
struct ColumnSet {
  static constexpr int kSize = 4096;
  std::vector<int32_t> key, pos, stamp;
  int32_t now = 0;
  ColumnSet() : key(kSize), pos(kSize), stamp(kSize, 0) {}
  void clear() { ++now; }
  // Slot of c, or the free one where it goes.
  uint32_t slot(int32_t c) const {
    uint32_t at = ((uint32_t)c * 2654435761u) >> 20;
    while (stamp[at] == now && key[at] != c) at = (at + 1) & (kSize - 1);
    return at;
  }
};

void build_part(int64_t r0, int64_t r1, const int32_t *rp, const int32_t *ci, int32_t K, int64_t s1, int64_t s2, Part &P) {
  const int64_t n = r1 - r0;
  std::vector<uint8_t> used(n, 0);
  ColumnSet cs;
  const int lines = s2 ? kBoxLinesY : s1 ? kBoxLinesY * kBoxLinesZ : 1, planes = s2 ? kBoxLinesZ : 1;
  const int len = s1 ? kBoxLineX : kBoxRows;
  // the row in [r0, r1) that row i's columns name at about distance d, or -1
  auto step = [&](int64_t i, int64_t d) -> int64_t {
    int64_t best = -1, off = d / 2 + 1;
    for (int32_t j = rp[i]; j < rp[i + 1]; ++j) {
      const int64_t e = (int64_t)ci[j] - i, t = e > d ? e - d : d - e;
      if (e > 1 && t < off) off = t, best = ci[j];
    }
    return best < r1 ? best : -1;
  };
  auto from = [&](int64_t base, int64_t d) -> int64_t {  // the second row of a line decides: the first may wrap
    if (base + 1 < r1) {
      const int64_t t = step(base + 1, d);
      if (t > 0) return t - 1;
    }
    return step(base, d);
  };
  std::vector<int32_t> rows, cols, order, place;
  std::vector<uint16_t> pos;  // of every entry of the box's rows: its column's position in `cols`
  rows.reserve(kBoxRows);
  cols.reserve(kBoxCols);
  order.reserve(kBoxCols);
  place.reserve(kBoxCols);
  pos.reserve((size_t)kBoxRows * K);
  const size_t guess = (size_t)(n / 224 + 16);
  P.rows.reserve(guess * kBoxRows);
  P.cols.reserve(guess * kBoxCols);
  P.loc.reserve(guess * kBoxRows * K);
  int64_t next = r0;
  while (next < r1) {
    if (used[next - r0]) {
      ++next;
      continue;
    }
    rows.clear();
    cols.clear();
    pos.clear();
    cs.clear();
    // a row joins when the box has room for it and for its new columns; one that does not fit closes the box
    auto take = [&](int64_t i) -> bool {
      if ((int)rows.size() == kBoxRows) return false;
      const size_t ncols = cols.size(), nent = pos.size();
      for (int32_t j = rp[i]; j < rp[i + 1]; ++j) {
        const uint32_t at = cs.slot(ci[j]);
        if (cs.stamp[at] != cs.now) {
          if ((int)cols.size() == kBoxCols) {  // (the set still names this row's columns: nothing joins any more)
            cols.resize(ncols);
            pos.resize(nent);
            return false;
          }
          cs.stamp[at] = cs.now;
          cs.key[at] = ci[j];
          cs.pos[at] = (int32_t)cols.size();
          cols.push_back(ci[j]);
        }
        pos.push_back((uint16_t)cs.pos[at]);
      }
      rows.push_back((int32_t)i);
      used[i - r0] = 1;
      return true;
    };
    bool full = false;
    int64_t plane = next;
    for (int z = 0; z < planes && plane >= 0 && !full; ++z) {
      int64_t line = plane;
      for (int y = 0; y < lines && line >= 0 && !full; ++y) {
        for (int x = 0; x < len && line + x < r1 && !used[line + x - r0]; ++x)
          if (!take(line + x)) {
            full = true;
            break;
          }
        line = s1 ? from(line, s1) : -1;
        if (line >= 0 && (line < r0 || line >= r1)) line = -1;
      }
      plane = s2 ? from(plane, s2) : -1;
      if (plane >= 0 && (plane < r0 || plane >= r1)) plane = -1;
    }
    if (rows.empty()) {  // one row with more columns than a box holds: no plan
      P.ucols = INT64_MAX / 4;
      return;
    }
    // Columns in ascending order: neighbouring rows of the box then read neighbouring X rows, staged from
    // whole lines of memory and read from shared memory without bank conflicts.
    const int32_t nc = (int32_t)cols.size();
    order.resize(nc);
    place.resize(nc);
    for (int32_t k = 0; k < nc; ++k) order[k] = k;
    std::sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return cols[a] < cols[b]; });
    for (int32_t k = 0; k < nc; ++k) place[order[k]] = k;
    const size_t l0 = P.loc.size();
    P.loc.resize(l0 + (size_t)kBoxRows * K, (uint16_t)kBoxCols);  // missing entries: the row of zeros
    size_t e = 0;
    for (size_t r = 0; r < rows.size(); ++r)
      for (int32_t k = 0, len = rp[rows[r] + 1] - rp[rows[r]]; k < len; ++k) P.loc[l0 + (size_t)k * kBoxRows + r] = (uint16_t)place[pos[e++]];
    const size_t c0 = P.cols.size();
    P.cols.resize(c0 + kBoxCols, 0);
    for (int32_t k = 0; k < nc; ++k) P.cols[c0 + k] = cols[order[k]];
    P.cnt.push_back(make_int2((int32_t)rows.size(), nc));
    P.ucols += nc;
    rows.resize(kBoxRows, -1);
    P.rows.insert(P.rows.end(), rows.begin(), rows.end());
  }
}

// Values of every box slot from the CSR arrays (0 in the padding): split pairs and float32.
__global__ void k_box_values(int32_t boxes, int32_t K, const int32_t *__restrict__ brow, const int2 *__restrict__ bcnt,
                             const int32_t *__restrict__ rp, const double *__restrict__ va, float2 *__restrict__ bvs,
                             float *__restrict__ bv32) {
  const int64_t total = (int64_t)boxes * K * kBoxRows;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = (int32_t)(e % kBoxRows);
    const int64_t q = e / kBoxRows;
    const int32_t k = (int32_t)(q % K), b = (int32_t)(q / K);
    double v = 0.0;
    if (r < bcnt[b].x) {
      const int32_t i = brow[(int64_t)b * kBoxRows + r], j = rp[i] + k;
      if (j < rp[i + 1]) v = va[j];
    }
    const float hi = (float)v;
    bvs[e] = make_float2(hi, (float)(v - (double)hi));
    bv32[e] = hi;
  }
}

}  // namespace

struct HostBoxes {
  std::vector<Part> part;
  int64_t boxes = 0;
};

void free_plan(HostBoxes *h) { delete h; }

void free_box(BoxPlan &B) {
  cudaFree(B.shape);
  cudaFree(B.values);
  B = BoxPlan{};
}

namespace {

HostBoxes *plan(int64_t n, int64_t nnz, int32_t K, const int32_t *rp, const int32_t *ci) {
  if (n < kBoxMinRows || K < 1 || K > kBoxMaxLen || (double)nnz < 0.75 * (double)K * (double)n) return nullptr;
  int64_t s1 = 0, s2 = 0;
  common_steps(n, rp, ci, s1, s2);
  const int64_t per_min = 1 << 13;
  const int parts = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)std::max(1u, std::thread::hardware_concurrency()), 16, n / per_min}));
  std::unique_ptr<HostBoxes> h(new HostBoxes);
  h->part.resize(parts);
  // ranges end on whole bricks of planes where the planes are known
  const int64_t unit = s2 ? s2 * kBoxLinesZ : kBoxRows;
  auto bound = [&](int p) { return p == parts ? n : std::min(n, (n * p / parts + unit / 2) / unit * unit); };
  std::vector<uint8_t> failed(parts, 0);
  {
    std::vector<std::thread> th;
    auto work = [&](int p) {
      try {
        build_part(bound(p), bound(p + 1), rp, ci, K, s1, s2, h->part[p]);
      } catch (...) {
        failed[p] = 1;
      }
    };
    int started = 1;
    try {
      th.reserve(parts);
      for (; started < parts; ++started) th.emplace_back(work, started);
    } catch (...) {  // no more threads: the rest runs here
    }
    work(0);
    for (int p = started; p < parts; ++p) work(p);
    for (auto &t : th) t.join();
  }
  for (uint8_t f : failed)
    if (f) return nullptr;
  int64_t ucols = 0;
  for (auto &p : h->part) h->boxes += (int64_t)p.cnt.size(), ucols += p.ucols;
  if (ucols > (int64_t)(0.45 * (double)nnz) || h->boxes * kBoxRows > n + n / 4 * 3 + 64 * kBoxRows) return nullptr;
  return h.release();
}

}  // namespace

HostBoxes *plan_boxes(int64_t n, int64_t nnz, int32_t K, const int32_t *rp, const int32_t *ci) {
  try {
    return plan(n, nnz, K, rp, ci);
  } catch (...) {  // no memory for it
    return nullptr;
  }
}

cudaError_t upload_boxes(ens_matrix *A, const HostBoxes *h, const BoxPlan *shape, cudaStream_t s) {
  BoxPlan &B = A->box;
  cudaError_t e = cudaSuccess;
  if (shape) {
    B = *shape;
    B.shape = B.values = nullptr;  // the shape stays with its owner
  } else {
    B.boxes = (int32_t)h->boxes;
    B.K = A->max_row_len;
    const size_t boxes = (size_t)B.boxes, slots = boxes * B.K * kBoxRows;
    const size_t row = boxes * kBoxRows * sizeof(int32_t), col = boxes * kBoxCols * sizeof(int32_t), loc = slots * sizeof(uint16_t);
    char *p = nullptr;  // one block; every array's size is a multiple of 16 bytes
    e = cudaMalloc((void **)&p, row + col + loc + boxes * sizeof(int2));
    B.shape = p;
    B.row = (int32_t *)p;
    B.col = (int32_t *)(p + row);
    B.loc = (uint16_t *)(p + row + col);
    B.cnt = (int2 *)(p + row + col + loc);
    size_t at = 0;  // boxes of the parts before
    for (auto &part : h->part) {
      auto put = [&](auto *dst, const auto &src, size_t per_box) {
        if (e == cudaSuccess && !src.empty())
          e = cudaMemcpyAsync(dst + at * per_box, src.data(), src.size() * sizeof(src[0]), cudaMemcpyHostToDevice, s);
      };
      put(B.row, part.rows, kBoxRows);
      put(B.col, part.cols, kBoxCols);
      put(B.cnt, part.cnt, 1);
      put(B.loc, part.loc, (size_t)kBoxRows * B.K);
      at += part.cnt.size();
    }
  }
  if (e == cudaSuccess) {
    const size_t slots = (size_t)B.boxes * B.K * kBoxRows;
    char *p = nullptr;
    e = cudaMalloc((void **)&p, slots * (sizeof(float2) + sizeof(float)));
    B.values = p;
    B.vs = (float2 *)p;
    B.v32 = (float *)(p + slots * sizeof(float2));
  }
  if (e == cudaSuccess) {
    k_box_values<<<A->num_sms * 8, 256, 0, s>>>(B.boxes, B.K, B.row, B.cnt, A->row, A->val, B.vs, B.v32);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    cudaStreamSynchronize(s);  // copies from the plan in flight
    free_box(B);
  }
  if (e == cudaErrorMemoryAllocation) {  // the matrix works without boxes
    cudaGetLastError();
    e = cudaSuccess;
  }
  return e;
}

}  // namespace ens
