// The operator and its transpose on whole arrays (ccm_apply, ccm_apply_T, ccm_level_apply).
//
// One launch covers the box's 64 x 32 tiles and, in CTAs ahead of them, the fitted rows (or the
// boundary part of the transpose), for all vectors (grid y).  The arrays are read and written
// in the caller's layout, with the empty cells masked by their class (their values are never
// used), so that nothing is packed into the padded layout and back: what is left is one read of
// the vector's active cells and one write of the whole result.  The regular stencil runs in
// integer form (fixed.cuh).
#pragma once

#include "smooth.cuh"

namespace ccm {
namespace dev {

// a cell array: value (i, j) of vector z at p[z batch + j stride + i]
template <typename P>
struct Grid {
  P p;
  long stride, batch;
};

struct ApplyArgs {
  Grid<const double*> u;
  Grid<double*> out;
  const uint8_t* cls;        // padded
  int nx, ny, pitch, tx;     // tx: tiles per row of the box
  int nrow;                  // CTAs [0, nrow): 256 fitted rows each
  int n2, W;
  const int32_t* cell;       // padded
  const int32_t* col;        // padded
  const double* val;
  const double* nb;
  const int32_t* seg;
  const double* g;           // forward: boundary data, or null
  double* og;                // transpose: N^T v, or null
  long nseg;
  double scale;              // 1 / h^2
  bool vec;                  // out rows start on 16 bytes
  bool uvec;                 // u rows start on 16 bytes
  const uint8_t* act;        // per 64 x 32 tile of the box: it holds a non-empty cell
  Stencil<double> S;
  QStencil Q;
};

// the offset of padded cell p in a cell array
__device__ __forceinline__ long cell_at(int p, int pitch, long stride) {
  const int j = (int)((unsigned)p / (unsigned)pitch), i = p - j * pitch;
  return (j - 2) * stride + (i - 2);
}

// two cells (i, j), (i + 1, j) of the result from their sums; c2: their classes
__device__ __forceinline__ void apply_put(const ApplyArgs& A, double* __restrict__ out, int i, int j, uint32_t c2, double s0,
                                          double s1) {
  if (j >= A.ny || i >= A.nx) return;
  // the fitted rows' cells are written by their own CTAs, or (transpose) by k_rows_T
  const bool g0 = (c2 & 0xffu) != 2u, g1 = (c2 >> 8) != 2u && i + 1 < A.nx;
  const double v0 = (c2 & 0xffu) ? A.scale * s0 : 0.0, v1 = (c2 >> 8) ? A.scale * s1 : 0.0;
  double* o = out + (long)j * A.out.stride + i;
  if (A.vec && g0 && g1) {
    *reinterpret_cast<double2*>(o) = make_double2(v0, v1);
  } else {
    if (g0) o[0] = v0;
    if (g1) o[1] = v1;
  }
}

// the classes of the pairs of rows 2 k, 2 k + 1 are the halves of c2[k]
__device__ __forceinline__ uint32_t pair_class(uint32_t ca, uint32_t cb, int kk) {
  return ((kk < 2 ? ca : cb) >> (16 * (kk & 1))) & 0xffffu;
}

// a thread's cells that the integer form does not serve well; a call, so that this rare path takes no
// registers from the common one
template <bool CROSS>
__device__ __noinline__ void apply_few(const ApplyArgs& A, const double* tile, const long long* ints, double* out, int cx0,
                                       int cy0, uint32_t ca, uint32_t cb) {
  const int x0 = 2 * (threadIdx.x & 31), y0 = (threadIdx.x >> 5) * 4;
  few_cells<CROSS>(tile, ints, x0, y0, A.S, A.Q, [&](int kk, int j) { return (pair_class(ca, cb, kk) >> (8 * j) & 0xffu) == 1u; },
                   [&](int kk, int j, double s) { out[(long)(cy0 + y0 + kk) * A.out.stride + cx0 + x0 + j] = A.scale * s; });
}

// out = L u + N g (TRANS: L^T v on the cells that no fitted row's stencil reaches, and N^T v).
// star 4096^2, 4.9 M of 16.8 M cells active, 39 MB read and 134 MB written (26 us at the copy rate):
// 68 to 71 us, by the values; without the look at the cells' sums 66 us (the quick test takes 1 us of
// the difference, the cells that fail it the rest); with the classes loaded first and cell by cell, so
// that a tile took two round trips and 10 loads a thread in place of 5, 85 us before that.
template <bool CROSS, bool TRANS>
__global__ void __launch_bounds__(256, 3) k_apply(const __grid_constant__ ApplyArgs A) {
  __shared__ __align__(16) double tile[HY * HX];
  __shared__ __align__(16) long long ints[HY * HX];
  __shared__ __align__(16) unsigned wmax[8];
  const int z = blockIdx.y;
  pdl_enter();
  const double* __restrict__ u = A.u.p + z * A.u.batch;
  double* __restrict__ out = TRANS && !A.out.p ? nullptr : A.out.p + z * A.out.batch;
  if ((int)blockIdx.x < A.nrow) {
    const int row = blockIdx.x * 256 + threadIdx.x;
    if (row >= A.n2) return;
    const int c = A.cell[row];
    if (TRANS) {
      const int sg = A.seg[row];
      if (sg >= 0) A.og[z * A.nseg + sg] = A.scale * A.nb[row] * u[cell_at(c, A.pitch, A.u.stride)];
      return;
    }
    double acc = 0.0;
#pragma unroll 15
    for (int k = 0; k < A.W; ++k)
      acc += A.val[(long)k * A.n2 + row] * u[cell_at(A.col[(long)k * A.n2 + row], A.pitch, A.u.stride)];
    if (A.g != nullptr && A.seg[row] >= 0) acc += A.nb[row] * A.g[z * A.nseg + A.seg[row]];
    out[cell_at(c, A.pitch, A.out.stride)] = A.scale * acc;
    return;
  }
  const int t = blockIdx.x - A.nrow;
  const int cx0 = (t % A.tx) * JX, cy0 = (t / A.tx) * JY;
  const int x0 = 2 * (threadIdx.x & 31), y0 = (threadIdx.x >> 5) * 4;
  const int i0 = cx0 + x0;
  if (!A.act[t]) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) apply_put(A, out, i0, cy0 + y0 + kk, 0u, 0.0, 0.0);
    return;
  }
  uint32_t c2[2] = {0, 0};      // the classes of two rows' pairs each
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const int j = cy0 + y0 + kk;
    if (i0 < A.nx && j < A.ny)
      c2[kk >> 1] |= (uint32_t)*reinterpret_cast<const uint16_t*>(A.cls + (long)(j + 2) * A.pitch + i0 + 2) << (16 * (kk & 1));
  }
  // the 68 x 36 tile with its halo, in pairs of cells; classes and values are loaded together (the
  // values of cells that do not count are dropped afterwards)
  const auto counts = [](uint32_t c) { return TRANS ? c == 1u : c != 0u; };
  constexpr int NP = HY * HX / 2;
  if (A.uvec) {
    constexpr int N = (NP + 255) / 256;
    double2 v[N];
    uint32_t c[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int idx = threadIdx.x + 256 * k, y = idx / (HX / 2), i = cx0 - 2 + 2 * (idx - y * (HX / 2)), j = cy0 - 2 + y;
      const bool in = idx < NP && (unsigned)i < (unsigned)A.nx && (unsigned)j < (unsigned)A.ny;
      c[k] = in ? *reinterpret_cast<const uint16_t*>(A.cls + (long)(j + 2) * A.pitch + i + 2) : 0u;
      v[k] = in ? *reinterpret_cast<const double2*>(u + j * A.u.stride + i) : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int idx = threadIdx.x + 256 * k;
      if (!counts(c[k] & 0xffu)) v[k].x = 0.0;
      if (!counts(c[k] >> 8)) v[k].y = 0.0;
      if (idx < NP) *reinterpret_cast<double2*>(tile + 2 * idx) = v[k];
    }
  } else {
#pragma unroll 5
    for (int idx = threadIdx.x; idx < HY * HX; idx += 256) {
      const int y = idx / HX, i = cx0 + idx - y * HX - 2, j = cy0 + y - 2;
      const bool in = (unsigned)i < (unsigned)A.nx && (unsigned)j < (unsigned)A.ny;
      const uint32_t c = in ? A.cls[(long)(j + 2) * A.pitch + i + 2] : 0u;
      tile[idx] = counts(c) ? u[j * A.u.stride + i] : 0.0;
    }
    __syncthreads();
  }
  // with pairs each thread reads back its own slots first (tile_stencil64's maximum): no barrier
  tile_stencil64<CROSS, true>(
      tile, ints, wmax, x0, y0, true, A.S, A.Q,
      [&](int kk, double s0, double s1) { apply_put(A, out, i0, cy0 + y0 + kk, pair_class(c2[0], c2[1], kk), s0, s1); },
      [&] { apply_few<CROSS>(A, tile, ints, out, cx0, cy0, c2[0], c2[1]); });
}

// L^T v at the cells that the fitted rows' stencils reach (every irregular cell is one): the regular
// cells' part, sum_d w_d v[c + d] over the regular c + d (the stencil is point-symmetric), and the
// fitted rows' by the transposed CSR (its entries' rows are given by their cells), scaled together,
// over what k_apply wrote there.  One thread per cell; its classes and row range, which no launch
// writes, before the wait.  (Adding the scaled fitted part to k_apply's scaled part instead rounds once
// more, an eighth more error; disk 1408^2, 4 vectors, whole call: 67.3 us that way, 70.0 this.)
struct RowsTArgs {
  int n;                     // cells
  const int32_t* ptr;
  const int32_t* cell;       // padded
  const int32_t* rcell;      // padded
  const double* val;
  const uint8_t* cls;        // padded
  int pitch;
  double scale;
  Grid<const double*> v;
  Grid<double*> out;
  Stencil<double> S;
};

template <bool CROSS>
__global__ void __launch_bounds__(128) k_rows_T(RowsTArgs A) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const bool on = k < A.n;
  const int c = on ? A.cell[k] : 2 * A.pitch + 2, e0 = on ? A.ptr[k] : 0, e1 = on ? A.ptr[k + 1] : 0;
  uint32_t reg = 0;          // bit 5 (dj + 2) + di + 2: a regular cell
#pragma unroll
  for (int dj = -2; dj <= 2; ++dj)
#pragma unroll
    for (int di = -2; di <= 2; ++di) {
      if (!CROSS && dj != 0 && di != 0) continue;
      reg |= (uint32_t)(A.cls[c + (long)dj * A.pitch + di] == 1) << (5 * (dj + 2) + di + 2);
    }
  pdl_enter();
  if (!on) return;
  const double* v = A.v.p + blockIdx.y * A.v.batch;
  const long p = cell_at(c, A.pitch, A.v.stride);
  double w[25], acc = 0, rows = 0;
#pragma unroll
  for (int t = 0; t < 25; ++t) w[t] = reg >> t & 1 ? v[p + (t / 5 - 2) * A.v.stride + t % 5 - 2] : 0.0;
#pragma unroll
  for (int t = 0; t < 25; ++t)
    if (CROSS || t / 5 == 2 || t % 5 == 2) acc += A.S.w[t] * w[t];
  for (int e = e0; e < e1; ++e) rows += A.val[e] * v[cell_at(A.rcell[e], A.pitch, A.v.stride)];
  A.out.p[blockIdx.y * A.out.batch + cell_at(c, A.pitch, A.out.stride)] = A.scale * (acc + rows);
}

}  // namespace dev
}  // namespace ccm
