// The small levels' part of a V-cycle as one dense matrix.
//
// From a zero iterate, Alg. 2 from level m down is a fixed linear map r^(m) -> u^(m): sweeps,
// transfers and the bottom solve are all linear.  On a level of a few thousand unknowns the map
// as a dense matrix is one matrix-vector product (k_bottom_split),
// where its seven launches a level, 3.3 us each, and its bottom solve take 25 us a level.  The
// matrix is the V-cycle applied to every unit vector, in FP64 (rounded to FP32 once for FP32
// cycles): k_dense_columns below, when a handle is set up or its cycle parameters change.
#pragma once

#include "kernels.cuh"

namespace ccm {
namespace dev {

constexpr int DENSE_MAXL = 8;        // levels above the bottom one
constexpr int DENSE_THREADS = 512;

struct DenseLevel {
  int nx, ny, pitch, n2, W, core;    // core: rows of an SMO-2 block's core
  const uint8_t* cls;
  const double* vol;
  const int32_t* cell;
  const int32_t* col;
  const double* val;
  const int32_t* blk;
  const int64_t* blk_off;
  const double* inv;
  long u[2], r, res;                 // offsets of its work arrays in a CTA's scratch
};

struct DenseArgs {
  int nlev, nu1, nu2;                // levels above the bottom
  DenseLevel L[DENSE_MAXL + 1];
  int nbot;
  const int32_t* bot_cell;
  const double* bot;                 // [column][bot_ld]
  int bot_ld;
  int n;                             // unknowns of the first level
  const int32_t* cell;
  Stencil<double> S;
  double* scratch;                   // zeroed, `stride` values a CTA
  long stride;
  int ld;                            // rows of a stored column (the rest stays 0)
  double* out64;                     // [column][ld], or null
  float* out32;
};

// One CTA a column at a time, its levels' arrays in global scratch (cached); the same steps as
// the V-cycle's kernels (block-Jacobi sweeps).
template <bool CROSS>
__global__ void __launch_bounds__(DENSE_THREADS) k_dense_columns(DenseArgs A) {
  double* w = A.scratch + (long)blockIdx.x * A.stride;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NW = DENSE_THREADS / 32;
  auto cells = [&](const DenseLevel& L, auto f) {      // a warp to a row of cells
    for (int j = warp; j < L.ny; j += NW)
      for (int i = lane; i < L.nx; i += 32) f(i, j, (long)(j + 2) * L.pitch + i + 2);
  };
  auto rows = [&](const DenseLevel& L, const double* u, double* out) {   // their residuals
    for (int q = tid; q < L.n2; q += DENSE_THREADS) {
      double acc = 0;
      for (int k = 0; k < L.W; ++k) acc += L.val[(long)k * L.n2 + q] * u[L.col[(long)k * L.n2 + q]];
      out[q] = w[L.r + L.cell[q]] - acc;
    }
  };
  auto sweep = [&](const DenseLevel& L, int b) {
    const double* u = w + L.u[b];
    double* v = w + L.u[1 - b];
    double* res = w + L.res;
    rows(L, u, res);
    cells(L, [&](int, int, long p) {
      if (L.cls[p] == 1) v[p] = u[p] + A.S.omega_d * (w[L.r + p] - stencil_apply<double, CROSS>(u, p, L.pitch, A.S));
    });
    __syncthreads();
    for (int q = tid; q < L.n2; q += DENSE_THREADS) {
      const int k = q / L.core;
      const int cs = L.blk[4 * k], nc = L.blk[4 * k + 1] - cs, es = L.blk[4 * k + 2], ne = L.blk[4 * k + 3] - es;
      const double* inv = L.inv + L.blk_off[k] + (q - cs);
      double acc = 0;
#pragma unroll 4
      for (int e = 0; e < ne; ++e) acc += inv[(long)e * nc] * res[es + e];
      const int p = L.cell[q];
      v[p] = u[p] + acc;
    }
    __syncthreads();
  };
  const DenseLevel& F = A.L[0];
  for (int c = blockIdx.x; c < A.n; c += gridDim.x) {
    for (int l = 0; l < A.nlev; ++l)
      cells(A.L[l], [&](int, int, long p) { w[A.L[l].u[0] + p] = 0.0; });
    cells(F, [&](int, int, long p) { w[F.r + p] = p == A.cell[c] ? 1.0 : 0.0; });
    __syncthreads();
    for (int l = 0; l < A.nlev; ++l) {
      const DenseLevel &L = A.L[l], &K = A.L[l + 1];
      for (int k = 0; k < A.nu1; ++k) sweep(L, k & 1);
      const double* u = w + L.u[A.nu1 & 1];
      double* t = w + L.u[1 - (A.nu1 & 1)];             // the residual, in the buffer that is free
      rows(L, u, w + L.res);
      cells(L, [&](int, int, long p) {
        if (L.cls[p] == 1) t[p] = w[L.r + p] - stencil_apply<double, CROSS>(u, p, L.pitch, A.S);
      });
      __syncthreads();
      for (int q = tid; q < L.n2; q += DENSE_THREADS) t[L.cell[q]] = w[L.res + q];
      __syncthreads();
      cells(K, [&](int I, int J, long p) {
        if (K.cls[p] == 0) return;
        const long f = (long)(2 * J + 2) * L.pitch + 2 * I + 2;
        double s = 0, sv = 0;
        for (int k = 0; k < 4; ++k) {
          const long q = f + (k >> 1) * L.pitch + (k & 1);
          if (L.cls[q] == 0) continue;
          s += L.vol[q] * t[q];
          sv += L.vol[q];
        }
        w[K.r + p] = sv > 0 ? 4 * s / sv : 0.0;
      });
      __syncthreads();
    }
    const DenseLevel& B = A.L[A.nlev];
    for (int k = tid; k < A.nbot; k += DENSE_THREADS) {
      double acc = 0;
#pragma unroll 4
      for (int q = 0; q < A.nbot; ++q) acc += A.bot[(long)q * A.bot_ld + k] * w[B.r + A.bot_cell[q]];
      w[B.u[0] + A.bot_cell[k]] = acc;
    }
    __syncthreads();
    for (int l = A.nlev - 1; l >= 0; --l) {
      const DenseLevel &L = A.L[l], &K = A.L[l + 1];
      const double* uc = w + K.u[l + 1 == A.nlev ? 0 : (A.nu1 + A.nu2) & 1];
      double* u = w + L.u[A.nu1 & 1];
      cells(L, [&](int i, int j, long p) {
        if (L.cls[p] == 1) u[p] += uc[(long)(j / 2 + 2) * K.pitch + i / 2 + 2];
      });
      __syncthreads();
      for (int k = 0; k < A.nu2; ++k) sweep(L, (A.nu1 + k) & 1);
    }
    const double* u = w + F.u[(A.nu1 + A.nu2) & 1];
    for (int k = tid; k < A.n; k += DENSE_THREADS) {
      const double v = u[A.cell[k]];
      if (A.out64) A.out64[(long)c * A.ld + k] = v;
      if (A.out32) A.out32[(long)c * A.ld + k] = (float)v;
    }
    __syncthreads();
  }
}

// The same product for several right-hand sides of a batch: the work split of k_bottom_split
// (clusters of BOTTOM_SPLIT CTAs over the columns of 32 rows), each matrix entry used for R
// right-hand sides.  One at a time a batch would read the matrix once per right-hand side.
template <typename T, int R>
__global__ void __launch_bounds__(256) k_bottom_multi(int n, int ld, int nb, const int32_t* __restrict__ cell,
                                                      const T* __restrict__ inv, const T* __restrict__ r,
                                                      T* __restrict__ u, long bs) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* rs = reinterpret_cast<T*>(smem_raw);               // [columns of this CTA][R]
  __shared__ T part[8][32][R + 1];
  const unsigned q = bottom_rank();
  const int rowblk = blockIdx.x / BOTTOM_SPLIT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int k = rowblk * 32 + lane, b0 = blockIdx.y * R, nr = min(R, nb - b0);
  const int c0 = (int)((long)n * q / BOTTOM_SPLIT), c1 = (int)((long)n * (q + 1) / BOTTOM_SPLIT);
  pdl_enter();
  for (int i = threadIdx.x; i < (c1 - c0) * R; i += 256) {
    const int b = i / (c1 - c0), c = i - b * (c1 - c0);
    rs[c * R + b] = b < nr ? r[(long)(b0 + b) * bs + cell[c0 + c]] : (T)0;
  }
  __syncthreads();
  T acc[R] = {};
  if (k < n)
#pragma unroll 4
    for (int c = c0 + warp; c < c1; c += 8) {
      const T a = inv[(long)c * ld + k];
#pragma unroll
      for (int b = 0; b < R; ++b) acc[b] += a * rs[(c - c0) * R + b];
    }
#pragma unroll
  for (int b = 0; b < R; ++b) part[warp][lane][b] = acc[b];
  __syncthreads();
  // the eight warps' sums into part[0], then the ranks' over the cluster in rank order
  for (int i = threadIdx.x; i < 32 * R; i += 256) {
    const int l = i / R, b = i - l * R;
    T s = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += part[w][l][b];
    part[0][l][b] = s;
  }
  bottom_cluster_sync();
  // rank q finishes the rows l with l % BOTTOM_SPLIT == q
  for (int i = threadIdx.x; i < (32 / BOTTOM_SPLIT) * R; i += 256) {
    const int l = (i / R) * BOTTOM_SPLIT + (int)q, b = i % R;
    const T s = bottom_sum(&part[0][l][b]);
    const int row = rowblk * 32 + l;
    if (row < n && b < nr) u[(long)(b0 + b) * bs + cell[row]] = s;
  }
  bottom_cluster_sync();
}

}  // namespace dev
}  // namespace ccm
