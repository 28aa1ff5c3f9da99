// The FP64 part of one outer iteration (eq. PoissonResidualForm): t = r_hat - (h^2 L) u_hat in
// FP64, max |t|, and in the mixed-precision solve the FP32 image of t as the next right-hand
// side of the FP32 V-cycles (where the last sweep does not do it, u_hat += e before).
//
// GB300 issues FP64 at 1/64 of the FP32 rate, so the regular stencil runs in integer form
// (fixed.cuh) on the TMA-staged tiles: 2 FP64 operations a cell are left (r_hat - L u_hat and
// its rounding to FP32) of 19.  The kernel serves every tolerance: its error anywhere in a tile is below
// the rounding of an FP64 sum at the tile's largest values.
#pragma once

#include "smooth.cuh"

namespace ccm {
namespace dev {

// dynamic shared memory of k_resid (offsets are multiples of 128 bytes)
struct ResidSmem {
  static constexpr uint32_t u_bytes = HY * HX * 8, r_bytes = JY * HX * 8, c_bytes = HY * CLX;
  static constexpr uint32_t r_off = u_bytes, c_off = r_off + r_bytes;
  static constexpr uint32_t tx = u_bytes + r_bytes + c_bytes, bytes = tx;
  static_assert(r_off % 128 == 0 && c_off % 128 == 0, "TMA destinations");
};

struct ResidArgs {
  const int32_t* tiles;      // the 64 x 32 tiles with a regular cell
  int nrow;                  // CTAs [0, nrow): the fitted rows, 256 each; the others a tile each
  int nx, pitch, n2, W;
  const int32_t* cell;
  const int32_t* col;
  const double* val;
  const double* u;
  const double* r;
  float* r32;                // or null: the norm alone
  unsigned long long* norm;
  Stencil<double> S;
  QStencil Q;
  int* err;
  long bs;                   // batch stride
};

// One launch over the regular cells' tiles and the fitted rows of the irregular cells.  A tile
// CTA stages u_hat (68 x 36 halo), r_hat (68 x 32) and the class bytes (80 x 36) by TMA.
template <bool CROSS>
__global__ void __launch_bounds__(256, 3) k_resid(const __grid_constant__ CUtensorMap tu,
                                                  const __grid_constant__ CUtensorMap tr,
                                                  const __grid_constant__ CUtensorMap tcls, ResidArgs A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ __align__(16) unsigned wmax[8];
  const int z = blockIdx.y;          // right-hand side of the batch
  unsigned long long m = 0;
  if ((int)blockIdx.x < A.nrow) {
    // t = r_hat - sum_k beta_k u_hat(col_k); the row's cell, columns and coefficients (static)
    // while the previous launch drains
    const int row = blockIdx.x * 256 + threadIdx.x;
    const int q = row < A.n2 ? A.cell[row] : 0;
    if (row < A.n2)
      for (int k = 0; k < A.W; ++k) {
        prefetch_l1(A.col + (long)k * A.n2 + row);
        prefetch_l1(A.val + (long)k * A.n2 + row);
      }
    pdl_enter();
    const double* u = A.u + (long)z * A.bs;
    if (row < A.n2) {
      double acc = 0.0;
#pragma unroll 15
      for (int k = 0; k < A.W; ++k) acc += A.val[(long)k * A.n2 + row] * u[A.col[(long)k * A.n2 + row]];
      const double t = A.r[(long)z * A.bs + q] - acc;
      if (A.r32) A.r32[(long)z * A.bs + q] = (float)t;
      m = abs_bits(t);
    }
  } else {
    double* ut = reinterpret_cast<double*>(smem_raw);
    const double* rt = reinterpret_cast<const double*>(smem_raw + ResidSmem::r_off);
    const uint8_t* ct = smem_raw + ResidSmem::c_off;
    // while the previous launch drains: the tile's origin, the copy barrier and the class
    // bytes (static), with the byte count of the whole copy
    const int t = blockIdx.x - A.nrow;
    const int cx0 = A.tiles[2 * t] * JX, cy0 = A.tiles[2 * t + 1] * JY;
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      mbar_expect_tx(&bar, ResidSmem::tx);
      tma_load_2d(smem_raw + ResidSmem::c_off, &tcls, &bar, cx0, cy0);
    }
    __syncthreads();
    pdl_enter();
    if (threadIdx.x == 0) {
      tma_load_3d(ut, &tu, &bar, cx0, cy0, z);
      tma_load_3d(smem_raw + ResidSmem::r_off, &tr, &bar, cx0, cy0 + 2, z);
    }
    const bool ok = __syncthreads_and(tile_wait(&bar, A.err));
    if (!ok) return;
    const int x0 = 2 * (threadIdx.x & 31), y0 = (threadIdx.x >> 5) * 4;
    const int i0 = cx0 + x0;
    float* r32 = A.r32 ? A.r32 + (long)z * A.bs : nullptr;
    tile_stencil64<CROSS, false>(ut, reinterpret_cast<long long*>(ut), wmax, x0, y0, i0 < A.nx, A.S, A.Q,
                                 [&](int kk, double s0, double s1) {
      const uint32_t c2 = *reinterpret_cast<const uint16_t*>(ct + (y0 + kk + 2) * CLX + x0 + 2);
      const double2 r2 = *reinterpret_cast<const double2*>(rt + (y0 + kk) * HX + x0 + 2);
      const double t0 = r2.x - s0, t1 = r2.y - s1;
      const bool g0 = (c2 & 0xffu) == 1u, g1 = (c2 >> 8) == 1u && i0 + 1 < A.nx;
      if (g0) m = max(m, abs_bits(t0));
      if (g1) m = max(m, abs_bits(t1));
      if (r32) {
        const long p = (long)(cy0 + y0 + kk + 2) * A.pitch + (i0 + 2);
        if (g0 && g1) {
          *reinterpret_cast<float2*>(r32 + p) = make_float2((float)t0, (float)t1);
        } else {
          if (g0) r32[p] = (float)t0;
          if (g1) r32[p + 1] = (float)t1;
        }
      }
    }, [] {});
  }
  // one atomic a CTA, and none where the norm is already larger (all of them hit one word)
  __shared__ unsigned long long wm[8];
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, wm[w]);
    if (m > *(volatile unsigned long long*)(A.norm + z)) atomicMax(A.norm + z, m);
  }
}

// u_hat += e on the non-empty cells of the 32 x 8 tiles that hold one
__global__ void k_axpy_tiles(const int32_t* __restrict__ tiles, const uint8_t* __restrict__ cls, int nx, int ny,
                             int pitch, const float* __restrict__ e, double* __restrict__ u, long bs) {
  // the cell and its class (static) while the previous launch drains
  const int i = tiles[2 * blockIdx.x] * TX + threadIdx.x;
  const int j = tiles[2 * blockIdx.x + 1] * TY + threadIdx.y;
  const long p = (long)(j + 2) * pitch + (i + 2);
  const bool on = i < nx && j < ny && cls[p] != 0;
  pdl_enter();
  e += blockIdx.y * bs;       // right-hand side blockIdx.y of the batch
  u += blockIdx.y * bs;
  if (on) u[p] += (double)e[p];
}

}  // namespace dev
}  // namespace ccm
