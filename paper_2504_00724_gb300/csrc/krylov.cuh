// Krylov acceleration of the mixed-precision outer iteration: the correction e of one outer
// step, which plain iterative refinement takes as e = M r (M = inner_cycles FP32 V-cycles of
// Alg. 2 from a zero guess), is instead the GMRES(m) solution of L e = r with M as a right
// preconditioner: e = Z y with z_j = M v_j, the v_j an orthonormal basis of the Krylov space
// of L M built by classical Gram-Schmidt with one re-orthogonalisation, and y minimising
// || beta e_1 - H y ||_2 over the (m + 1) x m Hessenberg matrix H.  Everything inside the step
// is FP32 on level 0 (vectors, the operator, the preconditioner) with FP64 dot products; the
// FP64 residual r_hat - L u_hat around it is unchanged, so the refinement still converges to
// the FP64 solution (GMRES-based iterative refinement).
//
// Vectors are padded level-0 arrays; only non-empty cells are ever written, so empty cells
// stay zero and the reductions may run over whole 32 x 8 tiles.  Every reduction is one launch:
// per-CTA partial sums in FP64, which the CTA that finishes last adds in a fixed order, so the
// results do not depend on scheduling; it also takes the step that the sum is for (a separate
// one-CTA launch for that cost 4 us each, seven a step of GMRES(2)).  Nothing here synchronises
// with the host: the scalars (Gram-Schmidt coefficients, H, y) stay in device memory and the
// step is captured into the outer iteration's graph.
//
// The vector kernels are bound by the latency of their loads, not by the few MB they move: a
// thread takes two adjacent cells of KRY_AHEAD tiles a step.  The reductions keep two CTAs an SM
// all the same: their FP64 sums cost a thread 64 clocks of its scheduler's FP64 pipe each.
#pragma once

#include "kernels.cuh"

namespace ccm {
namespace dev {

constexpr int KRY_MAXM = 8;          // largest GMRES restart length
constexpr int KRY_GRID = 304;        // most CTAs of a reduction (2 per SM), and of
constexpr int KRY_GRID_V = 1216;     // the other vector kernels
constexpr int KRY_THREADS = 256;     // two 32 x 8 tiles per CTA, two cells a thread
constexpr int KRY_TILES = 2;
constexpr int KRY_AHEAD = 4;         // tiles whose loads a thread of a reduction has in flight

struct KryVecs {
  const float* v[KRY_MAXM + 1];
};

// scalars of one GMRES step (device memory)
struct KryScalars {
  double part[(KRY_MAXM + 1) * KRY_GRID];   // per-CTA partial sums [vector][cta]
  double c[KRY_MAXM + 1];                   // coefficients of the last reduction
  double H[(KRY_MAXM + 1) * KRY_MAXM];      // Hessenberg matrix, column-major, leading dim m + 1
  double beta;                              // || r ||_2 at the start of the step
  double y[KRY_MAXM];                       // least-squares solution
  unsigned ticket;                          // CTAs of the running reduction that have finished
};

// FP32 arithmetic throughout: GB300 issues FP64 at 1/64 of the FP32 rate, so only the per-thread
// sums of the reductions leave FP32, compensated (Neumaier) until then.
struct Comp {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x;
    c += fabsf(s) >= fabsf(x) ? (s - t) + x : (x - t) + s;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// the two cells of this thread in tile t: p the first one's padded index (even); false beyond
// the grid (a second cell beyond it lies on the zero ring)
__device__ __forceinline__ bool kcell(const int32_t* __restrict__ tiles, int t, int nx, int ny, int pitch, long& p) {
  const int q = threadIdx.x & 127;
  const int ci = tiles[2 * t] * TX + 2 * (q & 15), cj = tiles[2 * t + 1] * TY + (q >> 4);
  p = (long)(cj + 2) * pitch + (ci + 2);
  return ci < nx && cj < ny;
}
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
// a pair to its non-empty cells (c: their class bytes)
__device__ __forceinline__ void st2(float* p, float2 v, uint32_t c) {
  if ((c & 0xffu) && (c >> 8)) *reinterpret_cast<float2*>(p) = v;
  else if (c & 0xffu) p[0] = v.x;
  else if (c >> 8) p[1] = v.y;
}
__device__ __forceinline__ uint32_t cls2(const uint8_t* cls, long p) { return *reinterpret_cast<const uint16_t*>(cls + p); }

// y = argmin || beta e_1 - H y ||_2 by Givens rotations (one thread; m <= KRY_MAXM).  A zero
// subdiagonal (the Krylov space became invariant) ends the basis there.
__device__ __noinline__ void klsq(int m, KryScalars* S) {
  double R[KRY_MAXM + 1][KRY_MAXM];
  double g[KRY_MAXM + 1];
  for (int jj = 0; jj < m; ++jj)
    for (int ii = 0; ii <= m; ++ii) R[ii][jj] = S->H[jj * (m + 1) + ii];
  for (int ii = 0; ii <= m; ++ii) g[ii] = 0.0;
  g[0] = S->beta;
  int k = m;
  for (int jj = 0; jj < m; ++jj) {
    const double a = R[jj][jj], b = R[jj + 1][jj];
    const double r = hypot(a, b);
    if (r == 0.0) {
      k = jj;
      break;
    }
    const double cs = a / r, sn = b / r;
    for (int q = jj; q < m; ++q) {
      const double x = R[jj][q], yv = R[jj + 1][q];
      R[jj][q] = cs * x + sn * yv;
      R[jj + 1][q] = -sn * x + cs * yv;
    }
    const double gx = g[jj], gy = g[jj + 1];
    g[jj] = cs * gx + sn * gy;
    g[jj + 1] = -sn * gx + cs * gy;
    if (b == 0.0) {        // invariant subspace: the columns after jj add nothing
      k = jj + 1;
      break;
    }
  }
  for (int q = m - 1; q >= 0; --q) {
    if (q >= k) {
      S->y[q] = 0.0;
      continue;
    }
    double a = g[q];
    for (int t = q + 1; t < k; ++t) a -= R[q][t] * S->y[t];
    S->y[q] = a / R[q][q];
  }
}

// What a reduction is for:
//   mode 0 (Gram-Schmidt pass of column j): c[i] = s_i, H[i][j] += s_i (= s_i with fresh);
//   mode 1 (new basis vector of column j):  H[j + 1][j] = sqrt(s_0), c[0] = 1 / that (0 if 0), and
//                                           after the last column (j = m - 1) the least squares;
//   mode 2 (start of the step):             beta = sqrt(s_0), c[0] = 1 / beta (0 if 0)
struct KryStep {
  int mode, j, m, fresh;
};

// the grid's sums of acc[0 .. n) and the step they are for: partial sums into part[i][cta], the
// last CTA adds them over the CTAs in a fixed order
__device__ __forceinline__ void kreduce(const Comp (&acc)[KRY_MAXM + 1], int n, KryStep T, KryScalars* __restrict__ S) {
  __shared__ double red[KRY_MAXM + 1][KRY_THREADS / 32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i <= KRY_MAXM; ++i) {
    if (i >= n) break;
    double a = acc[i].value();
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) red[i][warp] = a;
  }
  __syncthreads();
  if (threadIdx.x < n) {
    double a = 0.0;
    for (int k = 0; k < KRY_THREADS / 32; ++k) a += red[threadIdx.x][k];
    __stcg(&S->part[threadIdx.x * KRY_GRID + blockIdx.x], a);
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(&S->ticket, 1u) == gridDim.x - 1;
    if (last) {
      S->ticket = 0;
      __threadfence();
    }
  }
  __syncthreads();
  if (!last) return;
  // a warp to a sum: the partials of CTAs lane, lane + 32, ... then the lanes
  for (int i = warp; i < n; i += KRY_THREADS / 32) {
    double a = 0.0;
#pragma unroll 4
    for (int k = lane; k < gridDim.x; k += 32) a += __ldcg(&S->part[i * KRY_GRID + k]);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) {
      if (T.mode == 0) {
        S->c[i] = a;
        double* h = &S->H[T.j * (T.m + 1) + i];
        *h = T.fresh ? a : *h + a;
      } else {
        const double nrm = sqrt(fmax(a, 0.0));
        if (T.mode == 1) S->H[T.j * (T.m + 1) + T.j + 1] = nrm;
        else S->beta = nrm;
        S->c[0] = nrm > 0.0 ? 1.0 / nrm : 0.0;
      }
    }
  }
  if (T.mode == 1 && T.j == T.m - 1 && threadIdx.x == 0) klsq(T.m, S);   // (n = 1: warp 0 wrote H)
}

// w . v_i (i < n) over the grid
__global__ void __launch_bounds__(KRY_THREADS) k_kdot(const int32_t* __restrict__ tiles, int ntiles, int nx, int ny,
                                                      int pitch, const float* __restrict__ w, KryVecs V, int n,
                                                      KryStep T, KryScalars* __restrict__ S) {
  pdl_enter();
  Comp acc[KRY_MAXM + 1];
  const int step = KRY_TILES * gridDim.x;
  for (int t = KRY_TILES * blockIdx.x + (threadIdx.x >> 7); t < ntiles; t += KRY_AHEAD * step) {
    long p[KRY_AHEAD];
    float2 wv[KRY_AHEAD];
#pragma unroll
    for (int k = 0; k < KRY_AHEAD; ++k) {
      p[k] = 0;                                            // (0: the zero ring)
      if (t + k * step < ntiles && !kcell(tiles, t + k * step, nx, ny, pitch, p[k])) p[k] = 0;
    }
#pragma unroll
    for (int k = 0; k < KRY_AHEAD; ++k) wv[k] = ld2(w + p[k]);
#pragma unroll
    for (int i = 0; i <= KRY_MAXM; ++i)
      if (i < n) {
        float2 v[KRY_AHEAD];
#pragma unroll
        for (int k = 0; k < KRY_AHEAD; ++k) v[k] = ld2(V.v[i] + p[k]);
#pragma unroll
        for (int k = 0; k < KRY_AHEAD; ++k) {
          acc[i].add(wv[k].x * v[k].x);
          acc[i].add(wv[k].y * v[k].y);
        }
      }
  }
  kreduce(acc, n, T, S);
}

// w -= sum_{i < n} c[i] v_i on the non-empty cells, then the dot products of the new w with v_0 ..
// v_{n-1} (self = false) or with itself (self = true)
__global__ void __launch_bounds__(KRY_THREADS) k_ksubdot(const int32_t* __restrict__ tiles, int ntiles, int nx, int ny,
                                                         int pitch, const uint8_t* __restrict__ cls,
                                                         float* __restrict__ w, KryVecs V, int n, bool self,
                                                         KryStep T, KryScalars* __restrict__ S) {
  pdl_enter();
  float c[KRY_MAXM + 1];
#pragma unroll
  for (int i = 0; i <= KRY_MAXM; ++i) c[i] = i < n ? (float)S->c[i] : 0.f;
  Comp acc[KRY_MAXM + 1];
  const int step = KRY_TILES * gridDim.x;
  for (int t = KRY_TILES * blockIdx.x + (threadIdx.x >> 7); t < ntiles; t += KRY_AHEAD * step) {
    long p[KRY_AHEAD];
    float2 a[KRY_AHEAD];
    uint32_t cc[KRY_AHEAD];
#pragma unroll
    for (int k = 0; k < KRY_AHEAD; ++k) {
      p[k] = 0;                                            // (0: the zero ring, class 0)
      if (t + k * step < ntiles && !kcell(tiles, t + k * step, nx, ny, pitch, p[k])) p[k] = 0;
    }
#pragma unroll
    for (int k = 0; k < KRY_AHEAD; ++k) {
      a[k] = ld2(w + p[k]);
      cc[k] = cls2(cls, p[k]);
    }
#pragma unroll
    for (int i = 0; i <= KRY_MAXM; ++i)
      if (i < n) {
        float2 v[KRY_AHEAD];
#pragma unroll
        for (int k = 0; k < KRY_AHEAD; ++k) v[k] = ld2(V.v[i] + p[k]);
#pragma unroll
        for (int k = 0; k < KRY_AHEAD; ++k) {
          a[k].x = fmaf(-c[i], v[k].x, a[k].x);
          a[k].y = fmaf(-c[i], v[k].y, a[k].y);
        }
      }
#pragma unroll
    for (int k = 0; k < KRY_AHEAD; ++k) st2(w + p[k], a[k], cc[k]);
    if (self) {
#pragma unroll
      for (int k = 0; k < KRY_AHEAD; ++k) {
        acc[0].add(a[k].x * a[k].x);
        acc[0].add(a[k].y * a[k].y);
      }
    } else {
#pragma unroll
      for (int i = 0; i <= KRY_MAXM; ++i)
        if (i < n) {
          float2 v[KRY_AHEAD];                             // (from L1)
#pragma unroll
          for (int k = 0; k < KRY_AHEAD; ++k) v[k] = ld2(V.v[i] + p[k]);
#pragma unroll
          for (int k = 0; k < KRY_AHEAD; ++k) {
            acc[i].add(a[k].x * v[k].x);
            acc[i].add(a[k].y * v[k].y);
          }
        }
    }
  }
  kreduce(acc, self ? 1 : n, T, S);
}

// out = c[0] x (out may be x) and, when r != nullptr, r = out too (the preconditioner's input)
__global__ void __launch_bounds__(KRY_THREADS) k_kscale(const int32_t* __restrict__ tiles, int ntiles, int nx, int ny,
                                                        int pitch, const uint8_t* __restrict__ cls, const float* x,
                                                        float* out, float* r, const KryScalars* __restrict__ S) {
  pdl_enter();
  const float c0 = (float)S->c[0];
  for (int t = KRY_TILES * blockIdx.x + (threadIdx.x >> 7); t < ntiles; t += KRY_TILES * gridDim.x) {
    long p;
    if (!kcell(tiles, t, nx, ny, pitch, p)) continue;
    const uint32_t cc = cls2(cls, p);
    const float2 v = ld2(x + p), o = make_float2(c0 * v.x, c0 * v.y);
    st2(out + p, o, cc);
    if (r) st2(r + p, o, cc);
  }
}

// w = (h^2 L) z and zj = z on every non-empty cell: CTAs [0, nrow) the fitted rows (256 each), the others a 32 x 8 tile each (FP32 stencil)
template <bool CROSS>
__global__ void __launch_bounds__(KRY_THREADS) k_kapply(const int32_t* __restrict__ tiles, int nx, int ny, int pitch,
                                                        const uint8_t* __restrict__ cls, const float* __restrict__ z,
                                                        float* __restrict__ w, float* __restrict__ zj,
                                                        Stencil<float> St, int nrow, int n2, int W,
                                                        const int32_t* __restrict__ cell, const int32_t* __restrict__ col,
                                                        const float* __restrict__ val) {
  if ((int)blockIdx.x < nrow) {
    const int row = blockIdx.x * KRY_THREADS + threadIdx.x;
    pdl_enter();
    if (row >= n2) return;
    float acc = 0;
#pragma unroll 15
    for (int k = 0; k < W; ++k) acc += val[(long)k * n2 + row] * z[col[(long)k * n2 + row]];
    w[cell[row]] = acc;
    return;
  }
  pdl_enter();
  const int t = blockIdx.x - nrow;
  const int i = tiles[2 * t] * TX + (threadIdx.x & 31);
  const int j = tiles[2 * t + 1] * TY + (threadIdx.x >> 5);
  if (i >= nx || j >= ny) return;
  const long p = (long)(j + 2) * pitch + (i + 2);
  const uint8_t c = cls[p];
  if (c == 0) return;
  zj[p] = z[p];
  if (c == 1) w[p] = stencil_apply<float, CROSS>(z, p, pitch, St);
}

// u_hat += sum_{j < n} y_j z_j on the non-empty cells (the sum in FP32, the update in FP64)
__global__ void __launch_bounds__(KRY_THREADS) k_kupdate(const int32_t* __restrict__ tiles, int ntiles, int nx, int ny,
                                                         int pitch, const uint8_t* __restrict__ cls, KryVecs Z, int n,
                                                         const KryScalars* __restrict__ S, double* __restrict__ u) {
  pdl_enter();
  float y[KRY_MAXM];
#pragma unroll
  for (int k = 0; k < KRY_MAXM; ++k) y[k] = k < n ? (float)S->y[k] : 0.f;
  for (int t = KRY_TILES * blockIdx.x + (threadIdx.x >> 7); t < ntiles; t += KRY_TILES * gridDim.x) {
    long p;
    if (!kcell(tiles, t, nx, ny, pitch, p)) continue;
    const uint32_t cc = cls2(cls, p);
    float2 a = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < KRY_MAXM; ++k)
      if (k < n) {
        const float2 v = ld2(Z.v[k] + p);
        a.x = fmaf(y[k], v.x, a.x);
        a.y = fmaf(y[k], v.y, a.y);
      }
    if (cc & 0xffu) u[p] += (double)a.x;
    if (cc >> 8) u[p + 1] += (double)a.y;
  }
}

}  // namespace dev
}  // namespace ccm
