// One block-Jacobi smoothing sweep of a level (SMO-1 on the regular cells and the SMO-2
// overlapping-block corrections of the irregular cells, both from the old iterate, Sec. 4.1)
// as one persistent launch.
//
// Work items: the SMO-2 blocks first, then the 64 x 32 cell tiles with a regular cell.  CTA c
// takes items c, c + G, c + 2G, ... (G = grid size, a multiple of the SM count where the
// level is large).  Every item's operands arrive in one of two shared-memory stages, so the
// copy of item k + 1 is in flight while item k computes:
//   tile item:  the 68 x 36 halo tile of u, the 68 x 32 box of r over the tile's rows and the
//               80 x 36 class bytes (one 2-D TMA box each; x origin 64a, 16-byte aligned),
//               and with PRO the 36 x 18 box of the coarse iterate under the tile;
//   block item: the block's rows of inv(L22[ext, ext]) by one bulk copy (cp.async.bulk; in FP64
//               two copies of half the rows each, in consecutive stages); the residuals of its
//               extended rows are gathered from global memory meanwhile.
// With PRO the sweep is the first post-smoothing sweep of Alg. 2 and reads u + P uc, the
// coarse correction added to regular cells only (Sec. 4.1).  A level's first sweep may start
// from a zero iterate (zero_u: no iterate copied or gathered), and the last level-0 sweep of
// an outer iteration may add its new values to the FP64 solution (uhat).
// Before the grid dependency wait each CTA does what depends on no earlier launch: copy
// barriers, prefetches of its blocks' fitted rows, and the copies of its first two items'
// static parts (inverse rows, class bytes); the iterate and r follow the wait.
// Waits are bounded by the SM clock; a wait that runs out sets the error word, waits (again
// bounded) for every copy still in flight, and the CTA leaves, all threads together.
#pragma once

#include "blocks.cuh"
#include "kernels.cuh"

namespace ccm {
namespace dev {

// stages that one block item takes: its inverse rows whole in FP32; half of them at a time in
// FP64, where the whole (57 KB at 64 core and 112 extended rows) would make a stage so large
// that one CTA per SM is resident instead of two
template <typename T>
constexpr int BLOCK_PARTS = sizeof(T) == 8 ? 2 : 1;
// Right-hand sides of a batch that share block items (FP32; 256 threads update 64 core rows of 4), in
// batches of at least BATCH_SHARE_FROM.  A shared item takes its four residual gathers one after the
// other, which is the launch's critical path until every CTA has many items.  Solves, sharing / apart, ms
// (star 256^2, disk 512^2, star 1024^2): 4 right-hand sides 2.30 / 1.29, 3.43 / 2.33, 5.42 / 3.49; 24: 3.44 / 2.62,
// 7.47 / 6.82, 13.1 / 12.6; 32: 3.56 / 4.23, 10.1 / 11.8, 21.1 / 24.3; 64: 7.20 / 7.67, 20.5 / 22.6.  Only the 128^2
// grids still lose at 32 (star 1.77 / 1.76, disk 2.18 / 2.02), and only the larger ones gain at 16 (up to 9 %).
constexpr int BATCH_SHARE_FROM = 32;
constexpr int BATCH_SHARE = 4;

template <typename T>
struct SmoothArgs {
  SweepArgs<T> a;      // level arrays, stencil, iterates, blocks (chunks == 1)
  int nbi;             // block items (= a.nblk)
  int nitems;          // nbi + a.ntiles: items of one right-hand side
  int nb;              // right-hand sides of the launch (grid y: groups of R of them)
  int ctas;            // CTAs per right-hand side
  uint32_t stage;      // bytes per stage (multiple of 128)
  int max_ext;         // most extended rows of a block (the per-row scratch after the stages)
};


// two adjacent values of T (8 or 16 bytes, aligned)
template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

__device__ __forceinline__ float2 pair(float a) { return make_float2(a, a); }

// w[0..5] = row[0..5] as three aligned pair loads (row at an even element offset)
template <typename T>
__device__ __forceinline__ void load_six(const T* row, T (&w)[6]) {
  using V2 = typename Pair<T>::type;
  const V2 a = *reinterpret_cast<const V2*>(row);
  const V2 b = *reinterpret_cast<const V2*>(row + 2);
  const V2 c = *reinterpret_cast<const V2*>(row + 4);
  w[0] = a.x;
  w[1] = a.y;
  w[2] = b.x;
  w[3] = b.y;
  w[4] = c.x;
  w[5] = c.y;
}

// offsets inside a stage of a tile item
template <typename T>
struct TileStage {
  static constexpr uint32_t al(uint32_t b) { return (b + 127u) & ~127u; }
  static constexpr uint32_t u_bytes = HY * HX * sizeof(T);
  static constexpr uint32_t r_bytes = JY * HX * sizeof(T);
  static constexpr uint32_t c_bytes = HY * CLX;
  static constexpr uint32_t uc_bytes = UCY * UCX * sizeof(T);
  static constexpr uint32_t r_off = al(u_bytes);
  static constexpr uint32_t c_off = r_off + al(r_bytes);
  static constexpr uint32_t uc_off = c_off + al(c_bytes);
  static constexpr uint32_t bytes(bool pro) { return pro ? uc_off + uc_bytes : c_off + c_bytes; }
};

__device__ __forceinline__ bool wait_parity(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (clock64() - t0 < TMA_WAIT_CYCLES)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// The copy of an item (of the given half of a block's rows where BLOCK_PARTS is 2) into stage
// st, completing on bar.  part 0: all of it; part 1: what
// does not depend on the previous launch (a block's inverse rows; a tile's class bytes, with
// the byte count of the whole tile), issued before the grid dependency wait; part 2: the rest
// of a tile (iterate, right-hand side, coarse iterate), after it.
template <typename T, bool PRO>
__device__ __forceinline__ void smooth_issue(const SmoothArgs<T>& A, const CUtensorMap* tin, const CUtensorMap* tr,
                                             const CUtensorMap* tcls, const CUtensorMap* tuc, int z, int item, int half,
                                             unsigned char* st, uint64_t* bar, int part = 0) {
  const SweepArgs<T>& a = A.a;
  if (item < A.nbi) {
    if (part == 2) return;
    const int b = item;
    const int nc = a.blk[4 * b + 1] - a.blk[4 * b], ne = a.blk[4 * b + 3] - a.blk[4 * b + 2];
    const int e0 = BLOCK_PARTS<T> == 2 && half ? block_split(ne) : 0;
    const int e1 = BLOCK_PARTS<T> == 2 && !half ? block_split(ne) : ne;
    const uint32_t abytes = block_copy_bytes(e1 - e0, nc, sizeof(T));
    mbar_expect_tx(bar, abytes);
    if (abytes) bulk_load(st, a.inv + a.blk_off[b] + (long)e0 * nc, abytes, bar);   // (a block of 1 or 2 rows: an empty part)
  } else {
    using S = TileStage<T>;
    const int t = item - A.nbi;
    const int cx0 = a.tiles[2 * t] * JX, cy0 = a.tiles[2 * t + 1] * JY;
    const bool no_u = !PRO && a.zero_u;     // the old iterate is 0
    if (part != 2) {
      mbar_expect_tx(bar, (no_u ? 0u : S::u_bytes) + S::r_bytes + S::c_bytes + (PRO ? S::uc_bytes : 0));
      tma_load_2d(st + S::c_off, tcls, bar, cx0, cy0);
    }
    if (part != 1) {
      if (!no_u) tma_load_3d(st, tin, bar, cx0, cy0, z);
      tma_load_3d(st + S::r_off, tr, bar, cx0, cy0 + 2, z);
      if (PRO) tma_load_3d(st + S::uc_off, tuc, bar, cx0 / 2, cy0 / 2 + 1, z);
    }
  }
}

// SMO-2 residuals of block b's extended rows from u_old (u_old + P uc with PRO) into sres,
// and each row's cell and old value (an irregular cell: no coarse correction) into scell and
// sold for the update of the core rows; the block's core start, core size and extended size
// come back, the core's first row at extended row cs - es.  CG: u_old is read through L2
// only (iterates that other CTAs of the same launch wrote).
template <typename T, bool PRO, bool CG>
__device__ __forceinline__ void block_residuals(const SweepArgs<T>& a, int b, const T* __restrict__ u_old,
                                                const T* __restrict__ rhs, const T* __restrict__ ucs, T* sres,
                                                T* sold, int* scell, int& cs, int& nc, int& ne, int& es) {
  cs = a.blk[4 * b];
  nc = a.blk[4 * b + 1] - cs;
  es = a.blk[4 * b + 2];
  ne = a.blk[4 * b + 3] - es;
  if (!PRO && a.zero_u) {   // the old iterate is 0: the residual is r
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      const int q = a.cell[es + e];
      sres[e] = rhs[q];
      sold[e] = (T)0;
      scell[e] = q;
    }
    return;
  }
  // Two threads a row (a block has at most 256 / 2 rows at the default shape), each every other
  // one of its coefficients.  The gathers' round trips are the launch's critical path on small
  // levels, so each thread has up to eight in flight and none hangs on a branch: a column without a
  // coarse parent reads cell 0, which lies in the zero ring, and adds nothing (one thread a row and a
  // branch a coefficient: a PRO sweep of a small level took 11.8 us cold, now 7.1).
  const int part = threadIdx.x & 1;
  for (int e0 = 0; e0 < ne; e0 += blockDim.x / 2) {
    const int e = e0 + (int)(threadIdx.x >> 1);
    const bool on = e < ne;
    const int row = es + (on ? e : 0);
    const int q = a.cell[row];
    const T rq = rhs[q], uq = CG ? __ldcg(u_old + q) : u_old[q];    // (with the gathers in flight)
    T acc = 0;
    for (int m0 = part; m0 < a.W; m0 += 16) {
      int cq[8], pq[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const long o = (long)min(m0 + 2 * k, a.W - 1) * a.n2 + row;
        cq[k] = a.col[o];
        pq[k] = PRO ? a.par[o] : 0;
      }
      T v[8], c[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        v[k] = CG ? __ldcg(u_old + cq[k]) : u_old[cq[k]];
        c[k] = PRO ? ucs[max(pq[k], 0)] : (T)0;
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int m = m0 + 2 * k;
        if (PRO && pq[k] >= 0) v[k] += c[k];
        if (m < a.W) acc += a.val[(long)m * a.n2 + row] * v[k];
      }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (on && part == 0) {
      sres[e] = rq - acc;
      sold[e] = uq;
      scell[e] = q;
    }
  }
}

// FP32: u_new = u_old + inv(L22[ext, ext]) sres on the block's core cells; As = the staged rows
// [ne][nc] of the inverse, two columns a lane, extended rows over warps (two barriers for a
// block of 64 core rows); the core cells and their old values from scell and sold (no global
// round trip before the stores)
// for nr <= R right-hand sides, sres and sold of one `slot` values after the other's, u_new and
// uhat `bs` apart
template <int R>
__device__ __forceinline__ void block_apply(const float* As, const float* sres, const float* sold, int slot, const int* scell,
                                            int c0, int nc, int ne, int nr, float* __restrict__ u_new,
                                            double* __restrict__ uhat, long bs, float (*part)[8][64]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int cb = 0; cb < nc; cb += 64) {
    if (cb) __syncthreads();      // part is free
    const int c = cb + 2 * lane;
    float2 acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = make_float2(0.0f, 0.0f);
    if (c + 1 < nc && !(nc & 1)) {
#pragma unroll 4
      for (int e = warp; e < ne; e += 8) {
        const float2 m = *reinterpret_cast<const float2*>(As + e * nc + c);
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (R == 1 || r < nr) acc[r] = __ffma2_rn(m, pair(sres[r * slot + e]), acc[r]);
      }
    } else if (c < nc) {          // an odd number of columns: the rows' pairs are not aligned
      for (int e = warp; e < ne; e += 8)
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (R > 1 && r >= nr) continue;
          acc[r].x += As[e * nc + c] * sres[r * slot + e];
          if (c + 1 < nc) acc[r].y += As[e * nc + c + 1] * sres[r * slot + e];
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) *reinterpret_cast<float2*>(&part[r][warp][2 * lane]) = acc[r];
    __syncthreads();
    const int r = threadIdx.x >> 6, l = threadIdx.x & 63, t = cb + l;
    if (r < nr && t < nc) {
      float tot = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) tot += part[r][w][l];
      const int q = scell[c0 + t];
      const float v = sold[r * slot + c0 + t] + tot;
      u_new[r * bs + q] = v;
      if (uhat) uhat[r * bs + q] += (double)v;
    }
  }
}

// FP64: the product of one part of the block's inverse rows with the residuals, one core
// column per thread and 256 / (64 or 128) groups of extended rows, added to acc; after the last
// part the groups' sums and the core cells' update as in block_apply.  FP64 issue bounds it (112
// x 64 FMA at two a clock are 1.7 us), so the columns spread over as many warps as there are
// for the final sums too.
__device__ __forceinline__ void block_apply_part(const double* As, const double* sres, const double* sold,
                                                 const int* scell, int c0, int nc, int e0, int e1, bool last, double& acc,
                                                 double* __restrict__ u_new, double* part) {
  const int ncp = nc > 64 ? 128 : 64, ng = 256 / ncp;
  const int c = threadIdx.x & (ncp - 1), g = threadIdx.x / ncp;
  if (c < nc)
    for (int e = e0 + g; e < e1; e += ng) acc += As[(e - e0) * nc + c] * sres[e];
  if (!last) return;
  part[threadIdx.x] = acc;
  acc = 0;
  __syncthreads();
  if (g == 0 && c < nc) {
    double tot = part[c];
    for (int w = 1; w < ng; ++w) tot += part[w * ncp + c];
    u_new[scell[c0 + c]] = sold[c0 + c] + tot;
  }
}

// FP64 sum of the stencil at a cell c of a staged tile, in factored form (the x-derivative of each row
// and 13 FMA): the cells that the integer form does not take
template <bool CROSS>
__device__ __forceinline__ double fp64_sum(const double* __restrict__ c, const Stencil<double>& S) {
  double acc = S.cc * c[0];
  acc = fma(S.lx[0], c[-2], acc);
  acc = fma(S.lx[1], c[-1], acc);
  acc = fma(S.lx[3], c[1], acc);
  acc = fma(S.lx[4], c[2], acc);
  acc = fma(S.ly[0], c[-2 * HX], acc);
  acc = fma(S.ly[1], c[-HX], acc);
  acc = fma(S.ly[3], c[HX], acc);
  acc = fma(S.ly[4], c[2 * HX], acc);
  if (CROSS)
    for (int dj = 0; dj < 5; ++dj) {
      const double* r = c + (dj - 2) * HX;
      if (dj != 2) acc = fma(S.gy[dj], S.gx[0] * r[-2] + S.gx[1] * r[-1] + S.gx[3] * r[1] + S.gx[4] * r[2], acc);
    }
  return acc;
}

// h^2 L u at the cells (x0, y0 + k) and (x0 + 1, y0 + k), k = 0 .. 3, of a staged tile of doubles
// for all 256 threads of a CTA (x0, y0: two columns and four rows a thread): in integer form, or as
// an FP64 sum where that does not apply (see fixed.cuh).  The integers go to q, with LOCAL an array
// beside the tile, else the tile itself.  emit(k, Lu0, Lu1) only where on.  With LOCAL few() is called
// afterwards by a thread with a cell whose own value is small; it looks at the cells' sums and replaces
// what it must (few_cells).  Barriers inside; without LOCAL a thread that needs the tile's
// own values reads them before the call.
template <bool CROSS, bool LOCAL, class Emit, class Few>
__device__ __forceinline__ void tile_stencil64(double* tile, long long* q, unsigned* wmax, int x0, int y0, bool on,
                                               const Stencil<double>& S, const QStencil& Q, Emit emit, Few few) {
  constexpr int NP = HY * HX / 2;
  QSlots<(NP + 255) / 256> v;
  const unsigned m = q_cta_max(v.load(tile, NP), wmax);
  const int E = q_scale(m, Q);
  if (E < 0) {
    if (on)
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        double s[2];
#pragma unroll 1
        for (int j = 0; j < 2; ++j) s[j] = fp64_sum<CROSS>(tile + (y0 + k + 2) * HX + x0 + j + 2, S);
        emit(k, s[0], s[1]);
      }
    return;
  }
  v.template store<LOCAL>(q, NP, E);
  __syncthreads();
  const int e = E - 1022 + (LOCAL ? Q.cexp : Q.plain.cexp);
  if (on) {
    const bool ok = q_rows<CROSS, HX, LOCAL>(q, x0, y0, Q, [&](int k, long long s0, long long s1) { emit(k, q_double(s0, e), q_double(s1, e)); });
    if (LOCAL && !ok && m != 0) few();
  }
}

// FP64 sums for those of a thread's cells that the caller needs and whose sum of |w u| is too small for
// the integer form: one(k, j, Lu), need(k, j): cell (x0 + j, y0 + k)
template <bool CROSS, class Need, class One>
__device__ __forceinline__ void few_cells(const double* tile, const long long* q, int x0, int y0, const Stencil<double>& S,
                                          const QStencil& Q, Need need, One one) {
  unsigned skip = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) skip |= need(t >> 1, t & 1) ? 0u : 1u << t;
  if (skip == 255u) return;
  const unsigned few = q_few<CROSS, HX>(q, tile, x0, y0, Q, skip);
#pragma unroll 1
  for (int t = 0; t < 8; ++t)
    if (few >> t & 1)
      one(t >> 1, t & 1, fp64_sum<CROSS>(tile + (y0 + (t >> 1) + 2) * HX + x0 + (t & 1) + 2, S));
}

// FP32: h^2 L u at the cells (x0, y0 + k) and (x0 + 1, y0 + k), k = 0 .. 3, of a staged tile.
// Issue slots bound this loop, so the two cells go through packed operations (two FMA an issue slot)
// and the mixed term is factored: the x-derivative of each of the eight rows once (its weights 1
// and 8 are exact) and four operations a cell, in place of 16 FMA a cell.  The nine taps of the
// two second derivatives keep the order of a plain sum; odd taps would need the pairs at odd
// columns and stay scalar.  Error against 64-bit sums, rms over smooth and rough fields: 0.52 to
// 0.95 of the 25-tap FMA chain's, equal to it without the mixed term.
// emit(k, Lu, u) with both cells' values.  A sweep of the star 4096^2's finest level, cold: 22.5 us
// with the 25-tap sum and a class test a cell, 20.2 us with this and one test for eight cells.
template <bool CROSS, class Emit>
__device__ __forceinline__ void stencil32(const float* __restrict__ tile, int x0, int y0, const Stencil<float>& S,
                                          Emit emit) {
  float2 u[8], d[8], e[8], f[8];    // of a row: the cells' pair, its x-derivatives times 12, the pairs left and right of it
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    float w[6];
    load_six(tile + (y0 + q) * HX + x0, w);
    u[q] = make_float2(w[2], w[3]);
    e[q] = make_float2(w[0], w[1]);
    f[q] = make_float2(w[4], w[5]);
    if (CROSS)
      d[q] = __ffma2_rn(pair(8.0f), make_float2(w[3] - w[1], w[4] - w[2]), __ffma2_rn(pair(-1.0f), f[q], e[q]));
    if (q < 4) continue;
    const int k = q - 4, c = k + 2;
    float2 s;
    if (CROSS) {
      const float2 g = __ffma2_rn(pair(8.0f), __ffma2_rn(pair(-1.0f), d[c - 1], d[c + 1]),
                                  __ffma2_rn(pair(-1.0f), d[c + 2], d[c - 2]));
      s = __ffma2_rn(pair(S.w[2]), u[c - 2], __fmul2_rn(pair(S.w[0]), g));
    } else {
      s = __fmul2_rn(pair(S.w[2]), u[c - 2]);
    }
    s = __ffma2_rn(pair(S.w[7]), u[c - 1], s);
    s = __ffma2_rn(pair(S.w[10]), e[c], s);
    s.x = fmaf(S.w[11], e[c].y, s.x);
    s.y = fmaf(S.w[11], u[c].x, s.y);
    s = __ffma2_rn(pair(S.w[12]), u[c], s);
    s.x = fmaf(S.w[13], u[c].y, s.x);
    s.y = fmaf(S.w[13], f[c].x, s.y);
    s = __ffma2_rn(pair(S.w[14]), f[c], s);
    s = __ffma2_rn(pair(S.w[17]), u[c + 1], s);
    s = __ffma2_rn(pair(S.w[22]), u[c + 2], s);
    emit(k, s, u[c]);
  }
}

// SMO-1 on the regular cells of a staged 64 x 32 tile (halo box of u, box of r and class bytes
// at the TileStage offsets of st; with PRO the coarse box too, whose parent values are first
// added to the staged regular cells: the sweep then reads u + P uc)
template <typename T, bool CROSS, bool PRO, bool LOCAL>
__device__ __forceinline__ void tile_sweep(const SweepArgs<T>& a, unsigned char* st, long long* q, int cx0, int cy0,
                                           T* __restrict__ u_new, double* __restrict__ uhat, unsigned* wmax) {
  using S = TileStage<T>;
  T* tile = reinterpret_cast<T*>(st);
  const T* rt = reinterpret_cast<const T*>(st + S::r_off);
  const uint8_t* ct = st + S::c_off;
  if (PRO) {
    // staged cell (y, x) has its parent at (y / 2, x / 2 + 1) of the coarse box; four cells
    // (one 32-bit word of class bytes, two parents, two aligned pairs of the tile) per step,
    // the tile's 36 x 17 quads spread over all threads
    using P2 = typename Pair<T>::type;
    const T* uct = reinterpret_cast<const T*>(st + S::uc_off);
    for (int q = threadIdx.x; q < HY * (HX / 4); q += blockDim.x) {
      const int y = q / (HX / 4), xq = q - y * (HX / 4), x0 = 4 * xq;
      const uint32_t c4 = *reinterpret_cast<const uint32_t*>(ct + y * CLX + x0);
      const T p0 = uct[(y >> 1) * UCX + 2 * xq + 1], p1 = uct[(y >> 1) * UCX + 2 * xq + 2];
      P2* tr = reinterpret_cast<P2*>(tile + y * HX + x0);
      P2 v0 = tr[0], v1 = tr[1];
      if ((c4 & 0xffu) == 1u) v0.x += p0;
      if (((c4 >> 8) & 0xffu) == 1u) v0.y += p0;
      if (((c4 >> 16) & 0xffu) == 1u) v1.x += p1;
      if ((c4 >> 24) == 1u) v1.y += p1;
      tr[0] = v0;
      tr[1] = v1;
    }
    __syncthreads();
  }
  if constexpr (sizeof(T) == 8) {
    // FP64: the same two columns and four rows per thread as below; the stencil in integer form
    // (FP64 issue would bound it: 19 operations a cell, 9.4 us a tile)
    using V2 = double2;
    const int x0 = 2 * (threadIdx.x & 31), y0 = (threadIdx.x >> 5) * 4;
    const int i0 = cx0 + x0;
    auto put = [&](int kk, double v0, double v1) {
      const uint32_t c2 = *reinterpret_cast<const uint16_t*>(ct + (y0 + kk + 2) * CLX + x0 + 2);
      const bool g0 = (c2 & 0xffu) == 1u, g1 = (c2 >> 8) == 1u && i0 + 1 < a.nx;
      const long p = (long)(cy0 + y0 + kk + 2) * a.pitch + (i0 + 2);
      if (g0 && g1) {
        *reinterpret_cast<V2*>(u_new + p) = make_double2(v0, v1);
      } else {
        if (g0) u_new[p] = v0;
        if (g1) u_new[p + 1] = v1;
      }
    };
    if (!PRO && a.zero_u) {
      if (i0 < a.nx)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const V2 r2 = *reinterpret_cast<const V2*>(rt + (y0 + kk) * HX + x0 + 2);
          put(kk, a.S.omega_d * r2.x, a.S.omega_d * r2.y);
        }
      return;
    }
    V2 c[4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) c[kk] = *reinterpret_cast<const V2*>(tile + (y0 + kk + 2) * HX + x0 + 2);
    if (!LOCAL) q = reinterpret_cast<long long*>(tile);
    const auto emit = [&](int kk, double s0, double s1) {
      const V2 r2 = *reinterpret_cast<const V2*>(rt + (y0 + kk) * HX + x0 + 2);
      const V2 u = kk == 0 ? c[0] : kk == 1 ? c[1] : kk == 2 ? c[2] : c[3];
      put(kk, u.x + a.S.omega_d * (r2.x - s0), u.y + a.S.omega_d * (r2.y - s1));
    };
    const auto need = [&](int kk, int j) { return ct[(y0 + kk + 2) * CLX + x0 + j + 2] == 1; };
    const auto one = [&](int kk, int j, double s) {      // (a needed cell: regular, in the grid)
      const double u = tile[(y0 + kk + 2) * HX + x0 + j + 2], r = rt[(y0 + kk) * HX + x0 + j + 2];
      u_new[(long)(cy0 + y0 + kk + 2) * a.pitch + (i0 + j + 2)] = u + a.S.omega_d * (r - s);
    };
    tile_stencil64<CROSS, LOCAL>(tile, q, wmax, x0, y0, i0 < a.nx, a.S, a.Q, emit,
                                 [&] { if constexpr (LOCAL) few_cells<CROSS>(tile, q, x0, y0, a.S, a.Q, need, one); });
  } else {
    // FP32: two adjacent cells (x0, x0 + 1) in four rows per thread; class bytes, right-hand sides
    // and new values move in pairs.  A thread whose eight cells are all regular (most are) stores
    // without looking at them one by one.
    const int x0 = 2 * (threadIdx.x & 31), y0 = (threadIdx.x >> 5) * 4;
    const uint8_t* cp = ct + (y0 + 2) * CLX + x0 + 2;
    uint32_t c2[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c2[k] = *reinterpret_cast<const uint16_t*>(cp + k * CLX);
    const uint32_t all = c2[0] & c2[1] & c2[2] & c2[3];     // class bytes are 0 (empty, and outside the grid), 1, 2
    const float* rp = rt + y0 * HX + x0 + 2;
    float2 v[4];
    if (!PRO && a.zero_u) {
      // the old iterate is 0 (its tile was not copied): u_new = omega_d r on the regular cells
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 r2 = *reinterpret_cast<const float2*>(rp + k * HX);
        v[k] = make_float2(a.S.omega_d * r2.x, a.S.omega_d * r2.y);
      }
    } else {
      stencil32<CROSS>(tile, x0, y0, a.S, [&](int k, float2 s, float2 u) {
        const float2 r2 = *reinterpret_cast<const float2*>(rp + k * HX);
        v[k] = __ffma2_rn(pair(a.S.omega_d), __ffma2_rn(pair(-1.0f), s, r2), u);
      });
    }
    // into u_new, and added to u_hat where the sweep folds in the outer iteration's update
    const long p = (long)(cy0 + y0 + 2) * a.pitch + (cx0 + x0 + 2);
    T* o = u_new + p;
    double* h = uhat ? uhat + p : nullptr;
    if (all == 0x0101u) {
      double2 w[4];
      if (h)
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = *reinterpret_cast<const double2*>(h + (long)k * a.pitch);
#pragma unroll
      for (int k = 0; k < 4; ++k) *reinterpret_cast<float2*>(o + (long)k * a.pitch) = v[k];
      if (h)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          *reinterpret_cast<double2*>(h + (long)k * a.pitch) = make_double2(w[k].x + (double)v[k].x, w[k].y + (double)v[k].y);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const long q = (long)k * a.pitch;
        if ((c2[k] & 0xffu) == 1u) {
          o[q] = v[k].x;
          if (h) h[q] += (double)v[k].x;
        }
        if ((c2[k] >> 8) == 1u) {
          o[q + 1] = v[k].y;
          if (h) h[q + 1] += (double)v[k].y;
        }
      }
    }
  }
}

// R: right-hand sides of a batch that share a CTA's items (grid y: groups of R).  A block item
// serves all of them with one copy of its inverse rows (28 KB; one right-hand side at a time
// these copies were two fifths of a sweep's L2 reads), then come the tile items of the first, the
// second, ...
// LOCAL (FP64, one sweep by itself): the regular cells' stencil as accurate cell by cell as an FP64
// sum (tile_stencil64), with the integers after the blocks' scratch; that leaves one CTA an SM
template <typename T, bool CROSS, bool PRO, int R = 1, bool LOCAL = false>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 2 : 3) k_smooth(const __grid_constant__ CUtensorMap tin,
                                                const __grid_constant__ CUtensorMap tr,
                                                const __grid_constant__ CUtensorMap tcls,
                                                const __grid_constant__ CUtensorMap tuc, SmoothArgs<T> A) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ __align__(16) T part[R][8][sizeof(T) == 8 ? 32 : 64];
  __shared__ __align__(16) unsigned wmax[8];
  const SweepArgs<T>& a = A.a;
  // While the previous launch drains: pull the static fitted-row data (columns, coefficients,
  // cells, parents) of this CTA's SMO-2 block items into L1, so that each block's residual
  // gathers need one round trip to the iterate instead of two
  for (int b = blockIdx.x; b < A.nbi; b += gridDim.x) {
    const int es = a.blk[4 * b + 2], ne = a.blk[4 * b + 3] - es;
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
      const int row = es + e;
      prefetch_l1(a.cell + row);
#pragma unroll 15
      for (int m = 0; m < a.W; ++m) {
        prefetch_l1(a.col + (long)m * a.n2 + row);
        prefetch_l1(a.val + (long)m * a.n2 + row);
        if (PRO && a.par) prefetch_l1(a.par + (long)m * a.n2 + row);
      }
    }
    if (threadIdx.x == 0) prefetch_l1(a.blk_off + b);
  }
  // (the last group may be a small one: fewer items, and CTAs only of its right-hand sides)
  const int z0 = blockIdx.y * R, nr = R == 1 ? 1 : min(R, A.nb - z0);
  const int nitems = R == 1 ? A.nitems : A.nbi + nr * a.ntiles;
  const int G = R == 1 ? (int)gridDim.x : min((int)gridDim.x, nr * A.ctas);
  if (R > 1 && (int)blockIdx.x >= min(G, nitems)) return;
  const int K = (nitems - (int)blockIdx.x + G - 1) / G;     // items of this CTA (>= 1)
  // its block items come first and take BLOCK_PARTS steps of the ring each: NB block steps in
  // all, K steps with the tiles'
  constexpr int BP = BLOCK_PARTS<T>;
  const int kb = (int)blockIdx.x < A.nbi ? (A.nbi - 1 - (int)blockIdx.x) / G + 1 : 0;
  const int NB = BP * kb, KS = K + (BP - 1) * kb;
  auto item_of = [&](int k) { return (int)blockIdx.x + (k < NB ? k / BP : k - NB + kb) * G; };
  // the right-hand side and the item among its own of a group's item
  auto rhs_of = [&](int item) { return R == 1 || item < A.nbi ? z0 : z0 + (item - A.nbi) / a.ntiles; };
  auto own_of = [&](int item) { return R == 1 || item < A.nbi ? item : A.nbi + (item - A.nbi) % a.ntiles; };
  auto issue = [&](int k, int half, int sb, int part) {
    const int item = item_of(k);
    smooth_issue<T, PRO>(A, &tin, &tr, &tcls, &tuc, rhs_of(item), own_of(item), half, smem_raw + sb * A.stage, &bar[sb], part);
  };
  // also before the wait: the copy barriers, and the parts of the first two items' copies
  // that no earlier launch writes (the rest follows the wait)
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    issue(0, 0, 0, 1);
    if (KS > 1) issue(1, 1, 1, 1);
  }
  __syncthreads();
  pdl_enter();
  // per extended row of a block item: residual, old value, cell (slots of max_ext, the first two for each right-hand side)
  const uint32_t slot = (uint32_t)(((long)A.max_ext * sizeof(T) + 15) & ~15L);
  T* sres = reinterpret_cast<T*>(smem_raw + 2 * A.stage);
  T* sold = reinterpret_cast<T*>(smem_raw + 2 * A.stage + R * slot);
  int* scell = reinterpret_cast<int*>(smem_raw + 2 * A.stage + 2 * R * slot);
  long long* ints = reinterpret_cast<long long*>(smem_raw + 2 * A.stage + (2 * R + 1) * slot);     // LOCAL
  if (threadIdx.x == 0) {
    issue(0, 0, 0, 2);
    if (KS > 1) issue(1, 1, 1, 2);
  }
  T acc = 0;                     // BP == 2: a block's product, carried from its first half to its second
  int cs = 0, nc = 0, ne = 0, es = 0;
  for (int k = 0; k < KS; ++k) {
    const int item = item_of(k), half = k % BP;      // half: of a block item
    const int sb = k & 1;
    const uint32_t parity = (k >> 1) & 1;
    int cx0 = 0, cy0 = 0;
    if (item < A.nbi) {
      if (half == 0)
        for (int r = 0; r < nr; ++r) {
          const long bo = (long)(z0 + r) * a.bs;
          block_residuals<T, PRO, false>(a, item, a.u_old + bo, a.r + bo, PRO ? a.uc + (long)(z0 + r) * a.bsc : nullptr,
                                         sres + r * (slot / sizeof(T)), sold + r * (slot / sizeof(T)), scell, cs, nc, ne, es);
        }
    } else {
      const int t = own_of(item) - A.nbi;       // the tile's origin, read before the wait
      cx0 = a.tiles[2 * t] * JX;
      cy0 = a.tiles[2 * t + 1] * JY;
    }
    const bool ok = __syncthreads_and(wait_parity(&bar[sb], parity));
    if (!ok) {
      // this copy and the other stage's (if one was issued) must land before the CTA leaves
      wait_parity(&bar[sb], parity);
      if (k + 1 < KS) wait_parity(&bar[sb ^ 1], ((k + 1) >> 1) & 1);
      if (threadIdx.x == 0) atomicExch(a.err, 1);
      return;
    }
    if (item < A.nbi) {
      const T* As = reinterpret_cast<const T*>(smem_raw + sb * A.stage);
      if constexpr (BP == 2) {
        const int e0 = half ? block_split(ne) : 0, e1 = half ? ne : block_split(ne);
        block_apply_part(As, sres, sold, scell, cs - es, nc, e0, e1, half == 1, acc, a.u_new + z0 * a.bs, &part[0][0][0]);
      } else {
        block_apply<R>(As, sres, sold, (int)(slot / sizeof(T)), scell, cs - es, nc, ne, nr, a.u_new + z0 * a.bs,
                       a.uhat ? a.uhat + z0 * a.bs : nullptr, a.bs, part);
      }
    } else {
      const long bo = rhs_of(item) * a.bs;
      tile_sweep<T, CROSS, PRO, LOCAL>(a, smem_raw + sb * A.stage, ints, cx0, cy0, a.u_new + bo,
                                       a.uhat ? a.uhat + bo : nullptr, wmax);
    }
    __syncthreads();      // stage sb is free
    if (threadIdx.x == 0 && k + 2 < KS) {
      fence_proxy_async();
      issue(k + 2, k % BP, sb, 0);
    }
  }
}

}  // namespace dev
}  // namespace ccm

namespace ccm {
namespace dev {

// The weights 4 |C_k| / sum |C| of the volume-weighted sums (Sec. 4.1) over the children of every coarse
// cell, once for each precision used (w64 or w32 may be null): two FP64 divisions a thread cost a tile of
// k_restrict_p 2.6 us.
__global__ void k_restrict_weights(int nxc, int nyc, int pitchf, const double* __restrict__ vol, double* __restrict__ w64,
                                   float* __restrict__ w32) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y;
  if (I >= nxc || J >= nyc) return;
  const long p = (long)(2 * J + 2) * pitchf + (2 * I + 2);
  const double2 a = *reinterpret_cast<const double2*>(vol + p), b = *reinterpret_cast<const double2*>(vol + p + pitchf);
  const double sv = a.x + a.y + b.x + b.y;
  const double v[4] = {a.x, a.y, b.x, b.y};
  for (int k = 0; k < 4; ++k) {
    const double w = sv > 0 ? 4 * v[k] / sv : 0.0;
    const long q = p + (k >> 1) * pitchf + (k & 1);
    if (w64) w64[q] = w;
    if (w32) w32[q] = (float)w;
  }
}

// ---- residual + restriction of a level (Alg. 2: the coarse right-hand side and a zero coarse
// iterate) as one persistent launch over the fine 64 x 32 tiles that restriction visits.
// A tile item's halo tile of u, its boxes of r and (FP32) of the restriction weights (68 x 32 over the
// tile's rows) and its class bytes (80 x 36) arrive by TMA in one of two stages while the
// previous item computes.  In FP64 each thread loads the weights of its coarse cells' children
// into registers before the wait instead: without their box two CTAs per SM are resident, not
// one.  The fitted rows of the tile's irregular cells (listed per tile:
// row and position) are gathered from global memory before the wait, and so are the class
// bytes of the coarse cells the thread restricts to; regular cells take the stencil from the
// staged tile; then the 32 x 16 coarse cells get the volume-weighted 2 x 2 sums.
template <typename T>
struct RestrictArgs {
  const int32_t* tiles;
  int ntiles, nxf, nyf, pitchf;
  const int32_t* rr_off;
  const int32_t* rr;
  int n2, W;
  const int32_t* irr_cell;
  const int32_t* col;
  const T* val;
  const T* u;
  const T* r;
  int nxc, nyc, pitchc;
  const uint8_t* clsc;
  T* rc;
  T* uc;
  const T* wt;         // restriction weights of the fine cells (k_restrict_weights)
  Stencil<T> S;
  QStencil Q;
  int* err;
  uint32_t stage;
  long bs, bsc;        // batch strides (elements) of the fine and the coarse level arrays
  int nrr;             // the tiles' irregular rows in tile order: (cell, position) pairs, and
  const int32_t* rq;   // the rows' columns and coefficients [W][nrr]
  const int32_t* rq_col;
  const T* rq_val;
};

template <typename T>
struct RestrictStage {
  static constexpr uint32_t al(uint32_t b) { return (b + 127u) & ~127u; }
  static constexpr uint32_t u_bytes = HY * HX * sizeof(T);
  static constexpr uint32_t r_bytes = JY * HX * sizeof(T);
  static constexpr uint32_t c_bytes = HY * CLX;
  static constexpr uint32_t r_off = al(u_bytes);
  static constexpr uint32_t c_off = r_off + al(r_bytes);
  static constexpr bool vbox = sizeof(T) == 4;     // the weights arrive by TMA too
  static constexpr uint32_t v_off = c_off + al(c_bytes);
  static constexpr uint32_t bytes = al(v_off + (vbox ? r_bytes : 0));
  static constexpr uint32_t tx = u_bytes + (vbox ? 2 : 1) * r_bytes + c_bytes;
};

// the static data of restriction tile t's irregular rows (cell and position pairs, columns
// and coefficients, contiguous in tile order) into L1: k0, k1 = the tile's row range
template <typename T>
__device__ __forceinline__ void prefetch_tile_rows(const RestrictArgs<T>& A, int k0, int k1) {
  for (int q = k0 + 16 * (int)threadIdx.x; q < k1; q += 16 * (int)blockDim.x) {
    prefetch_l1(A.rq + 2 * (long)q);
#pragma unroll 15
    for (int m = 0; m < A.W; ++m) {
      prefetch_l1(A.rq_col + (long)m * A.nrr + q);
      prefetch_l1(A.rq_val + (long)m * A.nrr + q);
    }
  }
}

template <typename T, bool CROSS, bool LOCAL = false>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 2 : 3) k_restrict_p(const __grid_constant__ CUtensorMap tin,
                                                       const __grid_constant__ CUtensorMap tr,
                                                       const __grid_constant__ CUtensorMap tcls,
                                                       const __grid_constant__ CUtensorMap tvol, RestrictArgs<T> A) {
  using S = RestrictStage<T>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ T res[JY][JX];      // residuals of the tile's irregular cells
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ __align__(16) unsigned wmax[8];
  const int G = gridDim.x;
  const int K = (A.ntiles - (int)blockIdx.x + G - 1) / G;
  // the first tile's row range and rows while the previous launch drains
  int n0 = A.rr_off[blockIdx.x], n1 = A.rr_off[blockIdx.x + 1];
  prefetch_tile_rows(A, n0, n1);
  // this CTA's right-hand side of the batch (blockIdx.y)
  const int z = blockIdx.y;
  // tile t's copy into stage sb.  part 0: all of it; part 1: the class bytes and weights,
  // which no launch writes, with the byte count of the whole tile (before the grid
  // dependency wait); part 2: the iterate and the right-hand side (after it)
  auto issue = [&](int t, int sb, int part) {
    unsigned char* st = smem_raw + sb * A.stage;
    const int cx0 = A.tiles[2 * t] * JX, cy0 = A.tiles[2 * t + 1] * JY;
    if (part != 2) {
      mbar_expect_tx(&bar[sb], S::tx);
      tma_load_2d(st + S::c_off, &tcls, &bar[sb], cx0, cy0);
      if (S::vbox) tma_load_2d(st + S::v_off, &tvol, &bar[sb], cx0, cy0 + 2);
    }
    if (part != 1) {
      tma_load_3d(st, &tin, &bar[sb], cx0, cy0, z);
      tma_load_3d(st + S::r_off, &tr, &bar[sb], cx0, cy0 + 2, z);
    }
  };
  // the copy barriers and the static parts of the first two tiles' copies too
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    issue(blockIdx.x, 0, 1);
    if (K > 1) issue(blockIdx.x + G, 1, 1);
  }
  __syncthreads();
  pdl_enter();
  const T* __restrict__ uf = A.u + (long)z * A.bs;
  const T* __restrict__ rf = A.r + (long)z * A.bs;
  T* __restrict__ rcz = A.rc + (long)z * A.bsc;
  T* __restrict__ ucz = A.uc + (long)z * A.bsc;
  if (threadIdx.x == 0) {
    issue(blockIdx.x, 0, 2);
    if (K > 1) issue(blockIdx.x + G, 1, 2);
  }
  for (int k = 0; k < K; ++k) {
    const int t = blockIdx.x + k * G;
    const int sb = k & 1;
    const uint32_t parity = (k >> 1) & 1;
    const int cx0 = A.tiles[2 * t] * JX, cy0 = A.tiles[2 * t + 1] * JY;
    const int k0 = n0, k1 = n1;
    // the next tile's row range: loaded now, used after this tile's stencil
    if (k + 1 < K) {
      n0 = A.rr_off[t + G];
      n1 = A.rr_off[t + G + 1];
    }
    for (int q = k0 + (int)threadIdx.x; q < k1; q += blockDim.x) {
      const int cell = A.rq[2 * q], loc = A.rq[2 * q + 1];
      T acc = 0;
#pragma unroll 15
      for (int m = 0; m < A.W; ++m) acc += A.rq_val[(long)m * A.nrr + q] * uf[A.rq_col[(long)m * A.nrr + q]];
      res[loc >> 6][loc & 63] = rf[cell] - acc;
    }
    // class bytes of this thread's two coarse cells (0 outside the coarse level), and in FP64
    // their children's weights
    uint8_t cc[2];
    typename Pair<T>::type vv[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int I = cx0 / 2 + (threadIdx.x & 31), J = cy0 / 2 + 2 * (threadIdx.x >> 5) + h;
      cc[h] = (I < A.nxc && J < A.nyc) ? A.clsc[(long)(J + 2) * A.pitchc + (I + 2)] : (uint8_t)0;
      if constexpr (!S::vbox)
        if (I < A.nxc && J < A.nyc) {
          const T* v = A.wt + (long)(2 * J + 2) * A.pitchf + (2 * I + 2);
          vv[h][0] = *reinterpret_cast<const double2*>(v);
          vv[h][1] = *reinterpret_cast<const double2*>(v + A.pitchf);
        }
    }
    const bool ok = __syncthreads_and(wait_parity(&bar[sb], parity));
    if (!ok) {
      wait_parity(&bar[sb], parity);
      if (k + 1 < K) wait_parity(&bar[sb ^ 1], ((k + 1) >> 1) & 1);
      if (threadIdx.x == 0) atomicExch(A.err, 1);
      return;
    }
    unsigned char* st = smem_raw + sb * A.stage;
    T* tile = reinterpret_cast<T*>(st);
    const T* rt = reinterpret_cast<const T*>(st + S::r_off);
    const uint8_t* ct = st + S::c_off;
    const T* vt = reinterpret_cast<const T*>(st + S::v_off);
    // A thread's eight cells (two columns of four rows) are the children of two coarse cells, one
    // above the other: their volume-weighted sums stay in registers; irregular cells' residuals
    // come from shared memory.
    const int x0 = 2 * (threadIdx.x & 31), y1 = (threadIdx.x >> 5) * 4;
    using V2 = typename Pair<T>::type;
    V2 rs[4];
    auto resid = [&](int kk, T s0, T s1) {
      const uint32_t c2 = *reinterpret_cast<const uint16_t*>(ct + (y1 + kk + 2) * CLX + x0 + 2);
      const V2 r2 = *reinterpret_cast<const V2*>(rt + (y1 + kk) * HX + x0 + 2);
      V2 t;
      t.x = r2.x - s0;
      t.y = r2.y - s1;
      if (c2 != 0x0101u) {
        const uint32_t c0 = c2 & 0xffu, c1 = c2 >> 8;
        if (c0 != 1u) t.x = c0 ? res[y1 + kk][x0] : (T)0;
        if (c1 != 1u) t.y = c1 ? res[y1 + kk][x0 + 1] : (T)0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)       // (kk may be a run-time value: rs stays in registers)
        if (j == kk) rs[j] = t;
    };
    if constexpr (sizeof(T) == 4)
      stencil32<CROSS>(tile, x0, y1, A.S, [&](int kk, float2 s, float2) { resid(kk, s.x, s.y); });
    else {
      long long* ints = reinterpret_cast<long long*>(LOCAL ? smem_raw + 2 * A.stage : st);
      const auto need = [&](int kk, int j) { return ct[(y1 + kk + 2) * CLX + x0 + j + 2] == 1; };
      const auto one = [&](int kk, int j, double s) {
        const double t = rt[(y1 + kk) * HX + x0 + j + 2] - s;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k == kk) (j ? rs[k].y : rs[k].x) = t;
      };
      tile_stencil64<CROSS, LOCAL>(tile, ints, wmax, x0, y1, true, A.S, A.Q, resid,
                                   [&] { if constexpr (LOCAL) few_cells<CROSS>(tile, ints, x0, y1, A.S, A.Q, need, one); });
    }
    if (k + 1 < K) prefetch_tile_rows(A, n0, n1);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (cc[h] == 0) continue;
      const long pc = (long)(cy0 / 2 + y1 / 2 + h + 2) * A.pitchc + (cx0 / 2 + x0 / 2 + 2);
      const T* v = vt + (y1 + 2 * h) * HX + x0 + 2;
      const V2 va = S::vbox ? *reinterpret_cast<const V2*>(v) : vv[h][0];
      const V2 vb = S::vbox ? *reinterpret_cast<const V2*>(v + HX) : vv[h][1];
      const V2 ra = rs[2 * h], rb = rs[2 * h + 1];
      rcz[pc] = va.x * ra.x + va.y * ra.y + vb.x * rb.x + vb.y * rb.y;
      ucz[pc] = (T)0;
    }
    __syncthreads();      // res and stage sb are free
    if (threadIdx.x == 0 && k + 2 < K) {
      fence_proxy_async();
      issue(t + 2 * G, sb, 0);
    }
  }
}

}  // namespace dev
}  // namespace ccm
