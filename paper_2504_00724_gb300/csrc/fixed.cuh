// The FP64 regular stencil (Sec. 3.2) in 64-bit integer arithmetic.
//
// GB300 issues FP64 at 2 FMA per clock per SM, 1/64 of the FP32 rate: a warp-wide FP64 FMA
// occupies its scheduler's pipe for 64 clocks, and the 17 FMA of the factored 25-tap stencil
// bound every FP64 pass over a level (9.4 us per 64 x 32 tile and SM).  Integer adds run at
// half the FP32 rate or better, so the stencil runs on fixed-point images of the staged values:
//
//   q = round(u 2^(60 - s)),  2^s the power of two above the largest |u| of the staged tile,
//   Lap  = (q_-1 + q_+1 - 2 q_0) - (q_-2 + q_+2 - 2 q_0) / 16    (eq. stdLap times 12 / 16),
//   Grad = (q_+1 - q_-1) + (q_-2 - q_+2) / 8                      (eq. stdGrad times 12 / 8),
//   h^2 L u = 2^.. (hi(A Lap_x) + hi(C Lap_y) + hi(B Grad_y(Grad_x))),
//
// with A = 16 a / 12, C = 16 c / 12, B = 64 b / 144 as 63-bit integers on one common power of two
// and hi() the upper half of the 128-bit product.  All of it stays below 2^63 for |q| < 2^60.  What
// is rounded is q (to 2^-61 of 2^s; a value within 2^7 of the largest not at all), the sixteenths
// and the eighths, the three products and the conversion to FP64.
//
// These errors are relative to the tile's largest value, those of an FP64 sum to the cell's own
// terms.  A pass whose results are the operator's values themselves (apply.cuh, a single sweep or
// restriction) keeps the doubles beside the integers and looks at every cell (FINE): where the sum of
// its |w u| is so small, against the tile's largest value, that their bound exceeds 3 2^-53 of that
// sum (near a spike, in the tail of a narrow kernel, at some zeros of a smooth field: in one warp of 14
// at most), the FP64 sum replaces the result (q_few).  Errors relative to a cell's sum of |w u| over the
// tiles of random plane waves on 64^2 .. 4096^2 grids against 64-bit mantissas, rms / worst: FP64 sum
// 4.5e-17 / 2.0e-16, this 0.1 - 0.6e-17 / 1.7e-16.
//
// Inside a solve no cell is looked at, and the form is plainer: q on 57 bits, 16 Lap and 8 Grad as whole
// numbers, A = a / 12, C = c / 12, B = 8 b / 144 as 62-bit integers (its shifts fold into adds, some six
// operations a cell fewer: star 1024^2 FP64 solve 4.06 ms, 4.14 with the form above; of the plane waves'
// cells 0.3 - 1.4e-17 / 1.0e-15).  Everywhere in the tile its error is below the FP64 rounding at the
// tile's largest value, which the max-norm of the residual and the elliptic coupling of the cells see
// just as well, and corrections that fall by decades within a tile are common on coarse levels (with
// the look at every cell that solve takes 12.7 ms).
//
// Tiles that hold an infinity or a NaN, or whose largest value is outside 2^-800 .. 2^700, take the
// FP64 sum, and so do operators with a coefficient outside 2^-100 .. 2^100.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define CCM_HD __host__ __device__ __forceinline__
#else
#define CCM_HD inline
#endif

namespace ccm {
namespace dev {

// coefficients times 2^k; the sum of the upper products times 2^(E - 1022 + cexp) is h^2 L u
struct QCoef {
  long long A = 0, C = 0, B = 0;
  int cexp = 0;
};

struct QStencil : QCoef {          // 16 a / 12, 16 c / 12, 64 b / 144 (FINE)
  QCoef plain;                     // a / 12, c / 12, 8 b / 144
  int ok = 0;                      // the coefficients are in range
  // least sum of |w u| over 2^s for which the integer form is as accurate as the FP64 sum, the
  // weights of the axis taps (centre, x +- 1, x +- 2, y +- 1, y +- 2), and the upper word of the
  // centre's q for which its term alone is as much
  float least = 0, wc = 0, wx1 = 0, wx2 = 0, wy1 = 0, wy2 = 0;
  unsigned near = 0;
};

// v_i 2^(bits - e) as integers, |v_i| < 2^e; false where e is out of range
inline bool q_coef(long double A, long double C, long double B, int bits, int qbits, QCoef& S, int& e) {
  long double m = std::fabs(A);
  if (std::fabs(C) > m) m = std::fabs(C);
  if (std::fabs(B) > m) m = std::fabs(B);
  if (!(m > 0) || !std::isfinite((double)m)) return false;
  std::frexp((double)m, &e);                    // m < 2^e (a rounding up to 2^e only widens it)
  if (e < -100 || e > 100) return false;
  const int k = bits - e;
  const auto fix = [&](long double v) {
    const long double t = std::ldexp(v, k);
    return t >= 9223372036854775807.0L ? 9223372036854775807LL : t <= -9223372036854775807.0L ? -9223372036854775807LL
                                                                                             : (long long)std::llround(t);
  };
  S.A = fix(A);
  S.C = fix(C);
  S.B = fix(B);
  S.cexp = 64 - k - qbits;
  return true;
}

inline QStencil q_stencil(double a, double b, double c) {
  QStencil S;
  int e = 0;
  const long double la = a, lb = b, lc = c;
  if (!q_coef(la / 12.0L, lc / 12.0L, lb / 18.0L, 62, 57, S.plain, e) ||
      !q_coef(16.0L * la / 12.0L, 16.0L * lc / 12.0L, 64.0L * lb / 144.0L, 63, 60, S, e))
    return S;
  S.ok = 1;
  // The bound on the error in units of 2^(s - 60): the values' rounding, half a unit in every tap
  // (64 / 12 in all along x and along y, 324 / 144 of the mixed term); the sixteenths' floors, times 16 / 12,
  // up along x and down along y; the eighths' (at most 1.125 and 1 units, times 64 / 144); the products'
  // floors, of 2^(1 + e): one down and one up, and another down with the mixed term.
  const double ax = std::fabs(a), cy = std::fabs(c), bm = std::fabs(b), n = std::ldexp(1.0, -e);
  const double bound = n * ((ax + cy) * 64 / 24 + (ax > cy ? ax : cy) * 16 / 12 + bm * (324.0 / 288 + 2.125 * 64 / 144)) +
                       (b != 0 ? 4.0 : 2.0);
  const double least = bound / (128.0 * 3);     // bound 2^-60 <= 3 2^-53 least, with 2^-e taken out
  S.least = (float)(least * 1.0001);             // (its own and the sums' roundings in FP32)
  S.wc = (float)(30.0 / 12 * n * std::fabs(a + c));
  S.wx1 = (float)(16.0 / 12 * n * ax);
  S.wx2 = (float)(1.0 / 12 * n * ax);
  S.wy1 = (float)(16.0 / 12 * n * cy);
  S.wy2 = (float)(1.0 / 12 * n * cy);
  const double near = S.wc > 0 ? std::ceil(S.least / S.wc * 268435456.0) : 4e9;     // |q| >= 2^32 near
  S.near = near < 4e9 ? (unsigned)near : 0xffffffffu;
  return S;
}

// the tile's scale from m, the largest q_word of its values: the exponent field (any for a tile
// of zeros), or -1 where the integer form does not apply
CCM_HD unsigned q_word(unsigned hi, unsigned lo) { return (hi & 0x7fffffffu) | (lo != 0 ? 1u : 0u); }
CCM_HD int q_scale(unsigned m, const QStencil& S) {
  const int E = m == 0 ? 220 : (int)(m >> 20);
  return (S.ok && E >= 220 && E <= 1720) ? E : -1;
}

// q of the double with words (hi, lo) at tile scale E (its exponent field is at most E)
template <bool FINE = true>
CCM_HD long long q_fixed(unsigned hi, unsigned lo, int E) {
  const unsigned mh = (hi << 11) | (lo >> 21) | 0x80000000u, ml = lo << 11;
  const unsigned long long m = ((unsigned long long)mh << 32) | ml;   // 1.f times 2^63
  const unsigned sh = (unsigned)(E - (int)((hi >> 20) & 0x7ffu)) + (FINE ? 3u : 6u);
  unsigned long long q;
#ifdef __CUDA_ARCH__
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(m), "r"(sh));            // 0 from 64 on (zeros: 220 and up)
#else
  q = sh < 64 ? m >> sh : 0;
#endif
  q = (q >> 1) + (q & 1);
  const long long s = (long long)((int)hi >> 31);
  return ((long long)q ^ s) - s;
}

// Lap, and (where it is not FINE, 16 times) as a whole number; Grad likewise, and its rounded eighth
template <bool FINE = true>
CCM_HD long long q_lap(long long m2, long long m1, long long c, long long p1, long long p2) {
  const long long c2 = c + c;
  return FINE ? (m1 + p1 - c2) - ((m2 + p2 - c2) >> 4) : (m1 + p1 - c2) * 16 - (m2 + p2 - c2);
}
template <bool FINE = true>
CCM_HD long long q_grad(long long m2, long long m1, long long p1, long long p2) {
  return FINE ? (p1 - m1) + ((m2 - p2) >> 3) : (m2 - p2) + (p1 - m1) * 8;
}
template <bool FINE = true>
CCM_HD long long q_grad8(long long m2, long long m1, long long p1, long long p2) {
  return FINE ? q_grad<true>(m2, m1, p1, p2) : (q_grad<false>(m2, m1, p1, p2) + 4) >> 3;
}
CCM_HD long long q_hi(long long x, long long y) {
#ifdef __CUDA_ARCH__
  return __mul64hi(x, y);
#else
  return (long long)(((__int128)x * y) >> 64);
#endif
}

// hi(A Lap_x) + hi(C Lap_y) from hx = hi(A Lap_x) and Lap_y of the negated values, so that the floors
// along y go up where those along x go down and cancel on average (and zeros give 0)
CCM_HD long long q_lap_neg(long long m2, long long m1, long long c, long long p1, long long p2) {
  const long long c2 = c + c;
  return (c2 - m1 - p1) - ((c2 - m2 - p2) >> 4);
}
CCM_HD long long q_axes(long long hx, long long neg_y, const QCoef& S) { return hx - q_hi(neg_y, S.C); }

// |q| 2^-60 from the upper word of q, rounded down (a lone unit of it is 2^-28)
CCM_HD float q_part(long long q) {
  const int v = (int)(q >> 32);
  return (float)(v ^ (v >> 31)) * 3.7252902984619140625e-9f;
}
// the sum of |w u| 2^-s over a cell's axis taps, a lower bound on all its taps' (c, and the sums of q_part at
// x +- 1, x +- 2, y +- 1, y +- 2)
CCM_HD float q_sum(const QStencil& S, float c, float x1, float x2, float y1, float y2) {
  return S.wc * c + S.wx1 * x1 + S.wx2 * x2 + S.wy1 * y1 + S.wy2 * y2;
}

// x times 2^e as a double, rounded to nearest (ties away), for e that keeps it in the normal range
CCM_HD double q_double(long long x, int e) {
  const long long s = x >> 63;
  unsigned long long m = (unsigned long long)((x ^ s) - s);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)m);
#else
  const int lz = m ? __builtin_clzll(m) : 64;
#endif
  if (lz > 63) return 0.0;
  m <<= lz;                                             // the leading bit at 63
  // exponent field 1023 + 63 - lz + e, less the leading bit that the mantissa adds to it
  unsigned long long b = ((unsigned long long)(unsigned)(1023 + 62 - lz + e) << 52) + (m >> 11) + ((m >> 10) & 1);
  b |= (unsigned long long)s & 0x8000000000000000ULL;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}

#ifdef __CUDACC__
// the largest exponent-and-mantissa word of a CTA's values (one per thread, 256 threads): every
// warp's maximum through wmax, which the next call may overwrite only after a later barrier
__device__ __forceinline__ unsigned q_cta_max(unsigned m, unsigned* wmax) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  const uint4 a = *reinterpret_cast<const uint4*>(wmax), b = *reinterpret_cast<const uint4*>(wmax + 4);
  return max(max(max(a.x, a.y), max(a.z, a.w)), max(max(b.x, b.y), max(b.z, b.w)));
}

// this thread's pairs threadIdx.x + 256 k of a staged tile of n pairs of doubles, and their largest
// word
template <int N>
struct QSlots {
  unsigned hi[2 * N], lo[2 * N];
  __device__ __forceinline__ unsigned load(const double* tile, int n) {
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int idx = threadIdx.x + 256 * k;
      const double2 v = idx < n ? *reinterpret_cast<const double2*>(tile + 2 * idx) : make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(j ? v.y : v.x);
        hi[2 * k + j] = (unsigned)(b >> 32);
        lo[2 * k + j] = (unsigned)b;
        m = max(m, q_word(hi[2 * k + j], lo[2 * k + j]));
      }
    }
    return m;
  }
  template <bool FINE>
  __device__ __forceinline__ void store(long long* q, int n, int E) const {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int idx = threadIdx.x + 256 * k;
      if (idx < n)
        *reinterpret_cast<longlong2*>(q + 2 * idx) =
            make_longlong2(q_fixed<FINE>(hi[2 * k], lo[2 * k], E), q_fixed<FINE>(hi[2 * k + 1], lo[2 * k + 1], E));
    }
  }
};

// The stencil sums (before the scale) of the cells (x0, y0 + k), (x0 + 1, y0 + k), k = 0 .. 3,
// x0 even, on a staged tile q [.][ROW] of integers whose cell (0, 0) is at (2, 2): two columns
// and four rows a thread, each staged row read as aligned pairs that serve both columns; the
// rows' Lap_x and Grad_x are formed as a row enters and kept until their cells are complete.
// emit(k, s0, s1).  With FINE the result says whether every cell's own value alone is large enough
// for the integer form (on the upper words, which are in registers: 2 operations a cell).
template <bool CROSS, int ROW, bool FINE, class Emit>
__device__ __forceinline__ bool q_rows(const long long* __restrict__ q, int x0, int y0, const QStencil& Q, Emit emit) {
  const QCoef& S = FINE ? static_cast<const QCoef&>(Q) : Q.plain;
  long long c[2][8], d[2][8], X[2][4];
  unsigned least = 0xffffffffu;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const longlong2* row = reinterpret_cast<const longlong2*>(q + (y0 + r) * ROW + x0);
    const longlong2 b = row[1];
    c[0][r] = b.x;
    c[1][r] = b.y;
    if (FINE && r >= 2 && r < 6) {
      const int v0 = (int)(b.x >> 32), v1 = (int)(b.y >> 32);
      least = min(least, min((unsigned)(v0 ^ (v0 >> 31)), (unsigned)(v1 ^ (v1 >> 31))));
    }
    if (CROSS || (r >= 2 && r < 6)) {
      const longlong2 a = row[0], e = row[2];
      if (CROSS) {
        d[0][r] = q_grad8<FINE>(a.x, a.y, b.y, e.x);
        d[1][r] = q_grad8<FINE>(a.y, b.x, e.x, e.y);
      }
      if (r >= 2 && r < 6) {
        X[0][r - 2] = q_hi(q_lap<FINE>(a.x, a.y, b.x, b.y, e.x), S.A);
        X[1][r - 2] = q_hi(q_lap<FINE>(a.y, b.x, b.y, e.x, e.y), S.A);
      }
    }
    if (r >= 4) {
      long long s[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const long long m2 = c[j][r - 4], m1 = c[j][r - 3], m = c[j][r - 2], p1 = c[j][r - 1], p2 = c[j][r];
        if (FINE) s[j] = q_axes(X[j][r - 4], q_lap_neg(m2, m1, m, p1, p2), S);
        else s[j] = X[j][r - 4] + q_hi(q_lap<false>(m2, m1, m, p1, p2), S.C);
        if (CROSS) s[j] += q_hi(q_grad<FINE>(d[j][r - 4], d[j][r - 3], d[j][r - 1], d[j][r]), S.B);
      }
      emit(r - 4, s[0], s[1]);
    }
  }
  return !FINE || least >= Q.near;
}

// Of these cells those whose sum of |w u| is too small for the integer form (bit 2 k + j: cell
// (x0 + j, y0 + k)), less those of `skip`: first from the integers, then, as the integers of small values
// are 0 too, without the cells whose taps are all 0 in the tile of doubles
template <bool CROSS, int ROW>
__device__ __forceinline__ unsigned q_few(const long long* __restrict__ q, const double* __restrict__ tile, int x0, int y0,
                                          const QStencil& S, unsigned skip) {
  float b[8][2], x1[4][2], x2[4][2];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const longlong2* row = reinterpret_cast<const longlong2*>(q + (y0 + r) * ROW + x0);
    const longlong2 m = row[1];
    b[r][0] = q_part(m.x);
    b[r][1] = q_part(m.y);
    if (r < 2 || r > 5) continue;
    const longlong2 a = row[0], e = row[2];
    const float a1 = q_part(a.y), e0 = q_part(e.x);
    x1[r - 2][0] = a1 + b[r][1];
    x1[r - 2][1] = b[r][0] + e0;
    x2[r - 2][0] = q_part(a.x) + e0;
    x2[r - 2][1] = a1 + q_part(e.y);
  }
  unsigned few = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (q_sum(S, b[k + 2][j], x1[k][j], x2[k][j], b[k + 1][j] + b[k + 3][j], b[k][j] + b[k + 4][j]) < S.least)
        few |= 1u << (2 * k + j);
  few &= ~skip;
  for (unsigned m = few; m; m &= m - 1) {
    const int t = __ffs(m) - 1;
    const double* c = tile + (y0 + (t >> 1) + 2) * ROW + x0 + (t & 1) + 2;
    bool any = c[0] != 0.0 || c[-1] != 0.0 || c[1] != 0.0 || c[-ROW] != 0.0 || c[ROW] != 0.0;
    if (!any)
#pragma unroll
      for (int dj = -2; dj <= 2; ++dj)
#pragma unroll
        for (int di = -2; di <= 2; ++di)
          if (CROSS || dj == 0 || di == 0) any |= c[dj * ROW + di] != 0.0;
    if (!any) few &= ~(1u << t);
  }
  return few;
}
#endif

}  // namespace dev
}  // namespace ccm
