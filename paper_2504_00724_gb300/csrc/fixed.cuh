// The FP64 regular stencil (Sec. 3.2) in 64-bit integer arithmetic.
//
// GB300 issues FP64 at 2 FMA per clock per SM, 1/64 of the FP32 rate: a warp-wide FP64 FMA
// occupies its scheduler's pipe for 64 clocks, and the 17 FMA of the factored 25-tap stencil
// bound every FP64 pass over a level (9.4 us per 64 x 32 tile and SM).  Integer adds run at
// half the FP32 rate or better, so the stencil runs on fixed-point images of the staged values:
//
//   q = round(u 2^(57 - s)),  2^s the power of two above the largest |u| of the staged tile,
//   Lap  = 16 (q_-1 + q_+1) - (q_-2 + q_+2) - 30 q_0      (eq. stdLap times 12; |Lap| < 2^63),
//   Grad = (q_-2 - q_+2) + 8 (q_+1 - q_-1)                (eq. stdGrad times 12),
//   h^2 L u = 2^.. (hi(A Lap_x) + hi(C Lap_y) + hi(B Grad_y(Grad_x / 8))),
//
// with A = a / 12, C = c / 12, B = 8 b / 144 as 62-bit integers on one common power of two and
// hi() the upper half of the 128-bit product.  Lap and Grad are exact in q; what is rounded is
// q (to 2^-58 of the tile's largest value; a value within 2^4 of the largest not at all),
// Grad_x / 8, the three products and the conversion to FP64, each below that.  The FP64 sum
// rounds every partial sum to 2^-53 of terms of the size of 30/12 u.  Errors against 128-bit
// sums, relative 2-norm, FP64 / integer: plane waves 4e-12 / 6e-14, N(0, 1) values 1.6e-16 /
// 4.8e-17, values that fall by e^40 over the tile 9.2e-16 / 9.4e-16.  Where |u| in a cell's
// window is far below the tile's largest value the error stays 2^-58 of that value.  Tiles
// that hold an infinity or a NaN, or whose largest value is outside 2^-800 .. 2^700, take the
// FP64 sum, and so do operators with a coefficient outside 2^-100 .. 2^100.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define CCM_HD __host__ __device__ __forceinline__
#else
#define CCM_HD inline
#endif

namespace ccm {
namespace dev {

struct QStencil {
  long long A = 0, C = 0, B = 0;   // a / 12, c / 12, b / 18 times 2^k
  int cexp = 0;                    // the sum of the upper products times 2^(E - 1022 + cexp) is h^2 L u
  int ok = 0;                      // the coefficients are in range
};

inline QStencil q_stencil(double a, double b, double c) {
  QStencil S;
  const long double A = (long double)a / 12.0L, C = (long double)c / 12.0L, B = (long double)b / 18.0L;
  long double m = std::fabs(A);
  if (std::fabs(C) > m) m = std::fabs(C);
  if (std::fabs(B) > m) m = std::fabs(B);
  if (!(m > 0) || !std::isfinite((double)m)) return S;
  int e = 0;
  std::frexp((double)m, &e);                    // m < 2^e (a rounding up to 2^e only widens it)
  if (e < -100 || e > 100) return S;
  const int k = 62 - e;
  S.A = (long long)std::llround(std::ldexp(A, k));
  S.C = (long long)std::llround(std::ldexp(C, k));
  S.B = (long long)std::llround(std::ldexp(B, k));
  S.cexp = 64 - k - 57;
  S.ok = 1;
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
CCM_HD long long q_fixed(unsigned hi, unsigned lo, int E) {
  const unsigned mh = (hi << 11) | (lo >> 21) | 0x80000000u, ml = lo << 11;
  const unsigned long long m = ((unsigned long long)mh << 32) | ml;   // 1.f times 2^63
  const unsigned sh = (unsigned)(E - (int)((hi >> 20) & 0x7ffu)) + 6u;
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

CCM_HD long long q_lap(long long m2, long long m1, long long c, long long p1, long long p2) {
  const long long c2 = c + c;
  return (m1 + p1 - c2) * 16 - (m2 + p2 - c2);
}
CCM_HD long long q_grad(long long m2, long long m1, long long p1, long long p2) { return (m2 - p2) + (p1 - m1) * 8; }
CCM_HD long long q_grad8(long long m2, long long m1, long long p1, long long p2) {   // rounded eighth
  return (q_grad(m2, m1, p1, p2) + 4) >> 3;
}
CCM_HD long long q_hi(long long x, long long y) {
#ifdef __CUDA_ARCH__
  return __mul64hi(x, y);
#else
  return (long long)(((__int128)x * y) >> 64);
#endif
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
  __device__ __forceinline__ void store(long long* q, int n, int E) const {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int idx = threadIdx.x + 256 * k;
      if (idx < n)
        *reinterpret_cast<longlong2*>(q + 2 * idx) =
            make_longlong2(q_fixed(hi[2 * k], lo[2 * k], E), q_fixed(hi[2 * k + 1], lo[2 * k + 1], E));
    }
  }
};

// The stencil sums (before the scale) of the cells (x0, y0 + k), (x0 + 1, y0 + k), k = 0 .. 3,
// x0 even, on a staged tile q [.][ROW] of integers whose cell (0, 0) is at (2, 2): two columns
// and four rows a thread, each staged row read as aligned pairs that serve both columns; the
// rows' Lap_x and Grad_x are formed as a row enters and kept until their cells are complete.
// emit(k, s0, s1).
template <bool CROSS, int ROW, class Emit>
__device__ __forceinline__ void q_rows(const long long* __restrict__ q, int x0, int y0, const QStencil& S, Emit emit) {
  long long c[2][8], d[2][8], X[2][4];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const longlong2* row = reinterpret_cast<const longlong2*>(q + (y0 + r) * ROW + x0);
    const longlong2 b = row[1];
    c[0][r] = b.x;
    c[1][r] = b.y;
    if (CROSS || (r >= 2 && r < 6)) {
      const longlong2 a = row[0], e = row[2];
      if (CROSS) {
        d[0][r] = q_grad8(a.x, a.y, b.y, e.x);
        d[1][r] = q_grad8(a.y, b.x, e.x, e.y);
      }
      if (r >= 2 && r < 6) {
        X[0][r - 2] = q_hi(q_lap(a.x, a.y, b.x, b.y, e.x), S.A);
        X[1][r - 2] = q_hi(q_lap(a.y, b.x, b.y, e.x, e.y), S.A);
      }
    }
    if (r >= 4) {
      long long s[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        s[j] = X[j][r - 4] + q_hi(q_lap(c[j][r - 4], c[j][r - 3], c[j][r - 2], c[j][r - 1], c[j][r]), S.C);
        if (CROSS) s[j] += q_hi(q_grad(d[j][r - 4], d[j][r - 3], d[j][r - 1], d[j][r]), S.B);
      }
      emit(r - 4, s[0], s[1]);
    }
  }
}
#endif

}  // namespace dev
}  // namespace ccm
