"""The integer form of the regular stencil cell by cell (csrc/fixed.cuh, compiled for the host): every
cell's error against its own sum of |w u|, and against the FP64 sum's, on fields whose values span
many decades within a tile."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "fixed.cuh"
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
using namespace ccm::dev;
static unsigned hi(double x) { unsigned long long b; memcpy(&b, &x, 8); return (unsigned)(b >> 32); }
static unsigned lo(double x) { unsigned long long b; memcpy(&b, &x, 8); return (unsigned)b; }
static double u[36][68];
static long long q[36][68];
int main(int, char** v) {
  const double a = atof(v[1]), b = atof(v[2]), c = atof(v[3]);
  const int kind = atoi(v[4]);
  const QStencil S = q_stencil(a, b, c);
  const double lap[5] = {-1, 16, -30, 16, -1}, gra[5] = {1, -8, 0, 8, -1};
  std::mt19937_64 g(11);
  std::normal_distribution<double> N;
  std::uniform_real_distribution<double> U(0, 1);
  double worst = 0, worst64 = 0, plain = 0;
  long ints = 0, all = 0;
  for (int tile = 0; tile < (kind == 4 ? 200 : 4); ++tile) {
    const int n = 64 << (tile % 7);
    double am[6], kx[6], ky[6], ph[6];
    for (int k = 0; k < 6; ++k) { am[k] = N(g); kx[k] = 4 * M_PI * U(g); ky[k] = 4 * M_PI * (2 * U(g) - 1); ph[k] = 2 * M_PI * U(g); }
    unsigned m = 0;
    for (int j = 0; j < 36; ++j) for (int i = 0; i < 68; ++i) {
      const double x = i - 20.3 - 7 * tile, y = j - 13.7;
      double w = 0;
      for (int k = 0; k < 6; ++k) w += am[k] * std::sin(kx[k] * i / n + ky[k] * j / n + ph[k]);
      u[j][i] = kind == 0 ? std::exp(-(x * x + y * y) / 18) : kind == 1 ? w : kind == 2 ? std::exp(-0.8 * i) : kind == 3 ? N(g) * std::pow(10.0, -40 * U(g))
              : kind == 4 ? w : kind == 5 ? (i < 30 ? 0.0 : 1e-20 * (1 + i % 3)) : N(g);
    }
    if (kind == 1) u[17][31 + tile] = 1e18;
    if (kind == 5) u[9][5] = 1;
    double top = 0, sum = 0;
    for (auto& r : u) for (double x : r) { m = std::max(m, q_word(hi(x), lo(x))); top = std::max(top, std::fabs(x)); }
    for (int d = 0; d < 5; ++d) for (int e = 0; e < 5; ++e)
      sum += std::fabs(b * gra[d] * gra[e] / 144 + (d == 2 ? a * lap[e] / 12 : 0) + (e == 2 ? c * lap[d] / 12 : 0));
    const int E = q_scale(m, S);
    if (E < 0) return 2;
    for (int j = 0; j < 36; ++j) for (int i = 0; i < 68; ++i) q[j][i] = q_fixed(hi(u[j][i]), lo(u[j][i]), E);
    for (int j = 2; j < 34; ++j) for (int i = 2; i < 66; ++i) {
      const auto p = [&](int dj, int di) { return q_part(q[j + dj][i + di]); };
      const bool few = q_sum(S, p(0, 0), p(0, -1) + p(0, 1), p(0, -2) + p(0, 2), p(-1, 0) + p(1, 0), p(-2, 0) + p(2, 0)) < S.least;
      long double x = 0, terms = 0;
      double f = 0;
      for (int d = 0; d < 5; ++d) for (int e = 0; e < 5; ++e) {
        const long double w = (long double)b * gra[d] * gra[e] / 144 + (d == 2 ? (long double)a * lap[e] / 12 : 0) + (e == 2 ? (long double)c * lap[d] / 12 : 0);
        x += w * u[j + d - 2][i + e - 2];
        terms += fabsl(w * u[j + d - 2][i + e - 2]);
        f = std::fma((double)w, u[j + d - 2][i + e - 2], f);
      }
      ++all;
      if (terms > 0) worst64 = std::max(worst64, (double)(fabsl(f - x) / terms));
      // the plain form of the solves' passes: relative to the tile's largest value
      const auto P = [&](int dj, int di) { return q_fixed<false>(hi(u[j + dj][i + di]), lo(u[j + dj][i + di]), E); };
      long long ps = q_hi(q_lap<false>(P(0, -2), P(0, -1), P(0, 0), P(0, 1), P(0, 2)), S.plain.A) +
                     q_hi(q_lap<false>(P(-2, 0), P(-1, 0), P(0, 0), P(1, 0), P(2, 0)), S.plain.C);
      long long pd[5];
      for (int k = 0; k < 5; ++k) pd[k] = q_grad8<false>(P(k - 2, -2), P(k - 2, -1), P(k - 2, 1), P(k - 2, 2));
      if (b != 0) ps += q_hi(q_grad<false>(pd[0], pd[1], pd[3], pd[4]), S.plain.B);
      plain = std::max(plain, (double)(fabsl(q_double(ps, E - 1022 + S.plain.cexp) - x) / (top * sum)));
      if (few && terms > 0) continue;          // (a cell whose taps are all 0 keeps its integer result, 0)
      ++ints;
      const long long own = q[j][i] >> 32;
      if (few && (unsigned)(own ^ (own >> 63)) >= S.near) return 4;      // the quick test lets no such cell pass
      long long s = q_axes(q_hi(q_lap(q[j][i - 2], q[j][i - 1], q[j][i], q[j][i + 1], q[j][i + 2]), S.A),
                           q_lap_neg(q[j - 2][i], q[j - 1][i], q[j][i], q[j + 1][i], q[j + 2][i]), S);
      long long d[5];
      for (int k = 0; k < 5; ++k) d[k] = q_grad8(q[j + k - 2][i - 2], q[j + k - 2][i - 1], q[j + k - 2][i + 1], q[j + k - 2][i + 2]);
      if (b != 0) s += q_hi(q_grad(d[0], d[1], d[3], d[4]), S.B);
      const double r = q_double(s, E - 1022 + S.cexp);
      if (terms == 0) { if (r != 0) return 3; continue; }
      worst = std::max(worst, (double)(fabsl(r - x) / terms));
    }
  }
  printf("%.17g %.17g %.17g %.17g\n", worst, worst64, (double)ints / all, plain);
}
'''


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("local")
    (d / "h.cpp").write_text(SRC)
    inc = os.path.join(ROOT, "paper_2504_00724_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", inc, str(d / "h.cpp"), "-o", str(d / "h")], check=True)
    return str(d / "h")


# a Gaussian of 3 cells' width, a spike of 1e18 in a smooth field, e^(-0.8 i), 40 decades at random,
# smooth fields, tiny values beside zeros and a one, N(0, 1)
@pytest.mark.parametrize("abc", [(1, 0, 1), (1, 0.5, 2), (1.25, -0.8660254037844386, 1.75), (1, 0, 1e-3), (1e-3, 1e-4, 1e3)])
@pytest.mark.parametrize("kind", range(7))
def test_every_cell_is_as_accurate_as_its_fp64_sum(harness, abc, kind):
    out = subprocess.run([harness, *map(repr, map(float, abc)), str(kind)], capture_output=True, text=True, check=True).stdout
    worst, worst64, share, plain = map(float, out.split())
    # the bound of the integer form, and the rounding of its result
    assert worst <= (3 + 1) * 2.0 ** -53
    assert worst <= max(1.5 * worst64, 2.5e-16)     # the FP64 sum's worst cell on the same field: 1 to 2.5e-16
    # values to 2^-58, the eighth, three floors, and the rounding of the result
    assert plain <= 1.1 * 2.0 ** -53
    if kind in (4, 6):
        assert share >= 0.97                        # and it is the form that is used
