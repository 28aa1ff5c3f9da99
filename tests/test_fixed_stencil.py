"""The integer form of the regular stencil (csrc/fixed.cuh), compiled for the host: against the
FP64 sum it replaces, over value ranges, coefficients and the values at which it gives way."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include "fixed.cuh"
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
using namespace ccm::dev;
static unsigned hi(double x) { unsigned long long b; memcpy(&b, &x, 8); return (unsigned)(b >> 32); }
static unsigned lo(double x) { unsigned long long b; memcpy(&b, &x, 8); return (unsigned)b; }
int main(int, char** v) {
  const double a = atof(v[1]), b = atof(v[2]), c = atof(v[3]);
  const int kind = atoi(v[4]);
  std::mt19937_64 g(7);
  std::normal_distribution<double> N;
  std::uniform_real_distribution<double> U(0, 1);
  static double u[36][68];
  for (auto& r : u) for (double& x : r)
    x = kind == 0 ? N(g) : kind == 1 ? N(g) * std::pow(10.0, -16 * U(g)) : kind == 2 ? 1e-250 * N(g) : kind == 3 ? 0.0
      : kind == 4 ? 1e200 * N(g) : kind == 5 ? (U(g) < 0.5 ? 1.0 : -1.0) * (2 - 1e-16) : N(g);
  if (kind == 6) u[20][30] = INFINITY;
  if (kind == 7) u[20][30] = NAN;
  const QStencil S = q_stencil(a, b, c);
  unsigned m = 0;
  for (auto& r : u) for (double x : r) m = std::max(m, q_word(hi(x), lo(x)));
  const int E = q_scale(m, S);
  if (E < 0) { printf("fp64\n"); return 0; }
  static long long q[36][68];
  double top = 0;
  for (int j = 0; j < 36; ++j) for (int i = 0; i < 68; ++i) { q[j][i] = q_fixed(hi(u[j][i]), lo(u[j][i]), E); top = std::max(top, std::fabs(u[j][i])); }
  const long double L[5] = {-1, 16, -30, 16, -1}, G[5] = {1, -8, 0, 8, -1};
  double worst = 0, sum = 0;
  for (int d = 0; d < 5; ++d) for (int e = 0; e < 5; ++e)
    sum += std::fabs((double)(b * G[d] * G[e] / 144 + (d == 2 ? a * L[e] / 12 : 0) + (e == 2 ? c * L[d] / 12 : 0)));
  for (int j = 2; j < 34; ++j) for (int i = 2; i < 66; ++i) {
    long double x = 0;
    for (int d = 0; d < 5; ++d) for (int e = 0; e < 5; ++e)
      x += (b * G[d] * G[e] / 144 + (d == 2 ? a * L[e] / 12 : 0) + (e == 2 ? c * L[d] / 12 : 0)) * u[j + d - 2][i + e - 2];
    long long s = q_hi(q_lap(q[j][i - 2], q[j][i - 1], q[j][i], q[j][i + 1], q[j][i + 2]), S.A) +
                  q_hi(q_lap(q[j - 2][i], q[j - 1][i], q[j][i], q[j + 1][i], q[j + 2][i]), S.C);
    long long d[5];
    for (int k = 0; k < 5; ++k) d[k] = q_grad8(q[j + k - 2][i - 2], q[j + k - 2][i - 1], q[j + k - 2][i + 1], q[j + k - 2][i + 2]);
    s += q_hi(q_grad(d[0], d[1], d[3], d[4]), S.B);
    worst = std::max(worst, (double)std::fabs((long double)q_double(s, E - 1022 + S.cexp) - x));
  }
  printf("%.17g\n", top > 0 ? worst / (top * sum) : worst);
}
'''


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "h.cpp").write_text(SRC)
    inc = os.path.join(ROOT, "paper_2504_00724_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", inc, str(d / "h.cpp"), "-o", str(d / "h")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("abc", [(1, 0, 1), (1, 0.5, 2), (1.25, -0.8660254037844386, 1.75), (1e-3, 1e-4, 1e3), (1e20, 0, 1e20)])
@pytest.mark.parametrize("kind", range(8))
def test_integer_form_against_extended_precision(harness, abc, kind):
    out = subprocess.run([harness, *map(repr, map(float, abc)), str(kind)], capture_output=True, text=True, check=True).stdout.strip()
    if kind in (2, 6, 7):         # below the range, an infinity, a NaN: the FP64 sum
        assert out == "fp64"
        return
    # relative to the sum of |weights| times the tile's largest value: the values' rounding 2^-58,
    # three floors of 2^-61 .. 2^-58, the result's rounding 2^-53; extended precision itself 2^-60
    assert float(out) <= 2.0 ** -53 * 1.1


def test_operators_outside_the_coefficient_range_take_the_fp64_sum(harness):
    out = subprocess.run([harness, "1e40", "0", "1e40", "0"], capture_output=True, text=True, check=True).stdout.strip()
    assert out == "fp64"
