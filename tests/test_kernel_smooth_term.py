"""smooth_term of csrc/weno_fixed.cuh alone, compiled for the host, against
128-bit floating point: polynomial stencils of degree 2 to 4 with critical
points anywhere (the fifth difference is then 0, a few units, or far below the
second differences), sines, and polynomials with a jump.

Tolerance, wherever the term is accepted: its FP32 error, 2^-21 of a product of
at most 2^26 / 20 units, 1.6, and half a unit for the rounding to an integer.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "weno_fixed.cuh"
#ifdef __x86_64__
typedef __float128 Q;
#else
typedef long double Q;
#endif
using namespace weno::fx;
// sum_k D_k G_k (r_k - rm) / (20 + sum_k D_k G_k), exactly
static Q term(const i64 *i) {
  Q d[5];
  for (int k = 0; k < 5; ++k) d[k] = (Q)i[k];
  Q s[4], t[4] = {3 * d[1] - d[0], d[1] + d[2], 3 * d[2] - d[3], 3 * d[4] - 5 * d[3]}, b[4];
  for (int k = 0; k < 4; ++k) s[k] = d[k + 1] - d[k];
  for (int k = 0; k < 4; ++k) b[k] = (Q)13 / 3 * s[k] * s[k] + t[k] * t[k];
  b[3] = (b[0] + b[1] + b[2] + b[3]) / 4;
  const Q r5 = s[3] - s[0] + 3 * (s[1] - s[2]), D[4] = {1, 9, 9, 1};
  const Q r[4] = {5 * d[1] - 2 * d[0], d[1] + 2 * d[2], 4 * d[2] - d[3], 6 * d[2] - 5 * d[3] + 2 * d[4]};
  const Q rm = (r[0] + 9 * r[1] + 9 * r[2] + r[3]) / 20;
  Q num = 0, den = 20;
  for (int k = 0; k < 4; ++k) {
    const Q a = D[k] * (4 * r5 * r5 / (b[k] + (Q)1e-30));
    num += a * (r[k] - rm);
    den += a;
  }
  return num / den;
}
int main(int argc, char **argv) {
  const int kind = atoi(argv[1]);
  std::mt19937_64 g(7 + kind);
  std::uniform_real_distribution<double> U(-1, 1);
  double worst = 0;
  long taken = 0;
  for (int it = 0; it < 300000; ++it) {
    double c[5], w[6], mx = 0;
    for (double &x : c) x = U(g);
    const double x0 = 3 * U(g), th = std::pow(10.0, -2 + 2 * U(g)), top = std::pow(2.0, 52 + 7 * U(g));
    if (it % 3 == 0) c[1] = 0;
    for (int j = 0; j < 6; ++j) {
      const double x = x0 + j - 2.5;
      double p = 0;
      for (int k = 4; k >= 0; --k) p = p * x + (k <= kind ? c[k] : 0);
      if (kind >= 5) p = std::sin(th * x + 3 * c[0]);
      w[j] = p + (kind == 6 && j > it % 5 ? c[1] : 0);
    }
    for (int j = 0; j < 5; ++j) mx = std::fmax(mx, std::fabs(w[j + 1] - w[j]));
    if (mx == 0) continue;
    i64 v[6], d[5];
    for (int j = 0; j < 6; ++j) v[j] = (i64)(w[j] / mx * top);
    if (it % 2 == 0 && kind < 5) {  // exactly polynomial: the fifth difference is 0 (a third one, kind 2, 0)
      const i64 a = (i64)(top / 64 * c[3]), b = (i64)(top / 64 * c[2]), e = (i64)(top / 64 * c[4]), s = it % 10;
      for (int j = 0; j < 5; ++j) d[j] = (kind > 2 ? a * j * (j - 1) / 2 : 0) + b * (j - s) + (it % 4 ? e : 0);
    } else {
      for (int j = 0; j < 5; ++j) d[j] = v[j + 1] - v[j];
    }
    int corr;
    if (!smooth_term<false>(d, corr)) continue;
    ++taken;
    const Q off = term(d) - (Q)corr;
    worst = std::fmax(worst, (double)(off < 0 ? -off : off));
  }
  printf("%.17g %ld\n", worst, taken);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("smooth")
    (d / "s.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "paper_2603_26272_gb300", "csrc"), str(d / "s.cpp"), "-o",
                    str(d / "s")], check=True)
    return str(d / "s")


KINDS = {2: "quadratic", 3: "cubic", 4: "quartic", 5: "sine", 6: "sine_and_jump"}


@pytest.mark.parametrize("kind", KINDS, ids=KINDS.values())
def test_smooth_term_is_good_to_its_bound(harness, kind):
    worst, taken = subprocess.run([harness, str(kind)], check=True, capture_output=True,
                                  text=True).stdout.split()
    assert int(taken) > (0 if kind == 6 else 1000)
    assert float(worst) <= 2.1
