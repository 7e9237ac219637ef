"""The integer-pipe reconstruction (csrc/weno_fixed.cuh), compiled for the host
and compared with the paper's formulas (eqs. (11)-(22), p = 1) in 128-bit
floating point.

Tolerance, in units of 2^-57 of the largest of the ten differences: truncating
two differences (2 units) into candidates whose coefficients add up to 13, over
6, in both fluxes: 9; an indicator and its reciprocal good to 2^-54 (8 units)
on candidates up to 13/6 apart, in both fluxes: 35; the FP64 rounding of a
result of up to 4: 32.  Together below 128 units, 2^-50.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <cmath>
#include "weno_fixed.cuh"
#ifdef __x86_64__
typedef __float128 Q;
#else
typedef long double Q;
#endif
using namespace weno::fx;
static Q qabs(Q x) { return x < 0 ? -x : x; }
static Q paper(const Q *d, Q eps4, Q mu0, bool ai) {  // f - v2
  Q v[6] = {-d[0] - d[1], -d[1], 0, d[2], d[2] + d[3], d[2] + d[3] + d[4]}, m = 0, dev = 0;
  for (int j = 0; j < 6; ++j) m += v[j] / 6;
  for (int j = 0; j < 6; ++j) dev += qabs(v[j] - m);
  const Q mu = ai ? dev / 6 + mu0 : 1, e = eps4 * mu * mu;
  Q s[4], t[4] = {3 * d[1] - d[0], d[1] + d[2], 3 * d[2] - d[3], 3 * d[4] - 5 * d[3]}, b[4];
  for (int k = 0; k < 4; ++k) s[k] = d[k + 1] - d[k];
  for (int k = 0; k < 4; ++k) b[k] = (Q)13 / 3 * s[k] * s[k] + t[k] * t[k];
  b[3] = (b[0] + b[1] + b[2] + b[3]) / 4;
  const Q r5 = s[3] - s[0] + 3 * (s[1] - s[2]), T = 4 * r5 * r5, D[4] = {1, 9, 9, 1};
  const Q r[4] = {5 * d[1] - 2 * d[0], d[1] + 2 * d[2], 4 * d[2] - d[3], 6 * d[2] - 5 * d[3] + 2 * d[4]};
  Q num = 0, den = 0;
  for (int k = 0; k < 4; ++k) { const Q a = D[k] * (1 + T / (b[k] + e)); num += a * r[k]; den += a; }
  return num / den / 6;
}
// eps4 = 4 eps in the data's units; mode 0: left out, 1: added (Ai), 2: added (no Ai)
int main(int argc, char **argv) {
  const int kind = atoi(argv[1]), mode = atoi(argv[2]);
  const double eps4 = atof(argv[3]);
  std::mt19937_64 g(11 + kind);
  std::uniform_real_distribution<double> U(-1, 1);
  double worst = 0;
  for (int it = 0; it < 40000; ++it) {
    double xw[5], dg[5], mx = 0;
    const double sc = mode == 2 ? 1.0 : std::pow(10.0, 12 * U(g));
    const double ph = 3.2 * U(g), th = std::pow(10.0, -2 + 2 * U(g)), am = U(g);
    for (int j = 0; j < 5; ++j) {
      const double sm = am * (std::sin(ph + th * (j + 1)) - std::sin(ph + th * j));
      const bool at = j == it % 5;
      if (kind == 0) xw[j] = U(g), dg[j] = U(g);
      if (kind == 1) xw[j] = sm, dg[j] = 0.3 * sm;
      if (kind == 2) xw[j] = at ? 1.3 : 0, dg[j] = at ? ph : 0;
      if (kind == 3) xw[j] = sm + (at ? 1.3 : 0), dg[j] = -0.4 * sm + (at ? ph : 0);
      if (kind == 4) xw[j] = U(g), dg[j] = xw[j] * (1 + 1e-14 * U(g));
      if (kind == 5) xw[j] = (at ? 1.3 : 1e-16 * std::round(4 * U(g))), dg[j] = (at ? ph : 0);
      xw[j] *= sc;
      dg[j] *= sc;
      mx = std::fmax(mx, std::fmax(std::fabs(xw[j]), std::fabs(dg[j])));
    }
    if (mx == 0) continue;
    const int es = top_exponent(xw, dg);
    i64 p[5], n[5];
    Q qp[5], qn[5];
    for (int j = 0; j < 5; ++j) {
      const i64 x = to_fixed(xw[j], es), y = to_fixed(dg[j], es);
      p[j] = x + y; n[4 - j] = x - y;
      qp[j] = (Q)xw[j] + dg[j]; qn[4 - j] = (Q)xw[j] - dg[j];
    }
    const double mu0 = 2e-40;
    auto sens = [&](const Q *d) {  // 3 eps4 mu^2 in units squared
      double mu = 1;
      if (mode == 1) {
        Q v[6] = {-d[0] - d[1], -d[1], 0, d[2], d[2] + d[3], d[2] + d[3] + d[4]}, m = 0, dev = 0;
        for (int j = 0; j < 6; ++j) m += v[j] / 6;
        for (int j = 0; j < 6; ++j) dev += qabs(v[j] - m);
        mu = (double)(dev / 6 + mu0);
      }
      const u64 b = dbits(3 * eps4 * mu * mu);
      Flt e = {(b << 11) | 0x8000000000000000ull, (int)(b >> 52) - 1086 - 2 * (es - 1079)};
      return e;
    };
    i64 c;
    if (mode == 0)
      c = recon6<false>(p[0], p[1], p[2], p[3], p[4], Flt()) + recon6<false>(n[0], n[1], n[2], n[3], n[4], Flt());
    else
      c = recon6<true>(p[0], p[1], p[2], p[3], p[4], sens(qp)) + recon6<true>(n[0], n[1], n[2], n[3], n[4], sens(qn));
    const double h = std::fma((double)c, scale_back(es), -xw[2]);
    const Q ref = -(Q)xw[2] + paper(qp, eps4, mu0, mode != 2) + paper(qn, eps4, mu0, mode != 2);
    worst = std::fmax(worst, (double)(qabs((Q)h - ref) / mx));
  }
  double rw = 0;  // the reciprocal: below 2^127 / X by at most 2^-60 of it
  for (int it = 0; it < 200000; ++it) {
    u64 X = it < 64 ? (1ull << 63) | (it ? 1ull << (it - 1) : 0) : (it < 128 ? ~(u64)0 << (it - 64) | 1ull << 63 : (u64)g() | 1ull << 63);
    const Q exact = (Q)9223372036854775808.0 * (Q)18446744073709551616.0 / (Q)X;
    const Q off = (exact - (Q)rcp64(X)) / exact;
    if (off < 0) rw = 1;
    rw = std::fmax(rw, (double)off);
  }
  printf("%.17g %.17g\n", worst, rw);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fixed")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "paper_2603_26272_gb300", "csrc"), str(d / "h.cpp"), "-o",
                    str(d / "h")], check=True)
    return str(d / "h")


KINDS = ["random", "smooth", "jump", "jump_on_smooth", "cancelling", "jump_on_noise"]


@pytest.mark.parametrize("mode,eps4", [(0, 4e-40), (1, 4e-40), (1, 4e-12), (1, 4e-2), (2, 4e-40), (2, 4e-6)])
@pytest.mark.parametrize("kind", range(len(KINDS)), ids=KINDS)
def test_reconstruction_against_quadruple_precision(harness, kind, mode, eps4):
    out = subprocess.run([harness, str(kind), str(mode), repr(eps4)], check=True,
                         capture_output=True, text=True).stdout.split()
    assert float(out[0]) <= 2.0 ** -50
    assert float(out[1]) <= 2.0 ** -60
