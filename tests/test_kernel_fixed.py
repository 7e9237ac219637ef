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

FACE = r"""
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
static Q paper(const Q *d) {  // f - v2, eq. (11)-(22), p = 1, the sensitivity term left out
  Q s[4], t[4] = {3 * d[1] - d[0], d[1] + d[2], 3 * d[2] - d[3], 3 * d[4] - 5 * d[3]}, b[4];
  for (int k = 0; k < 4; ++k) s[k] = d[k + 1] - d[k];
  for (int k = 0; k < 4; ++k) b[k] = (Q)13 / 3 * s[k] * s[k] + t[k] * t[k];
  b[3] = (b[0] + b[1] + b[2] + b[3]) / 4;
  const Q r5 = s[3] - s[0] + 3 * (s[1] - s[2]), T = 4 * r5 * r5, D[4] = {1, 9, 9, 1};
  const Q r[4] = {5 * d[1] - 2 * d[0], d[1] + 2 * d[2], 4 * d[2] - d[3], 6 * d[2] - 5 * d[3] + 2 * d[4]};
  Q num = 0, den = 0;
  for (int k = 0; k < 4; ++k) { const Q a = D[k] * (1 + T / (b[k] + (Q)1e-80)); num += a * r[k]; den += a; }
  return num / den / 6;
}
int main(int argc, char **argv) {
  const int jump = atoi(argv[1]);
  const double phase = atof(argv[2]), cold = atof(argv[3]);
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> U(-1, 1);
  double worst = 0;
  long smooths = 0, fields = 0;
  for (int it = 0; it < 4000; ++it) {
    const double gm1 = 0.4, un = U(g), ut = U(g), c = cold * (1 + 0.5 * U(g)), ic = 1 / c;
    const double b1 = gm1 * ic * ic, b2 = b1 * 0.5 * (un * un + ut * ut);
    const double A[4] = {1.2 * (std::fabs(un) + c), std::fabs(un) + 0.1, std::fabs(un) + 0.1, 1.2 * (std::fabs(un) + c)};
    const double ph = 3 * U(g), a1 = 0.2 * U(g), a2 = 0.2 * U(g), jr = 0.5 * U(g), jp = 0.5 * U(g);
    double V[4][6], F[4][6];
    for (int j = 0; j < 6; ++j) {
      const double s1 = a1 * std::sin(ph + phase * j), s2 = a2 * std::cos(2 * ph + 0.7 * phase * j);
      const bool on = jump && j > it % 5;
      const double rho = 1 + s1 + (on ? jr : 0), u = un + c * s2, v = ut + c * s1;
      const double p = c * c / 1.4 * (1 + s2 + (on ? jp : 0)), E = p / gm1 + 0.5 * rho * (u * u + v * v);
      V[0][j] = rho; V[1][j] = rho * u; V[2][j] = rho * v; V[3][j] = E;
      F[0][j] = V[1][j]; F[1][j] = V[1][j] * u + p; F[2][j] = V[2][j] * u; F[3][j] = (E + p) * u;
    }
    const int a = exponent(std::fmax(A[0], A[1])) - 1022;
    double dU[4][5], dF[4][5];
    u64 pU[4][5], pF[4][5];
    int E[4];
    for (int q = 0; q < 4; ++q) {
      int eu = 0, ef = 0;
      for (int j = 0; j < 5; ++j) {
        pU[q][j] = pack(dU[q][j] = V[q][j + 1] - V[q][j]);
        pF[q][j] = pack(dF[q][j] = F[q][j + 1] - F[q][j]);
        eu = imax(eu, packed_exponent(pU[q][j]));
        ef = imax(ef, packed_exponent(pF[q][j]));
      }
      E[q] = imax(eu, ef - a);
    }
    const double t1 = un * ic, t2 = b1 * un, t3 = b1 * ut;
    const LeftRows<4> rows = left_rows<4>(E, b2, b1, t1, t2, t3, ic, ut);
    Proj PU[5], PF[5];
    i64 wu[5], wf[5];
    for (int j = 0; j < 5; ++j) {
      u64 v[4];
      for (int q = 0; q < 4; ++q) v[q] = pU[q][j];
      PU[j] = project<4>(rows, E, 0, v);
      for (int q = 0; q < 4; ++q) v[q] = pF[q][j];
      PF[j] = project<4>(rows, E, a, v);
      wu[j] = project_shear(rows, E, 0, pU[0][j], pU[2][j]);
      wf[j] = project_shear(rows, E, a, pF[0][j], pF[2][j]);
    }
    double h[4], top = 0;
    Q ref[4];
    for (int m = 0; m < 4; ++m) {
      auto part = [&](const Proj &p) { return m == 0 ? p.z + p.tc : m == 1 ? p.r - p.z : p.z - p.tc; };
      i64 x[5], y[5];
      for (int j = 0; j < 5; ++j) x[j] = times_speed(speed(A[m], a), m == 2 ? wu[j] : part(PU[j])), y[j] = m == 2 ? wf[j] : part(PF[j]);
      const int k0 = (m == 2 ? rows.us : rows.um) + a - 1592;
      i64 d[5], e[5];
      for (int j = 0; j < 5; ++j) d[j] = (x[j] + y[j]) >> 2, e[4 - j] = (x[j] - y[j]) >> 2;
      int cp, cm;
      const bool sp = smooth_term<false>(d, cp), sm = smooth_term<false>(e, cm);
      ++fields;
      smooths += sp && sm;
      h[m] = 0;
      if (sp && sm) {
        h[m] = from_fixed(smooth_sum(y, cp + cm), k0 + 2) / 6;
      } else {
        const int n = field_shift(x, y);
        shift_field(x, n);
        shift_field(y, n);
        const i64 S = rough_sum(x, y, [](const i64(&d)[5]) {
          return recon6<false>(d[0], d[1], d[2], d[3], d[4], Flt()); });
        h[m] = from_fixed(S, k0 + 6 - n) / 6;
      }
      Q row[4] = {0, 0, 0, 0}, P[5], N[5], X2 = 0;
      if (m == 0 || m == 3) { const Q s = m ? -1 : 1; row[0] = b2 + s * t1; row[1] = -t2 - s * ic; row[2] = -(Q)t3; row[3] = b1; }
      if (m == 1) { row[0] = 1 - (Q)b2; row[1] = t2; row[2] = t3; row[3] = -b1; }
      if (m == 2) { row[0] = -ut; row[2] = 1; }
      for (int j = 0; j < 5; ++j) {
        Q w = 0, f = 0;
        for (int q = 0; q < 4; ++q) {
          w += row[q] * dU[q][j];
          f += row[q] * dF[q][j];
          top = std::fmax(top, (double)qabs(A[m] * row[q] * dU[q][j]));
        }
        if (j == 2) X2 = A[m] * w;
        P[j] = A[m] * w + f;
        N[4 - j] = A[m] * w - f;
      }
      ref[m] = -X2 + paper(P) + paper(N);
    }
    for (int m = 0; m < 4; ++m) worst = std::fmax(worst, (double)(qabs((Q)h[m] - ref[m]) / top));
  }
  printf("%.17g %.17g\n", worst, (double)smooths / fields);
}
"""


@pytest.fixture(scope="module")
def face_harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("face")
    (d / "f.cpp").write_text(FACE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "paper_2603_26272_gb300", "csrc"), str(d / "f.cpp"), "-o",
                    str(d / "f")], check=True)
    return str(d / "f")


@pytest.mark.parametrize("cold", [1.0, 1e-3])
@pytest.mark.parametrize("jump,phase", [(0, 0.01), (0, 0.08), (0, 0.3), (0, 1.5), (1, 0.01), (1, 0.3)])
def test_projected_face_against_quadruple_precision(face_harness, jump, phase, cold):
    """The four fields of Euler faces from packed differences: projection,
    smooth test and weights together, at phases per cell where all, some and
    none of the fields pass the smooth test.  Tolerance: that of the
    reconstruction, 2^-50, relative to the largest alpha L dU term of the face."""
    out = subprocess.run([face_harness, str(jump), repr(phase), repr(cold)], check=True,
                         capture_output=True, text=True).stdout.split()
    assert float(out[0]) <= 2.0 ** -50
    assert (float(out[1]) > 0.5) == (phase < 0.1 and not jump)
