"""The integer path of csrc/weno_fixed.cuh beside strong jumps, where it leaves
fields to FP64 (strong_fields, uneven_fields; uneven for a scalar).

Euler: over a whole right-hand side (tests/line_harness.hpp), against the same
formulas in FP64, both measured in 128-bit floating point.  Tolerance per
component as in test_kernel_scales.py: 16 times the error of the FP64 formulas
on the same data, or 2^-47 of the component's largest value.

Scalars: single faces with a jump beside values far smaller.  Tolerance: eight
units of 2^-57 of a largest difference that is less than 2^5 times the centre
values or the larger of the smallest two adjacent differences, and as much
again for FP64's own roundings: 2^-48 of the larger of those, or 16 times the
error of the FP64 formulas on the same face.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include "line_harness.hpp"
template <int NC>
void run(const std::string &kind, double k) {
  std::mt19937_64 g(5);
  std::uniform_real_distribution<double> U(-1, 1);
  auto sn = [](double x) { return std::sin(6.283185307179586 * x); };
  const int n = 200;
  const double R = std::pow(10.0, k);
  const Line<NC> s = line<NC>(n, 0.4, [&](int i, double *w) {
    const double x = (i + 0.5) / n, at = x < 0.5 ? R : 1;
    w[0] = 1 + 0.2 * sn(3 * x);
    w[3] = 1;
    if (kind == "pressure") w[3] = at;
    if (kind == "pressure_right") w[3] = x < 0.5 ? 1 : R;
    if (kind == "pressure_waves")
      w[1] = 0.3 * sn(x + 0.2), w[2] = 0.4 * sn(2 * x), w[3] = at * (1 + 0.1 * sn(4 * x));
    if (kind == "contact") w[0] *= at, w[1] = 0.5 * (1 + 0.1 * sn(x)), w[2] = 0.1, w[3] = 1 + 0.1 * sn(2 * x);
    if (kind == "shear") w[1] = 0.1, w[2] = x < 0.5 ? R : 0;
    if (kind == "blast") w[3] = std::fabs(x - 0.5) < 0.01 ? R : 1;
    if (kind == "rough" || kind == "rough_dense") {
      w[0] = kind == "rough" ? 1 + 0.5 * U(g) : std::pow(10.0, k / 2 * U(g));
      w[1] = U(g), w[2] = U(g), w[3] = std::pow(10.0, k / 2 * U(g));
    }
  });
  const Errors<NC> e = errors<NC>(s);
  for (int q = 0; q < NC; ++q) printf("%.17g %.17g %.17g\n", e.top[q], e.fp64[q], e.fixed[q]);
}
// Faces of a scalar: f = u^2 / 2 (burgers) or u, states of size 1 on one side of
// a jump and down to 2^-k on the other; prints the largest error over its bound.
void scalar(bool burgers, double k) {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(-1, 1);
  double worst = 0;
  for (int it = 0; it < 100000; ++it) {
    const double small = std::pow(2.0, -k * std::fabs(U(g))), A = 1.5;
    double u[6], f[6], xw[5], dg[5], dw[5];
    const int at = it % 7;
    for (int j = 0; j < 6; ++j) {
      u[j] = (it % 2 ? j < at : j >= at) ? U(g) : small * U(g);
      if (it % 5 == 0 && std::fabs(u[j]) < small) u[j] = it % 10 ? 0 : small;
      f[j] = burgers ? 0.5 * (u[j] * u[j]) : u[j];
    }
    for (int j = 0; j < 5; ++j) {
      dw[j] = u[j + 1] - u[j];
      dg[j] = f[j + 1] - f[j];
      xw[j] = A * dw[j];
    }
    const double centre = f[2] + f[3];
    const int es = top_exponent(xw, dg);
    if (es < 64) continue;
    double d[2][5];
    i64 c[2][5];
    Q q[2][5];
    for (int j = 0; j < 5; ++j) {
      const Q X = (Q)A * ((Q)u[j + 1] - (Q)u[j]);
      const Q G = burgers ? ((Q)u[j + 1] * u[j + 1] - (Q)u[j] * u[j]) / 2 : (Q)u[j + 1] - (Q)u[j];
      q[0][j] = X + G, q[1][4 - j] = X - G;
      d[0][j] = std::fma(A, dw[j], dg[j]), d[1][4 - j] = std::fma(A, dw[j], -dg[j]);
      const i64 x = to_fixed(xw[j], es), y = to_fixed(dg[j], es);
      c[0][j] = x + y, c[1][4 - j] = x - y;
    }
    const double h64 = (centre - xw[2]) + (correction<double>(d[0]) + correction<double>(d[1]));
    double h = h64;
    if (!uneven(xw, dg, es, centre))
      h = std::fma((double)(recon6<false>(c[0][0], c[0][1], c[0][2], c[0][3], c[0][4], Flt()) +
                            recon6<false>(c[1][0], c[1][1], c[1][2], c[1][3], c[1][4], Flt())),
                   scale_back(es), centre - xw[2]);
    const Q fc = burgers ? ((Q)u[2] * u[2] + (Q)u[3] * u[3]) / 2 : (Q)u[2] + (Q)u[3];
    const Q ref = fc - (q[0][2] + q[1][2]) / 2 + correction<Q>(q[0]) + correction<Q>(q[1]);
    double pair = 1e300;
    for (int j = 0; j < 4; ++j) {
      double m = 0;
      for (int i = j; i < j + 2; ++i) m = std::max(m, std::max(std::fabs(xw[i]), std::fabs(dg[i])));
      pair = std::min(pair, m);
    }
    // (the dissipation of the centre pair, should that be the jump, is FP64's in both paths)
    const double at_face = std::max(std::fabs(f[2]) + std::fabs(f[3]), std::fabs(xw[2]));
    // (beside exact zeros only correction()'s stand-in for the sensitivity term is left, 2^-265 of the jump)
    const double tol = std::max(
        std::ldexp(std::max(std::max(at_face, pair), std::ldexp(1.0, es - 1023 - 200)), -48),
        16 * (double)mag(ref - (Q)h64));
    worst = std::max(worst, (double)mag(ref - (Q)h) / tol);
  }
  printf("%.17g\n", worst);
}
int main(int, char **argv) {
  const std::string kind = argv[2];
  if (kind == "burgers" || kind == "advection") scalar(kind == "burgers", atof(argv[3]));
  else if (atoi(argv[1]) == 3) run<3>(kind, atof(argv[3]));
  else run<4>(kind, atof(argv[3]));
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("jumps")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "tests"), "-I",
                    os.path.join(ROOT, "paper_2603_26272_gb300", "csrc"), str(d / "m.cpp"), "-o",
                    str(d / "m")], check=True)
    return str(d / "m")


@pytest.mark.parametrize("kind,k", [("pressure", k) for k in (1, 2, 3, 4, 5, 6, 7, 9, 12, 16, 18)] +
                         [("pressure_right", k) for k in (3, 6, 12)] +
                         [("pressure_waves", k) for k in (3, 6, 9, 18)] +
                         [("contact", k) for k in (1, 3, 6, 12)] + [("shear", k) for k in (1, 3, 6)] +
                         [("blast", k) for k in (3, 9, 15)] + [("rough", k) for k in (2, 4, 8, 12)] +
                         [("rough_dense", k) for k in (2, 4, 8, 12)])
@pytest.mark.parametrize("nc", [3, 4])
def test_small_differences_beside_a_jump_keep_their_precision(harness, nc, kind, k):
    out = subprocess.run([harness, str(nc), kind, str(k)], check=True, capture_output=True, text=True)
    for row in out.stdout.splitlines():
        top, fp64, fixed = map(float, row.split())
        assert fixed <= max(16 * fp64, 2.0 ** -47 * top), out.stdout


@pytest.mark.parametrize("k", [8, 30, 80])
@pytest.mark.parametrize("kind", ["advection", "burgers"])
def test_scalar_faces_beside_a_jump_keep_their_precision(harness, kind, k):
    out = subprocess.run([harness, "1", kind, str(k)], check=True, capture_output=True, text=True)
    assert float(out.stdout) <= 1.0
