"""The integer path of csrc/weno_fixed.cuh on coarse polynomial data, where the
fifth difference of a field cancels to far below the third: whole right-hand sides
of the Euler equations with a linear to quartic density at constant velocity and
pressure, against the same formulas in FP64, both measured in 128-bit floating point
(tests/line_harness.hpp).  Tolerance per component as in test_kernel_scales.py: 16
times the error of the FP64 formulas on the same data, or 2^-47 of the component's
largest value.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include "line_harness.hpp"
template <int NC>
void run(int degree, int n, double at) {
  const Line<NC> s = line<NC>(n, 0.4, [&](int i, double *w) {
    const double x = (i + 0.5) / n - at;  // critical points about x = at
    const double h = 1.0 / n;  // degree 3: three cells about x = at all but equal
    w[0] = degree == 1 ? 2 + x : degree == 2 ? 1 + x * x : degree == 3 ? 1.1 + 8 * x * (x * x - h * h)
                                                        : 1 + x * x * (0.3 - x + x * x);
    w[1] = 0.7;
    w[2] = 0.4;
    w[3] = 1;
  });
  const Errors<NC> e = errors<NC>(s);
  for (int q = 0; q < NC; ++q) printf("%.17g %.17g %.17g\n", e.top[q], e.fp64[q], e.fixed[q]);
}
int main(int, char **argv) {
  (atoi(argv[1]) == 3 ? run<3> : run<4>)(atoi(argv[2]), atoi(argv[3]), atof(argv[4]));
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("polynomials")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "tests"), "-I",
                    os.path.join(ROOT, "paper_2603_26272_gb300", "csrc"), str(d / "m.cpp"), "-o",
                    str(d / "m")], check=True)
    return str(d / "m")


@pytest.mark.parametrize("at", [0.0, 0.5, 0.5001, 0.503, 0.53])
@pytest.mark.parametrize("n", [7, 9, 12, 13, 17, 24, 33])
@pytest.mark.parametrize("degree", [1, 2, 3, 4])
@pytest.mark.parametrize("nc", [3, 4])
def test_polynomial_density(harness, nc, degree, n, at):
    out = subprocess.run([harness, str(nc), str(degree), str(n), str(at)], check=True,
                         capture_output=True, text=True)
    for row in out.stdout.splitlines():
        top, fp64, fixed = map(float, row.split())
        assert fixed <= max(16 * fp64, 2.0 ** -47 * top), out.stdout
