"""The integer path of csrc/weno_fixed.cuh where a state's magnitudes lie far
apart, against the same formulas in FP64, both measured in 128-bit floating point
over a whole right-hand side (tests/line_harness.hpp): flows far slower than
sound, dense cells beside light ones, a tangential velocity of rounding size.

Tolerance per component: 16 times the error of the FP64 formulas on the same
data (both paths round some dozens of operations a face, in another order), or
2^-47 of the component's largest value (two faces of 32 roundings each),
whichever is larger.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include "line_harness.hpp"
template <int NC>
void run(const char *kind, double k) {
  std::mt19937_64 g(5);
  std::uniform_real_distribution<double> U(-1, 1);
  auto sn = [](double x) { return std::sin(6.283185307179586 * x); };
  const std::string name = kind;
  const int n = 200;
  const Line<NC> s = line<NC>(n, 0.4, [&](int i, double *w) {
    const double x = (i + 0.5) / n, slow = std::pow(10.0, -k);
    w[0] = 1 + 0.2 * sn(3 * x);
    w[3] = 1 / 1.4;
    if (name == "slow") w[1] = slow;
    if (name == "slow_contact") w[0] *= x < 0.5 ? 1 : 0.125, w[1] = slow;
    if (name == "slow_waves")
      w[1] = slow * (1 + 0.1 * sn(x)), w[2] = slow * sn(2 * x), w[3] += slow * slow * 0.1 * sn(x);
    if (name == "dense")
      for (int q = 0; q < 4; ++q) w[q] = q == 1 || q == 2 ? U(g) : std::pow(10.0, k / 2 * U(g));
    if (name == "shear_noise")
      w[0] = (x < 0.5 ? 1 : 0.125) * (1 + slow * U(g)), w[1] = slow * U(g), w[2] = slow * U(g),
      w[3] = (x < 0.5 ? 1 : 0.1) * (1 + slow * U(g));
  });
  const Errors<NC> e = errors<NC>(s);
  for (int q = 0; q < NC; ++q) printf("%.17g %.17g %.17g\n", e.top[q], e.fp64[q], e.fixed[q]);
}
int main(int, char **argv) {
  if (atoi(argv[1]) == 3) run<3>(argv[2], atof(argv[3]));
  else run<4>(argv[2], atof(argv[3]));
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("scales")
    (d / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "tests"), "-I",
                    os.path.join(ROOT, "paper_2603_26272_gb300", "csrc"), str(d / "m.cpp"), "-o",
                    str(d / "m")], check=True)
    return str(d / "m")


@pytest.mark.parametrize("kind,k", [("slow", 0), ("slow", 4), ("slow", 8), ("slow_contact", 2),
                                    ("slow_contact", 8), ("slow_waves", 1), ("slow_waves", 8),
                                    ("dense", 2), ("dense", 4), ("dense", 8),
                                    ("shear_noise", 8), ("shear_noise", 13)])
@pytest.mark.parametrize("nc", [3, 4])
def test_no_field_is_cut_by_anothers_scale(harness, nc, kind, k):
    out = subprocess.run([harness, str(nc), kind, str(k)], check=True, capture_output=True, text=True)
    for row in out.stdout.splitlines():
        top, fp64, fixed = map(float, row.split())
        assert fixed <= max(16 * fp64, 2.0 ** -47 * top), out.stdout
