"""The window bounds' atan2 on the host: within the 3e-6 rad that the windows'
widening of 1.1e-5 rad allows for, in every octant and at the axes."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cmath>
#include <cstdio>
#include <initializer_list>
#include "kf_math.cuh"
int main() {
  double worst = 0;
  for (int i = 0; i <= 4000000; ++i) {
    const double phi = (i / 4000000.0 - 0.5) * 2 * M_PI;
    for (double r : {1e-3, 4.0, 1e3}) {
      const float x = float(r * std::cos(phi)), y = float(r * std::sin(phi));
      worst = std::fmax(worst, std::fabs(double(kf::atan2_approx(y, x)) - std::atan2(double(y), double(x))));
    }
  }
  for (float y : {0.f, -0.f, 1.f, -1.f})
    for (float x : {0.f, -0.f, 1.f, -1.f})
      if (x != 0.f || y != 0.f)
        worst = std::fmax(worst, std::fabs(double(kf::atan2_approx(y, x)) - std::atan2(double(y), double(x))));
  std::printf("%.3e\n", worst);
  return 0;
}
"""


def test_atan2_within_its_bound(tmp_path):
    src, exe = tmp_path / "atan2.cpp", tmp_path / "atan2"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1605_05508_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    worst = float(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout)
    assert worst < 3e-6, worst
