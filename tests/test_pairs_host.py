"""The Kalman update on pairs of rows gives the bits of the scalar one (the
track arithmetic's header compiled for the host, random covariances, gains
and residuals)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstring>
#include <random>
#include "kf_math.cuh"
int main() {
  std::mt19937 g(7);
  std::normal_distribution<float> N;
  int bad = 0;
  for (int t = 0; t < 20000; ++t) {
    float p[6], lo[3], C[21], A[6][6], Si[6], r[3];
    for (float& v : p) v = N(g);
    for (float& v : lo) v = 1e-8f * N(g);
    for (auto& row : A) for (float& v : row) v = 0.05f * N(g);
    for (int i = 0; i < 6; ++i)
      for (int j = 0; j <= i; ++j) {
        float s = 0;
        for (int k = 0; k < 6; ++k) s += A[i][k] * A[j][k];
        C[kf::sym(i, j)] = s;
      }
    kf::inverse_S(C, 1e-4f, 1e-4f, 1e-2f, Si);
    for (float& v : r) v = 0.02f * N(g);
    float q[6], ql[3], D[21];
    memcpy(q, p, sizeof p);
    memcpy(ql, lo, sizeof lo);
    memcpy(D, C, sizeof C);
    kf::kalman_update_pairs<true>(p, lo, C, Si, r[0], r[1], r[2], 1e-4f, 1e-4f, 1e-2f);
    kf::kalman_update_lanes<float, true>(q, ql, D, Si, r[0], r[1], r[2], 1e-4f, 1e-4f, 1e-2f, true);
    if (memcmp(p, q, sizeof p) || memcmp(lo, ql, sizeof lo) || memcmp(C, D, sizeof C)) ++bad;
  }
  printf("%d\n", bad);
  return bad != 0;
}
"""


def test_update_on_pairs_equals_the_scalar_update(tmp_path):
    src, exe = tmp_path / "pairs.cpp", tmp_path / "pairs"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1605_05508_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"
