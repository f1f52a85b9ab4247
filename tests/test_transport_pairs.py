"""The transport and the update on pairs of rows give the bits of the scalar
forms, on the host and on the GPU (the track arithmetic's header compiled into a
small program: random states and covariances, curling and missing tracks among
them)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1605_05508_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "kf_math.cuh"
struct Case {
  float p[6], lo[3], C[21], a, R, r[3];
};
struct Result {
  int bad, crossed;
};
template <bool LEAN>
KF_HD void check(const Case& c, Result& out) {
  float p[6], lo[3], C[21], q[6], ql[3], D[21];
  for (int i = 0; i < 6; ++i) p[i] = q[i] = c.p[i];
  for (int i = 0; i < 3; ++i) lo[i] = ql[i] = c.lo[i];
  for (int i = 0; i < 21; ++i) C[i] = D[i] = c.C[i];
  const int st = kf::propagate_lanes<float, 12, true, LEAN, true>(p, lo, C, c.a, c.R, true);
  bool same = st == kf::propagate_lanes<float, 12, true, LEAN, false>(q, ql, D, c.a, c.R, true);
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = 0; i < 6; ++i) same &= p[i] == q[i];
    for (int i = 0; i < 3; ++i) same &= lo[i] == ql[i];
    for (int i = 0; i < 21; ++i) same &= C[i] == D[i];
    if (pass || st) break;
    float Si[6];
    kf::inverse_S(C, 1e-4f, 1e-4f, 1e-2f, Si);
    kf::kalman_update_pairs<true>(p, lo, C, Si, c.r[0], c.r[1], c.r[2], 1e-4f, 1e-4f, 1e-2f);
    kf::kalman_update_lanes<float, true>(q, ql, D, Si, c.r[0], c.r[1], c.r[2], 1e-4f, 1e-4f, 1e-2f, true);
  }
  out.bad = !same;
  out.crossed = st == 0;
}
#ifdef __CUDACC__
__global__ void kernel(const Case* c, Result* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  Result a, b;
  check<false>(c[i], a);
  check<true>(c[i], b);
  out[i].bad = a.bad + b.bad;
  out[i].crossed = a.crossed;
}
#endif
int main() {
  const int n = 50000;
  std::mt19937 g(7);
  std::normal_distribution<float> N;
  std::uniform_real_distribution<float> U(0, 1);
  std::vector<Case> cs(n);
  for (Case& c : cs) {
    const float r = 1 + 30 * U(g), phi = 6.2831853f * U(g), pt = 0.15f + 8 * U(g) * U(g), dphi = 0.3f * N(g);
    c.p[0] = r * cosf(phi), c.p[1] = r * sinf(phi), c.p[2] = 5 * N(g);
    c.p[3] = pt * cosf(phi + dphi), c.p[4] = pt * sinf(phi + dphi), c.p[5] = pt * N(g);
    for (float& v : c.lo) v = 1e-7f * N(g);
    float A[6][6];
    for (auto& row : A) for (float& v : row) v = 0.05f * N(g);
    for (int i = 0; i < 6; ++i)
      for (int j = 0; j <= i; ++j) {
        float s = 0;
        for (int k = 0; k < 6; ++k) s += A[i][k] * A[j][k];
        c.C[kf::sym(i, j)] = s;
      }
    c.a = (U(g) < 0.5f ? 1.f : -1.f) * 0.0114f;
    c.R = r + 6 * U(g);
    for (float& v : c.r) v = 0.02f * N(g);
  }
  std::vector<Result> res(n);
#ifdef __CUDACC__
  Case* dc;
  Result* dr;
  if (cudaMalloc(&dc, n * sizeof(Case)) || cudaMalloc(&dr, n * sizeof(Result))) return 2;
  if (cudaMemcpy(dc, cs.data(), n * sizeof(Case), cudaMemcpyHostToDevice)) return 2;
  kernel<<<(n + 127) / 128, 128>>>(dc, dr, n);
  if (cudaMemcpy(res.data(), dr, n * sizeof(Result), cudaMemcpyDeviceToHost)) return 2;
#else
  for (int i = 0; i < n; ++i) {
    Result a, b;
    check<false>(cs[i], a);
    check<true>(cs[i], b);
    res[i] = {a.bad + b.bad, a.crossed};
  }
#endif
  int bad = 0, crossed = 0;
  for (const Result& r : res) bad += r.bad, crossed += r.crossed;
  std::printf("%d %d\n", bad, crossed);
  return 0;
}
"""


def _run(exe):
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True, timeout=120).stdout.split()
    assert out[0] == "0" and int(out[1]) > 25000, out  # the same bits; most tracks cross


def test_pairs_equal_scalar_on_the_host(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    _run(tmp_path / "t")


@pytest.mark.gpu
def test_pairs_equal_scalar_on_the_gpu(tmp_path):
    from paper_1605_05508_gb300 import build as B
    (tmp_path / "t.cu").write_text(SRC)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-I", CSRC, str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")],
                   check=True)
    _run(tmp_path / "t")
