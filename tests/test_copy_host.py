"""The serving loop's copy threads (compiled for the host): every byte copied,
from several threads at once, and no exception, nothing left queued when there
is no memory for the queue."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "kf_copy.h"
static thread_local int fail_at = -1;  // the allocation of this thread that fails, counted down
void* operator new(std::size_t n) {
  if (fail_at >= 0 && fail_at-- == 0) throw std::bad_alloc();
  if (void* p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

static bool round(kfi::CopyPool& pool, std::size_t bytes, int seed, int fail) {
  std::vector<char> a(bytes), b(bytes / 3), da(bytes), db(bytes / 3);
  for (std::size_t i = 0; i < a.size(); ++i) a[i] = char(i * 31 + seed);
  for (std::size_t i = 0; i < b.size(); ++i) b[i] = char(i * 17 - seed);
  const kfi::CopyPool::Piece pieces[] = {{da.data(), a.data(), a.size()}, {db.data(), b.data(), b.size()}};
  fail_at = fail;
  pool.copy(pieces, 2);
  fail_at = -1;
  return a == da && b == db;
}
int main() {
  kfi::CopyPool pool;
  pool.start(3);
  int bad = 0;
  for (int fail = -1; fail < 12; ++fail)  // no failure, then each allocation in turn
    for (std::size_t bytes : {std::size_t(0), std::size_t(1000), std::size_t(300000), std::size_t(40000001)})
      bad += !round(pool, bytes, fail, fail);
  std::vector<std::thread> ts;
  std::atomic<int> bad_t{0};
  for (int t = 0; t < 4; ++t)
    ts.emplace_back([&, t] {
      for (int k = 0; k < 10; ++k) bad_t += !round(pool, 3000000 + 1000 * t, k, k % 4 - 1);
    });
  for (auto& t : ts) t.join();
  pool.stop();
  std::printf("%d %d\n", bad, int(bad_t));
  return 0;
}
"""


def test_copies_are_whole_and_never_throw(tmp_path):
    src, exe = tmp_path / "copy.cpp", tmp_path / "copy"
    src.write_text("#include <atomic>\n" + SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_1605_05508_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "0 0", out
