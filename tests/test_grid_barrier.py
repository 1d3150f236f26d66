"""The barrier of the re-discretisation launch, compiled for the host: threads in the place of blocks, across both sides
of its word (the top bit) and the wrap at 2^32."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1102_2193_gb300", "csrc")
SRC = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "lclb_barrier.h"
struct Words {
  std::atomic<unsigned> bar{0};
  std::atomic<int> err{0};
  unsigned word() { return bar.load(std::memory_order_acquire); }
  unsigned arrive(unsigned add) { return bar.fetch_add(add, std::memory_order_acq_rel); }
  bool failed() { return err.load() != 0; }
  void fail() { err.fetch_or(1); }
  void pause() { std::this_thread::yield(); }
};
int main() {
  // n threads, 13 barriers: between two of them every thread must have passed the first
  for (unsigned n : {1u, 3u, 5u}) {
    Words w;
    std::vector<std::atomic<int>> at(n);
    for (auto& a : at) a = 0;
    std::atomic<int> bad{0};
    std::vector<std::thread> th;
    for (unsigned t = 0; t < n; ++t)
      th.emplace_back([&, t] {
        for (int r = 1; r <= 13; ++r) {
          at[t] = r;
          if (!lclb::barrier_wait(w, n, t == n - 1, 1 << 30)) bad = 1;
          for (unsigned k = 0; k < n; ++k)
            if (at[k] < r || at[k] > r + 1) bad = 1;
        }
      });
    for (auto& t : th) t.join();
    if (bad || w.bar != 0x80000000u || w.err) { std::printf("n = %u: broken\n", n); return 1; }
  }
  // a missing arrival ends the wait with the error set; a set error ends other waits early
  Words w;
  if (lclb::barrier_wait(w, 2, true, 1000) || !w.err) { std::printf("no error\n"); return 1; }
  Words v;
  v.err = 1;
  if (lclb::barrier_wait(v, 2, false, 2000000000)) { std::printf("waited\n"); return 1; }
  return 0;
}
"""


def test_barrier_across_the_wrap(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(tmp_path / "t.cpp"), "-o",
                           str(tmp_path / "t")])
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
