"""The loop over the host threads, compiled with an allocator that fails at every point in turn: each
index is done once, or the failure comes out as an exception, and nothing ends the process."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_02611_gb300", "csrc")

PROGRAM = r"""
#include "host_parallel.hpp"
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <stdexcept>
#include <vector>
static thread_local long fail_at = -1;  // allocations of this thread until one fails
void* operator new(size_t n) {
  if (fail_at >= 0 && fail_at-- == 0) throw std::bad_alloc();
  if (void* p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
int main() {
  for (long k = 0; k < 60; ++k) {
    std::vector<std::atomic<int>> a(1000);
    bool all = true;
    try {
      fail_at = k;
      gbdmrg::host_parallel(1000, 1L << 30, [&](long i) { ++a[i]; });
    } catch (const std::bad_alloc&) {
      all = false;
    }
    fail_at = -1;
    for (auto& x : a)
      if (x > 1 || (all && x != 1)) return 1;
  }
  int seen = 0;
  try {
    gbdmrg::host_parallel(1000, 1L << 30, [&](long i) { if (i == 500) throw std::runtime_error("x"); });
  } catch (const std::runtime_error&) {
    seen = 1;
  }
  return seen ? 0 : 2;
}
"""


def test_failing_allocations(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src),
                    os.path.join(CSRC, "host_parallel.cpp"), "-o", str(tmp_path / "t")], check=True)
    p = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert p.returncode == 0, (p.returncode, p.stderr)
