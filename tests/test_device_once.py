"""Set-up that the CUDA runtime keeps per device is done on each device that a kernel runs on, and
again where it failed (host code, compiled with a stand-in for the set-up)."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1605_02611_gb300", "csrc")

PROGRAM = r"""
#include "device_once.hpp"
#include <cstdio>
int main() {
  gbdmrg::DeviceOnce once;
  int calls[100] = {};
  bool work = false;
  auto on = [&](int dev) { return once(dev, [&] { ++calls[dev]; return work; }); };
  if (on(0) || calls[0] != 1) return 1;       // failed: not remembered
  work = true;
  if (!on(0) || !on(0) || calls[0] != 2) return 2;
  if (!on(1) || !on(1) || calls[1] != 1) return 3;  // the second device has its own
  if (!on(63) || !on(63) || calls[63] != 1 || !on(0) || calls[0] != 2) return 4;
  if (!on(70) || !on(70) || calls[70] != 2) return 5;  // beyond what is remembered: every time
  return 0;
}
"""


def test_rule(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(tmp_path / "t")], check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0


def test_no_limit_is_raised_once_per_process():
    for f in sorted(os.listdir(CSRC)):
        if f != "device_once.hpp":
            with open(os.path.join(CSRC, f)) as s:
                assert not re.search(r"cudaFuncSetAttribute\s*\(", s.read()), f
