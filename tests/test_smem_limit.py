"""The record of the kernels' shared-memory limits (csrc/smem_limit.h), with a fake of the CUDA call."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2205_06690_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <vector>
#include "smem_limit.h"
int main() {
  sbse::SmemLimits limits;
  static int kernel_a, kernel_b;
  struct Call { int device; const void *fn; size_t bytes; bool ok; };
  for (Call c : std::vector<Call>{{0, &kernel_a, 50000, true},
                                  {0, &kernel_a, 40000, true},    // lower: kept
                                  {1, &kernel_a, 40000, true},    // another device has its own
                                  {1, &kernel_a, 60000, false},   // refused: not recorded
                                  {1, &kernel_a, 55000, true},
                                  {0, &kernel_b, 50000, true},
                                  {0, &kernel_a, 70000, true},
                                  {1, &kernel_a, 55000, true}}) { // set already
    bool called = false;
    limits.raise(c.device, c.fn, c.bytes, [&](size_t) { return called = true, c.ok; });
    printf("%d", called);
  }
  return 0;
}
"""


def test_limits_are_raised_per_device_and_kernel(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t"), "-pthread"],
                   check=True)
    assert subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout == "10111110"
