"""Host-side record of raised shared-memory limits: every device gets the call
for itself, a larger size asks again, a smaller one does not, and a failed call
is not recorded."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_13055_gb300", "csrc")
PROGRAM = r"""
#include "smem_limits.h"
#include <cstdio>
int main() {
  ckks::SmemLimits l;
  int f = 0, g = 0;
  struct { int device; const void* fn; size_t bytes; bool ok; } calls[] = {
      {0, &f, 100, true}, {0, &f, 100, true}, {0, &f, 60, true},      // once
      {1, &f, 100, true}, {1, &f, 100, true},                          // the second device too
      {0, &g, 100, true}, {0, &f, 101, true},                          // another kernel, a larger size
      {2, &f, 100, false}, {2, &f, 100, true}, {2, &f, 100, true}};    // failed, again, recorded
  for (auto& c : calls) {
    int n = 0;
    l.at_least(c.device, c.fn, c.bytes, [&] { ++n; return c.ok; });
    std::printf("%d", n);
  }
  return 0;
}
"""


def test_limits_are_kept_per_device_and_only_on_success(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe), "-pthread"], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "1001011110"
    # and the column launchers go through it
    text = open(os.path.join(CSRC, "cols.cuh")).read()
    assert "cudaGetDevice" in text and text.count("cudaFuncSetAttribute") == 1
