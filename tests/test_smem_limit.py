"""Shared-memory limits of kernels (csrc/smem_limit.h): an attribute of the
function in each device's context. A solver on a second GPU raises its own
limit, however large the first GPU's already is; on one GPU a limit is only
ever raised; a call that failed is made again."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2403_17018_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "smem_limit.h"
int main() {
  henry::SmemLimits limits;
  int f = 0, g = 0, error = 0;
  auto call = [&](int device, const void* fn, std::size_t bytes) {
    int made = 0;
    const int rc = limits.raise(device, fn, bytes, [&](const void* h, std::size_t n) {
      made = h == fn && n == bytes ? 1 : -1;
      return error;
    });
    std::printf("%d%d ", made, rc);
  };
  call(0, &f, 40000);    // within what every launch may use
  call(0, &f, 96256);
  call(0, &f, 60000);    // lower: kept
  call(1, &f, 60000);    // the other device's own
  call(1, &f, 96256);
  call(0, &g, 96256);    // another kernel
  error = 1;
  call(1, &g, 60000);    // refused
  error = 0;
  call(1, &g, 60000);    // and made again
  call(1, &g, 60000);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_limits_are_kept_per_device_and_only_raised(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out.split() == ["00", "10", "00", "10", "10", "10", "11", "10", "00"]
