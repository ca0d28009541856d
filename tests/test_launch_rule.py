"""The row kernels' block size rule depends on the GPU's own SM count (csrc/row_common.cuh, a host function)."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_06640_gb300", "csrc")

PROGRAM = r"""
#include "row_common.cuh"
#include <cstdio>
using adg::row::block_threads;
int main() {
  for (int sms : {20, 152, 400}) {
    const long small = 8L * sms;
    // small launches: single warps, whatever the tuner chose; above: the choice, else the rule of the type and degree
    for (int choice : {0, 64, 128, 256})
      if (block_threads<double, 3>(choice, small, sms) != 32 || block_threads<float, 5>(choice, 1, sms) != 32) return 1;
    for (int choice : {64, 128, 256})
      if (block_threads<double, 3>(choice, small + 1, sms) != choice) return 2;
    if (block_threads<double, 5>(0, small + 1, sms) != 128 || block_threads<float, 3>(0, small + 1, sms) != 128) return 3;
    if (block_threads<float, 5>(0, small + 1, sms) != 256) return 4;
  }
  std::puts("ok");
}
"""


def test_block_size_follows_the_sm_count(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = str(tmp_path / "rule.cu"), str(tmp_path / "rule")
    open(src, "w").write(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + CSRC, src, "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n"
