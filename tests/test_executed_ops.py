"""Host check of the operation counts that roofline fractions are formed with
(csrc/ax_costs.cpp, executed_ops_per_node): the double-word kernel at order 7
against ncu's per-opcode counts of the kernel as it is (per node FADD 390.9, FFMA
145.5, FMUL 53.8, and FFMA2 63.0, FADD2 36.0, FMUL2 6.0 doing two operations
each), and its place below the design count, which only double-word arithmetic
differs from."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2504_07042_gb300", "csrc")
F64DW, TRILINEAR = 5, 1

DRIVER = r"""
#include <cstdio>
namespace ax { double pipe_ops_per_node(int, int, int); double executed_ops_per_node(int, int, int); }
int main() {
  for (int prec = 0; prec <= 5; ++prec)
    for (int kind = 0; kind <= 3; ++kind)
      for (int N1 = 2; N1 <= 16; ++N1)
        std::printf("%d %d %d %.6f %.6f\n", prec, kind, N1, ax::pipe_ops_per_node(N1, kind, prec),
                    ax::executed_ops_per_node(N1, kind, prec));
}
"""


def test_executed_operations(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no host C++ compiler or CUDA headers")
    drv, exe = tmp_path / "drv.cpp", str(tmp_path / "drv")
    drv.write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", inc, "-o", exe, str(drv), os.path.join(CSRC, "ax_costs.cpp")],
                   check=True, capture_output=True)
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.strip().splitlines():
        prec, kind, N1, design, executed = (float(v) for v in line.split())
        if prec != F64DW:
            assert executed == design
        elif N1 > 2:
            assert 0.8 * design < executed < design
        if (prec, kind, N1) == (F64DW, TRILINEAR, 8):
            measured = 390.9 + 145.5 + 53.8 + 2 * (63.0 + 36.0 + 6.0)
            assert abs(measured / executed - 1) < 0.02
