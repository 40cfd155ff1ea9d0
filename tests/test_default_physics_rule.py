"""Which parameter sets take the kernels' default-physics instances: a host rule,
compiled and evaluated without a GPU."""
import os
import subprocess

import pytest

from paper_2303_09671_gb300 import build as pfbuild

SOURCE = r"""
#include <cstdio>
#include "pf_line.cuh"
using namespace pf;
int main() {
    HostProblem P = {};
    P.dx = 0.5; P.k_e = 0.1; P.D_s = 1e-4; P.D_l = 1.0; P.c_inf = 1.0; P.b = 1.0; P.delta = 1e-3;
    auto say = [&]() { std::printf("%d%d%d ", std_physics(P, false), std_physics(P, true), line_std(P)); };
    say();
    HostProblem Q = P;
    P.delta = 0.0; say(); P = Q;
    P.b = 1e-12; say(); P = Q;
    P.c_inf = 1e-12; say(); P = Q;
    P.D_s = 1e12; say(); P = Q;
    P.interp = 1; say(); P = Q;
    P.mobility = 1; say(); P = Q;
    P.a = 0.3; say();
}
"""


def test_range_is_asked_of_kernels_with_the_product_only(tmp_path):
    """FP32 2D and 3D steps take two reciprocals side by side and need no range; FP64
    steps and the line kernels form 1/(Mbar G)."""
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(SOURCE)
    subprocess.run([pfbuild.nvcc(), *pfbuild.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", pfbuild.CSRC, "-I",
                    pfbuild.INCLUDE, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([os.fspath(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["111", "100", "100", "100", "100", "000", "000", "110"]
