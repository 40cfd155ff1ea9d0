"""Which FP32 2D grids the row-marching kernel takes: the host rule against measured
times of both kernels, and the grids it takes against the FP64 oracle."""
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2303_09671_gb300 import build as pfbuild
from paper_2303_09671_gb300 import pf

from conftest import rel_err
from test_gpu_march2d import KINDS, state

# us per step on 152 SMs: nx, ny, tiles, marching
MEASURED = [(8, 60000, 43.2, 49.4), (32, 20000, 16.4, 21.2), (60, 8000, 14.3, 13.2), (61, 8000, 14.3, 18.8),
            (64, 8192, 14.1, 18.2), (64, 32768, 46.5, 54.0), (100, 4000, 14.0, 13.1), (122, 6000, 19.1, 19.8),
            (128, 4096, 14.0, 15.7), (182, 4000, 19.0, 18.4), (200, 2000, 11.3, 13.0), (256, 2048, 13.9, 14.4),
            (330, 1000, 10.0, 11.8), (512, 1024, 13.9, 14.2), (600, 600, 10.0, 11.6), (960, 350, 9.9, 11.5),
            (1024, 400, 11.1, 11.5), (1024, 700, 18.1, 15.3), (1024, 1024, 23.8, 20.6), (2000, 200, 11.2, 11.5),
            (8192, 64, 14.0, 12.8), (20000, 24, 15.6, 12.8), (50000, 8, 19.1, 11.5), (1500, 1500, 49.5, 34.1),
            (2048, 2048, 92.9, 65.9)]
TAKEN = [(59, 8000), (120, 4000), (1201, 700), (1024, 700), (50001, 7), (5601, 131)]


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "rule.cu", d / "rule"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "pf_internal.cuh"\n#include "pf_kernels.h"\n'
                   "int main(int n, char** v) { for (int i = 1; i + 1 < n; i += 2)\n"
                   '    std::printf("%lld ", pf::march2d_rows(std::atoll(v[i]), std::atoll(v[i + 1]), 152)); }\n')
    subprocess.run([pfbuild.nvcc(), *pfbuild.ARCH, "-std=c++17", "-I", pfbuild.CSRC, "-I", pfbuild.INCLUDE, str(src), "-o",
                    str(exe)], check=True, capture_output=True)

    def call(sizes):
        args = [str(v) for n in sizes for v in n]
        return [int(v) for v in subprocess.run([os.fspath(exe), *args], check=True, capture_output=True).stdout.split()]

    return call


def test_rule_takes_the_faster_kernel(rows):
    for (nx, ny, tiles, march), r in zip(MEASURED, rows([m[:2] for m in MEASURED])):
        assert (r > 0) == (march < tiles), (nx, ny, r)
    assert all(r >= 4 for r in rows(TAKEN))
    assert rows([(512, 512), (8, 8), (1 << 20, 3)])[:2] == [0, 0]


@pytest.mark.gpu
@pytest.mark.parametrize("n", TAKEN)
@pytest.mark.parametrize("kw", KINDS)
def test_marching_grids(n, kw):
    """Strips that end within and at a warp's columns, one strip and many, fewer rows
    than the halo reaches; 1e-5 as in test_gpu_march2d.py, for the same reason."""
    pr, *f = state(n, kw)
    st = oracle.State(pr, *(a.astype(np.float64) for a in f))
    st.step(4)
    with pf.Sim(pr, "fp32") as s:
        s.set_fields(*f)
        s.step(4)
        for a, b in zip(s.get_fields(), (st.phi, st.cs, st.cl)):
            assert rel_err(a, b) <= 1e-5
