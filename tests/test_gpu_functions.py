"""The kernels' own logarithms and reciprocals against extended precision: each
within the bound stated beside it, and CUDA's values outside its range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_09671_gb300 import build as pfbuild
from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pf_line.cuh"
#include "pf_words.cuh"
using namespace pf;
__global__ void run(int op, const double* x, double* y, int n, const __grid_constant__ LogTable T) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (op == 0) y[i] = log64(x[i]);
    if (op == 1) y[i] = rcp64(x[i]);
    if (op == 2 || op == 3) {
        const float2 v = make_float2((float)x[i], 1.5f);
        float2 r = op == 2 ? ln_normal(v) : vrcp_n(v);
        if (op == 2 && !is_positive(v)) r = ln_fix(v, r);
        y[i] = (double)r.x;
    }
    if (op == 4) {
        const float h = (float)x[i], l = (float)(x[i] - (double)h);
        const Triple r = ln_triple(T, Triple{h, l, (float)(x[i] - (double)h - (double)l)});
        y[3 * i] = r.h;
        y[3 * i + 1] = r.l;
        y[3 * i + 2] = r.t;
    }
}
extern "C" int evaluate(int op, const double* x, double* y, int n, int width) {
    static const LogTable T(0);
    double *dx = nullptr, *dy = nullptr;
    if (cudaMalloc(&dx, n * sizeof(double)) != cudaSuccess) return 1;
    if (cudaMalloc(&dy, (size_t)n * width * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(dx, x, n * sizeof(double), cudaMemcpyHostToDevice);
    run<<<(n + 255) / 256, 256>>>(op, dx, dy, n, T);
    const cudaError_t e = cudaMemcpy(y, dy, (size_t)n * width * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dy);
    return e == cudaSuccess ? 0 : 2;
}
"""
OPS = {"log64": 0, "rcp64": 1, "ln_normal": 2, "vrcp_n": 3, "ln_triple": 4}


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    d = tmp_path_factory.mktemp("functions")
    src, so = d / "functions.cu", d / "libfunctions.so"
    src.write_text(SOURCE)
    subprocess.run([pfbuild.nvcc(), *pfbuild.ARCH, *pfbuild.NVFLAGS, "-shared", "-I", pfbuild.CSRC, "-I", pfbuild.INCLUDE,
                    str(src), "-o", str(so), "-lcudart"], check=True, capture_output=True)
    lib = ctypes.CDLL(os.fspath(so))

    def call(name, x):
        x = np.ascontiguousarray(x, np.float64)
        width = 3 if name == "ln_triple" else 1
        y = np.empty(x.size * width)
        assert lib.evaluate(OPS[name], x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p), x.size,
                            width) == 0
        return y.reshape(x.size, width).astype(np.longdouble).sum(1)

    return call


def arguments(lo, hi, dtype):
    """Spread over the range's logarithm, dense around 1, and the neighbours of the
    reduction's and the tables' interval ends."""
    g = np.random.default_rng(7)
    ends = np.concatenate([np.sqrt(0.5) * 2 ** (np.arange(257) / 256), 1 + np.arange(129) / 128, [1.0, 2.0, lo, hi]])
    x = np.concatenate([np.exp(g.uniform(np.log(lo), np.log(hi), 400000)), g.uniform(0.68, 1.45, 400000),
                        1 + g.uniform(-0.02, 0.02, 200000)] +
                       [np.nextafter(ends.astype(dtype), dtype(s)).astype(np.float64) for s in (0, 100)])
    x = x.astype(dtype).astype(np.float64)
    return x[(x >= lo) & (x <= hi)]


def ulps(y, ref, bits):
    """|y - ref| in units in the last place of a result of `bits` bits."""
    return np.abs(y - ref) / np.ldexp(np.longdouble(1), np.frexp(ref)[1] - bits)


# the functions' own bounds: log64 rounds once apart from terms below a quarter of
# an ulp; rcp64 once apart from 2^-16; CUDA's logf and rcp.approx.f32 have 1 ulp
@pytest.mark.parametrize("name,lo,hi,dtype,bits,bound", [
    ("log64", 1e-307, 1e307, np.float64, 53, 0.77), ("rcp64", 1e-300, 1e300, np.float64, 53, 0.501),
    ("ln_normal", 1.2e-38, 3.4e38, np.float32, 24, 1.0), ("vrcp_n", 1e-37, 1e37, np.float32, 24, 1.0)])
def test_function_within_its_bound(evaluate, name, lo, hi, dtype, bits, bound):
    x = arguments(lo, hi, dtype)
    y = evaluate(name, x)
    ref = 1 / x.astype(np.longdouble) if name in ("rcp64", "vrcp_n") else np.log(x.astype(np.longdouble))
    zero = ref == 0
    assert np.all(y[zero] == 0)
    assert ulps(y[~zero], ref[~zero], bits).max() <= bound


@pytest.mark.parametrize("name", ["log64", "ln_normal"])
def test_logarithm_of_special_values(evaluate, name):
    """Outside the positive normal numbers: what CUDA's function gives (the FP32 one is
    not made for +inf, see below)."""
    tiny = 1e-310 if name == "log64" else 1e-40
    y = evaluate(name, [0.0, -0.0, -1.0, np.inf, -np.inf, np.nan, tiny]).astype(np.float64)
    assert y[0] == y[1] == -np.inf and (name == "ln_normal" or y[3] == np.inf)
    assert np.isnan(y[[2, 4, 5]]).all()
    assert abs(y[6] - np.log(tiny if name == "log64" else float(np.float32(tiny)))) <= 1e-6 * abs(y[6])


def test_logarithm_in_three_words(evaluate):
    """Within 2^-53 of the larger of 1 and the logarithm, and NaN below 2^-70 and
    above FP32's range."""
    x = arguments(2.0 ** -69, 3e38, np.float64)
    ref = np.log(x.astype(np.longdouble))
    err = np.abs(evaluate("ln_triple", x) - ref) / np.maximum(1, np.abs(ref))
    assert err.max() <= 2.0 ** -53
    assert np.isnan(evaluate("ln_triple", [0.0, -1.0, 1e-30, np.inf, np.nan]).astype(np.float64)).all()


def test_infinite_concentration_ends_in_nan():
    """A line's cell of infinite c_s and c_l: phi is NaN after a step in both
    precisions, and a batched instance stops without converging."""
    pr, phi, cs, cl = wl.pulled_front_1d(N=100, V=1.0, front_cell=30, A=1.0, b=1.0)
    cs[30] = cl[30] = np.inf
    for precision, dtype in (("fp32", np.float32), ("fp64", np.float64)):
        f = [a.astype(dtype) for a in (phi, cs, cl)]
        with pf.Sim(pr, precision) as s:
            s.set_fields(*f)
            s.step(2)
            assert np.isnan(s.get_fields()[0][28:33]).all()
        r = pf.run_batch(pr, [100], [1.0], *f, precision=precision, max_steps=4, steps_per_launch=4,
                         launches_per_graph=1, check_every=2, tol=-1.0, want_fields=True)
        assert np.isnan(r["phi"][30]) and not r["converged"][0] and np.isnan(r["k_v"][0])
