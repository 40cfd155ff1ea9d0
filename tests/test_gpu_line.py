"""The strip kernels of 1D lines: batches whose lengths sit at the strips' edges,
on one CTA per instance and spread over clusters, against the FP64 oracle and
against each other."""
import numpy as np
import pytest

import oracle
from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

from conftest import rel_err

pytestmark = pytest.mark.gpu

# around multiples of 60 and 120 cells (a strip of two or four cells per lane)
LENGTHS = [8, 57, 60, 61, 118, 120, 121, 479, 960, 1021]


def fronts(lengths, v=1.5, **kw):
    prs, fields = [], []
    for n in lengths:
        pr, *f = wl.pulled_front_1d(N=n, dx=0.5, V=v, front_cell=max(2, min(24, n // 3)), **kw)
        prs.append(pr)
        fields.append(f)
    dt = min(0.9 * wl.stable_dt(prs[0]), 0.4 * prs[0]["dx"] / v)
    pr0 = dict(prs[0], x0=12.0)
    return pr0, [np.concatenate(f) for f in zip(*fields)], dt


@pytest.mark.parametrize("kw", [dict(A=1.0, b=1.0), dict(A=1.0, b=1.0, a=-0.3, interp="cubic", mobility="const", D_s=0.1)])
def test_strip_edges_fp64(kw):
    """A few instances (a cluster each) against the oracle with window shifts, and
    the same instances among many (one CTA each) bit for bit."""
    pr, f, dt = fronts(LENGTHS, **kw)
    steps = 77
    few = pf.run_batch(pr, LENGTHS, [1.5] * 10, *f, precision="fp64", dt=[dt] * 10, max_steps=steps, steps_per_launch=50,
                       launches_per_graph=1, check_every=steps, tol=-1.0, want_fields=True)
    many = pf.run_batch(pr, LENGTHS * 20, [1.5] * 200, *[np.tile(a, 20) for a in f], precision="fp64", dt=[dt] * 200,
                        max_steps=steps, steps_per_launch=steps, launches_per_graph=1, check_every=19, tol=-1.0,
                        want_fields=True)
    o = 0
    for n in LENGTHS:
        st = oracle.State(dict(pr, n=(n,), dt=dt), *[a[o:o + n] for a in f])
        st.step(steps)
        assert n == 8 or st.clock.shifts > 0
        for k, ref in (("phi", st.phi), ("cs", st.cs), ("cl", st.cl)):
            assert rel_err(few[k][o:o + n], ref) <= 1e-11, (n, k)
            assert np.array_equal(few[k][o:o + n], many[k][o:o + n]), (n, k)
        o += n


@pytest.mark.parametrize("cpt", [2, 4])
def test_strip_edges_fp32(cpt):
    """FP32, both numbers of cells per lane, on clusters and on single CTAs: the same
    bits, and within FP32 rounding of the FP64 run (77 steps of increments below
    1: 77 roundings of 6e-8 relative to each field's maximum)."""
    pr, f, dt = fronts(LENGTHS, A=1.0, b=1.0)
    f32 = [a.astype(np.float32) for a in f]
    kw = dict(max_steps=77, steps_per_launch=77, launches_per_graph=1, check_every=77, tol=-1.0, want_fields=True)
    ref = pf.run_batch(pr, LENGTHS, [1.5] * 10, *f32, precision="fp64", dt=[dt] * 10, **kw)
    few = pf.run_batch(pr, LENGTHS, [1.5] * 10, *f32, dt=[dt] * 10, cells_per_thread=cpt, **kw)
    many = pf.run_batch(pr, LENGTHS * 20, [1.5] * 200, *[np.tile(a, 20) for a in f32], dt=[dt] * 200,
                        cells_per_thread=cpt, **kw)
    for k in ("phi", "cs", "cl"):
        assert np.array_equal(few[k], many[k][:len(few[k])]), k
        assert np.abs(few[k] - ref[k]).max() <= 77 * 6e-8 * np.abs(ref[k]).max(), k


@pytest.mark.parametrize("kw", [dict(A=1.2, b=0.8), dict(A=1.0, b=1.0, a=-0.3, interp="cubic", mobility="const", D_s=0.1)])
def test_reverse_sweep_at_strip_edges(kw):
    """FP64 derivatives by the reverse sweep equal the tangent run's on lengths at
    the strips' edges, on clusters (10 instances) and on single CTAs (160): within
    1e-9 of the largest, the bound of the other reverse tests."""
    pr, f, dt = fronts(LENGTHS, v=0.8, **kw)
    for rep in (1, 16):
        args = (pr, LENGTHS * rep, [0.8] * (10 * rep), *[np.tile(a, rep) for a in f], 60)
        t = pf.adjoint(*args, precision="fp64", dt=[dt] * (10 * rep))
        r = pf.adjoint(*args, precision="fp64", dt=[dt] * (10 * rep), mode="reverse", checkpoint_every=13)
        assert np.abs(r["k"] - t["k"]).max() <= 1e-13 * np.abs(t["k"]).max()
        for j in range(3):
            assert np.abs(r["dk"][:, j] - t["dk"][:, j]).max() <= 1e-9 * np.abs(t["dk"][:, j]).max(), j
