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


LINES = [("pulled", dict(V=1.5)), ("closed", dict(bc_hi=("noflux",))),
         ("periodic", dict(bc_lo=("periodic",), bc_hi=("periodic",))),
         ("cold_dirichlet", dict(bc_lo=("dirichlet",), bc_hi=("noflux",)))]


def line_state(kind, kw, n):
    if kind == "pulled":
        pr, *f = wl.pulled_front_1d(N=n, front_cell=max(1, n // 3), A=1.0, b=1.0, **kw)
        return pr, f
    if kind == "closed":
        pr, *f = wl.random_state(1, (n,), A=1.2, b=0.7, a=0.2, seed=n, **kw)
        return pr, f
    pr, *f = wl.random_state(1, (n,), A=1.0, b=1.0, a=0.2, seed=n, amp=0.1, **kw)
    if kind == "periodic":   # a smooth profile that closes on itself
        f[0] = 0.5 + 0.1 * np.sin(2 * np.pi * (np.arange(n) + 0.3) / n)
    if kind == "cold_dirichlet":   # a solid cold end
        pr["dirichlet"] = (1.0, pr["k_e"], 1.0)
    return pr, f


@pytest.mark.parametrize("kind,kw", LINES)
@pytest.mark.parametrize("n", [3, 16, 17, 33, 113, 500, 2432, 2433])
def test_single_line_fp64(kind, kw, n):
    """A Sim's line over the sizes at which strips, their halos and the choice of
    kernel change: against the oracle, and the same bits however its steps are
    grouped into calls."""
    pr, f = line_state(kind, kw, n)
    steps = 21
    st = oracle.State(pr, *f)
    st.step(steps)
    out = []
    for groups in ([21], [1] * 21, [2, 9, 3, 7]):
        with pf.Sim(pr, "fp64") as s:
            s.set_fields(*f)
            for g in groups:
                s.step(g)
            out.append(s.get_fields())
            assert s.clock == (steps, st.clock.shifts)
    for got, ref in zip(out[0], (st.phi, st.cs, st.cl)):
        assert rel_err(got, ref) <= 1e-11
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))


@pytest.mark.parametrize("n", [3, 33, 500, 19456, 19457])
def test_single_line_fp32(n):
    """FP32 with a moving window, both kernels (19456 cells fill the SMs of the
    first): the same bits in one call and in single steps, and within 21 roundings
    of FP32 of the FP64 line."""
    pr, *f = wl.pulled_front_1d(N=n, front_cell=max(1, min(40, n // 3)), V=1.5, A=1.0, b=1.0)
    f = [a.astype(np.float32) for a in f]
    out = []
    for prec, groups in (("fp64", [21]), ("fp32", [21]), ("fp32", [1] * 21)):
        with pf.Sim(pr, prec) as s:
            s.set_fields(*f)
            for g in groups:
                s.step(g)
            out.append(s.get_fields())
    for ref, a, b in zip(*out):
        assert np.array_equal(a, b)
        assert np.abs(a - ref).max() <= 21 * 6e-8 * np.abs(ref).max()


def test_window_jumps_by_many_cells():
    """A clock set far ahead: the next step drops every cell it is behind by."""
    pr, *f = wl.pulled_front_1d(N=100, V=1.0, A=1.0, b=1.0)
    for prec in ("fp32", "fp64"):
        with pf.Sim(pr, prec) as s:
            s.set_fields(*f)
            s.set_clock(int(30 * pr["dx"] / pr["dt"]), 0)
            s.step(1)
            assert s.clock[1] in (30, 31)
            k = s.clock[1]
            g = s.get_fields()
        assert np.abs(g[0][:100 - k] - f[0][k:]).max() < 0.1 and np.all(np.abs(g[0][100 - k:]) < 1e-6)
