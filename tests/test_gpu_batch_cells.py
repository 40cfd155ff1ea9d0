"""The cells per lane of a batch: what a request is taken to, and that the choice
changes no bit (the autotuner picks by time)."""
import numpy as np
import pytest

from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def run(precision, cells, lengths=(61, 240, 500)):
    prs, fields = [], []
    for n in lengths:
        pr, *f = wl.pulled_front_1d(N=n, V=1.5, front_cell=24, A=1.1, b=1.0)
        prs.append(pr)
        fields.append(f)
    dtype = np.float32 if precision == "fp32" else np.float64
    f = [np.concatenate(a).astype(dtype) for a in zip(*fields)]
    return pf.run_batch(dict(prs[0], x0=12.0), lengths, [1.5, 0.7, 0.1], *f, precision=precision, max_steps=70,
                        steps_per_launch=25, launches_per_graph=1, check_every=70, tol=-1.0, want_fields=True,
                        cells_per_thread=cells)


@pytest.mark.parametrize("precision,cells,used", [("fp32", 1, 2), ("fp32", 2, 2), ("fp32", 4, 4), ("fp32", 8, 4),
                                                  ("fp64", 1, 2), ("fp64", 4, 2), ("fp64", 8, 2)])
def test_reported_cells_are_those_that_ran(precision, cells, used):
    assert run(precision, cells)["cells_per_thread"] == used


def test_cells_per_lane_change_no_bit():
    two, four = run("fp32", 2), run("fp32", 4)
    for k in ("phi", "cs", "cl", "k_v"):
        assert np.array_equal(two[k], four[k]), k
