"""Large FP32 2D grids (the row-marching kernel, at least four rows per warp) against
the FP64 oracle: widths at the edges of the 60-column strips and of the two-cell
lanes, ragged last rows, every kind of boundary, the general physics.

Tolerance 1e-5 of the field's largest value after four steps: inputs and results are
rounded at 6e-8, the logarithms carry 2.4e-7 absolute, and a step changes a field by a
rate with relative error below 1e-5 times at most a tenth of the field."""
import numpy as np
import pytest

import oracle
from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

from conftest import rel_err

pytestmark = pytest.mark.gpu

KINDS = [dict(lap=9, bc_lo=("noflux", "periodic"), bc_hi=("noflux", "periodic")),
         dict(lap=5, a=0.2, bc_lo=("periodic", "noflux"), bc_hi=("periodic", "noflux"), G_theta=0.0),
         dict(lap=9, bc_lo=("noflux", "noflux"), bc_hi=("dirichlet", "noflux")),
         dict(lap=5, bc_lo=("noflux", "noflux"), bc_hi=("noflux", "dirichlet")),
         dict(lap=9, a=0.2, interp="cubic", mobility="const")]


def state(n, kw):
    """A front along x; a stripe of solid instead where x is periodic, and melt
    toward a Dirichlet boundary at high y (no jump of phi at a boundary)."""
    pr, phi, cs, cl = wl.random_state(2, n, A=1.0, b=1.0, amp=0.1, seed=4, **kw)
    if kw.get("bc_lo", ("",))[0] == "periodic":
        phi = 4.0 * phi * (1.0 - phi)
    if kw.get("bc_hi", ("", ""))[1] == "dirichlet":
        y = np.arange(n[1])[:, None]
        phi = phi * 0.5 * (1.0 - np.tanh((y - 0.7 * n[1]) / 3.0))
    return (pr, *(a.astype(np.float32) for a in (phi, cs, cl)))


@pytest.mark.parametrize("n", [(60, 5474), (61, 2739), (59, 5501), (122, 1830), (1201, 301), (1024, 512),
                               (7, 5600), (5600, 62)])
@pytest.mark.parametrize("kw", KINDS)
def test_fp32_march(n, kw):
    pr, *f = state(n, kw)
    st = oracle.State(pr, *(a.astype(np.float64) for a in f))
    st.step(4)
    with pf.Sim(pr, "fp32") as s:
        s.set_fields(*f)
        s.step(4)
        for a, b in zip(s.get_fields(), (st.phi, st.cs, st.cl)):
            assert rel_err(a, b) <= 1e-5
