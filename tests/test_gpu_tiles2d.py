"""FP64 2D grids on both tile shapes against the FP64 oracle: sizes at the edges of
a 16 x 8 tile, the largest grid that takes them (304 tiles on 152 SMs) and one
past it, every kind of boundary."""
import numpy as np
import pytest

import oracle
from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

from conftest import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(5, 4), (16, 8), (17, 9), (15, 7), (33, 25), (304, 128), (305, 128), (40, 961)])
@pytest.mark.parametrize("kw", [dict(lap=9, bc_lo=("noflux", "periodic"), bc_hi=("noflux", "periodic")),
                                dict(lap=5, a=0.2, bc_lo=("noflux", "noflux"), bc_hi=("dirichlet", "noflux"))])
def test_fp64_tiles(n, kw):
    pr, *f = wl.random_state(2, n, A=1.0, b=1.0, amp=0.1, seed=4, **kw)
    st = oracle.State(pr, *f)
    st.step(4)
    with pf.Sim(pr, "fp64") as s:
        s.set_fields(*f)
        s.step(4)
        for a, b in zip(s.get_fields(), (st.phi, st.cs, st.cl)):
            assert rel_err(a, b) <= 1e-11
