"""Energy, solute and front of FP32 and FP64 states against the FP64 oracle over
dimensions, stencils, boundaries and grid shapes that put cells at every kind of
edge."""
import numpy as np
import pytest

import oracle
from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    (1, (67,), dict(bc_lo=("noflux",), bc_hi=("dirichlet",), G_theta=0.02)),
    (1, (3,), dict()),
    (2, (33, 5), dict(lap=5)),
    (2, (70, 21), dict(lap=9, bc_lo=("noflux", "periodic"), bc_hi=("dirichlet", "periodic"), G_theta=0.01)),
    (3, (19, 6, 5), dict(lap=7, bc_lo=("periodic",) * 3, bc_hi=("periodic",) * 3)),
    (3, (40, 13, 7), dict(lap=19, interp="cubic", a=-0.3)),
    (3, (9, 8, 3), dict(lap=19, bc_lo=("noflux", "dirichlet", "noflux"), bc_hi=("dirichlet", "noflux", "dirichlet"))),
]


@pytest.mark.parametrize("dim,n,kw", CASES)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_energy_solute_front(dim, n, kw, precision):
    """The state of an FP32 handle is FP32 pairs of the inputs' c: its sums are
    compared with the oracle's on the same FP32 inputs.  The conversion leaves
    2^-24 in p, which shifts c by p's error times d (below 6e-8 per cell, of a
    total near 1 per cell); the energy follows c by its chemical potentials, of
    order 10: 1e-6 of the sum of magnitudes bounds both, 1e-12 an FP64 state."""
    pr, *f = wl.random_state(dim, n, A=1.5, b=0.3, seed=3, **kw)
    if precision == "fp32":
        f = [a.astype(np.float32).astype(np.float64) for a in f]
    st = oracle.State(pr, *f)
    with pf.Sim(pr, precision) as s:
        s.set_fields(*f)
        E, S = s.energy(), s.solute_total()
        x, _, c = s.front()
    tol = 1e-12 if precision == "fp64" else 1e-6
    Eo = st.energy()
    cells = int(np.prod(n)) * pr["dx"] ** dim
    assert abs(E - Eo) <= tol * max(abs(Eo), cells)
    h = f[0] ** 3 * (6 * f[0] ** 2 - 15 * f[0] + 10) if pr["interp"] == "quintic" else f[0] ** 2 * (3 - 2 * f[0])
    pp = h + pr["a"] * (f[0] - 0.5) * (f[0] * (1 - f[0])) ** 2
    cc = pp * f[1] + (1 - pp) * f[2]
    assert abs(S - cc.sum() * pr["dx"] ** dim) <= tol * cells
    assert abs(c - cc.max()) <= tol
    cross = (f[0][..., :-1] >= 0.5) & (f[0][..., 1:] < 0.5)
    a, b = f[0][..., :-1][cross], f[0][..., 1:][cross]
    i = np.nonzero(cross)[-1]
    if len(i):
        assert abs(x - ((i + 0.5 + (a - 0.5) / (a - b)) * pr["dx"]).max()) <= 1e-12 * max(1.0, abs(x))
    else:
        assert np.isnan(x)


def test_fp32_energy_matches_fp64_arithmetic():
    """The allocation-free entry reads FP32 fields exactly, so its FP32-pair sums
    must equal the FP64 formula on them to the pairs' 2^-45 per cell."""
    torch = pytest.importorskip("torch")
    pr, *f = wl.random_state(3, (70, 33, 20), A=1.5, b=0.3, seed=5, G_theta=0.01, amp=0.5)
    f = [a.astype(np.float32) for a in f]
    st = oracle.State(pr, *[a.astype(np.float64) for a in f])
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    pf.energy_solute_noalloc(pr, *[torch.from_numpy(a).cuda() for a in f], out)
    Eo = st.energy()
    assert abs(out[0].item() - Eo) <= 3e-14 * max(abs(Eo), 70 * 33 * 20 * 10 * pr["dx"] ** 3)


def test_energy_of_a_broken_state():
    """A negative concentration: not finite, as in FP64 arithmetic."""
    pr, phi, cs, cl = wl.random_state(2, (40, 12), seed=1)
    cs[3, 3] = -0.5
    with pf.Sim(pr, "fp32") as s:
        s.set_fields(phi, cs, cl)
        with pytest.raises(pf.PFError) as e:
            s.energy()
        assert e.value.code == pf.PF_ENONFINITE
