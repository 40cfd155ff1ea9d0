"""F_h and S_h of FP32 fields as FP64 arithmetic gives them: against extended
precision on states whose cells all repeat a few values, so that no rounding of a
cell's terms averages out, with one and with many cells per thread."""
import numpy as np
import pytest

from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
q = np.longdouble


def exact_of_columns(pr, phi, cs, cl):
    """(F_h, S_h, sum of |F_h's terms|) per (y, z) column of a state that varies along
    x only, with mirror sides: 64 bits or more of mantissa."""
    f, s, l = (a.astype(q) for a in (phi, cs, cl))
    dx = q(pr["dx"])
    g = f * (1 - f)
    p = f ** 3 * (6 * f * f - 15 * f + 10) if pr["interp"] == "quintic" else f * f * (3 - 2 * f)
    p = p + q(pr["a"]) * (f - q(0.5)) * g * g
    theta = q(pr["theta_ref"]) - q(pr["G_theta"]) * ((np.arange(len(f)) + q(0.5)) * dx - q(pr["x0"]))
    fs = -(1 - q(pr["k_e"])) * theta + s * (np.log(s) - np.log(q(pr["k_e"])) - 1)
    fl = l * (np.log(l) - 1)
    step = np.diff(f) ** 2
    grad = np.concatenate([step, [0]]) + np.concatenate([[0], step])   # both neighbours of every cell
    e = q(pr["H"]) * g * g + p * fs + (1 - p) * fl + q(pr["sigma"]) * grad / (4 * dx * dx)
    vol = dx ** 3
    return e.sum() * vol, (p * s + (1 - p) * l).sum() * vol, np.abs(e).sum() * vol


@pytest.mark.parametrize("kw", [dict(), dict(interp="cubic", a=-0.3, G_theta=0.01)])
@pytest.mark.parametrize("columns", [(8, 9), (512, 320)])
def test_fp32_sums_carry_fp64_precision(columns, kw):
    """Unit u = 2^-53 of the sum of magnitudes.  Beyond a cell's own terms (1 u), the
    result passes about 23 roundings of partial sums (a thread's runs, the block's
    tree, the blocks' partials), of which all but the last ten are averaged over
    threads: 1.8 u rms; 8 u is over four times that.  (512 x 320 columns of 64 cells:
    33 per thread of the full grid.)"""
    ny, nz = columns
    pr, *_ = wl.random_state(3, (64, ny, nz), lap=7, **kw)
    x = (np.arange(64) + 0.5) * pr["dx"]
    phi = wl.tanh_profile(x, 20 * pr["dx"]).astype(np.float32)
    cs = np.full(64, pr["k_e"], np.float32)
    cl = np.ones(64, np.float32)
    cl[40:] = 0.9
    F, S, mag = exact_of_columns(pr, phi, cs, cl)
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    fields = [torch.from_numpy(a).cuda().repeat(nz, ny, 1).contiguous() for a in (phi, cs, cl)]
    pf.energy_solute_noalloc(pr, *fields, out)
    n, u = ny * nz, q(2) ** -53
    assert abs(q(out[0].item()) - n * F) <= 8 * u * n * mag
    assert abs(q(out[1].item()) - n * S) <= 8 * u * n * S


def test_fp32_energy_beyond_the_words_range():
    """Values whose squares or products leave FP32's range are summed in FP64: phi of
    1e20, and concentrations of 1e-30."""
    for phi, c, lap in ((1e20, 0.5, 9), (0.25, 1e-30, 5)):
        pr, *_ = wl.random_state(2, (24, 10), lap=lap, amp=0.1)
        f = np.full((10, 24), phi, np.float32)
        f[:, 12:] *= np.float32(0.5)
        s, l = (np.full((10, 24), v, np.float32) for v in (c, 2 * c))
        out = []
        for precision, dtype in (("fp32", np.float32), ("fp64", np.float64)):
            o = torch.zeros(2, dtype=torch.float64, device="cuda")
            pf.energy_solute_noalloc(pr, *[torch.from_numpy(a.astype(dtype)).cuda() for a in (f, s, l)], o,
                                     precision=precision)
            out.append(o.cpu().numpy())
        assert np.isfinite(out[1]).all()
        assert np.all(np.abs(out[0] - out[1]) <= 1e-14 * np.abs(out[1]))
