"""A reverse sweep whose checkpoints do not fit the device memory that is left takes
them farther apart, with the same results."""
import numpy as np
import pytest

from paper_2303_09671_gb300 import pf
from paper_2303_09671_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_dense_checkpoints_beyond_the_memory():
    """4 fronts of 1024 cells, a checkpoint of 24 bytes a cell before each of 30,000
    steps: 2.9 GB, with 2 GB left on the device; every second one fits."""
    pr, *f = wl.pulled_front_1d(N=1024, V=0.5, front_cell=200, A=1.1, b=1.0)
    f = [np.tile(a.astype(np.float32), 4) for a in f]
    args = (pr, [1024] * 4, [0.1, 0.2, 0.3, 0.5], *f, 30000)
    ref = pf.adjoint(*args, mode="reverse", checkpoint_every=173)
    free, _ = torch.cuda.mem_get_info()
    held = torch.empty(free - (2 << 30), dtype=torch.uint8, device="cuda")
    try:
        r = pf.adjoint(*args, mode="reverse", checkpoint_every=1)
    finally:
        del held
        torch.cuda.empty_cache()
    assert np.isfinite(ref["dk"]).all()
    assert np.array_equal(r["k"], ref["k"])
    assert np.abs(r["dk"] - ref["dk"]).max() <= 1e-5 * np.abs(ref["dk"]).max()
