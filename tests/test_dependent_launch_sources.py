"""Kernels started by programmatic dependent launch read a state that the kernel
before may still be writing when their blocks arrive: no read-only loads of it.
A stale read could not be provoked in a test, so the sources are read."""
import glob
import os
import re

from paper_2303_09671_gb300 import build as pfbuild


def test_state_inputs_take_coherent_loads():
    seen = set()
    for path in glob.glob(os.path.join(pfbuild.CSRC, "*.cu")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        if "launch_after(" not in text:
            continue
        assert "ld.global.nc" not in text, path
        for m in re.finditer(r"\b(\w+_kernel)\(([^;{]*?)\)\s*\{", text):
            if "_in" in m[2]:
                seen.add(m[1])
                assert not re.search(r"__restrict__\s+\w+_in\b", m[2]), m[1]
    assert {"march2d_kernel", "step2d_kernel", "step3d_kernel"} <= seen
