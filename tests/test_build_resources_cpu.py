"""What the compiler gave the persistent sweeps (the build's ptxas report):
the form with two blocks per SM, which the largest graphs run, has 64
registers a thread and must not spill what its units hold."""
import os
import re
import shutil

import pytest

from paper_2312_13936_gb300 import _build


def _kernels(unit):
    path = _build.resource_log(unit)
    if not os.path.exists(path):
        if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
            pytest.skip("no nvcc")
        _build.build(force=True)
    found = {}
    for m in re.finditer(r"Compiling entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads"
                         r".*?Used (\d+) registers", open(path).read(), re.S):
        if "k_sweep_coop" in m[1]:
            found[m[1]] = (int(m[2]), int(m[3]), int(m[4]))
    return found


@pytest.mark.parametrize("unit,forms,spill", [("k_sweep_async_2", 4, 256), ("k_sweep_async_1", 4, 512),
                                              ("k_sweep_det64_1", 8, 512), ("k_sweep_det64_2", 8, 1024),
                                              ("k_sweep_det_1", 8, 1024), ("k_sweep_det_2", 8, 1024)])
def test_persistent_sweeps_spill_little(unit, forms, spill):
    """At most spill bytes of spill stores, and of spill loads, in each form
    (the asynchronous two-block forms stored 2,000 to 3,394)."""
    got = _kernels(unit)
    assert len(got) == forms, sorted(got)
    for name, (st, ld, regs) in got.items():
        assert st <= spill and ld <= spill, (name, st, ld, regs)
        assert regs <= (64 if unit.endswith("_2") else 128), (name, regs)
