"""The persistent sweep's launch shape on CPU: csrc/sweep_shape.h, a host-only
header, compiled into a small program that answers queries line by line."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_13936_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "sweep_shape.h"
int main() {
    std::printf("%d %d\n", lgb::kCoopMaxBlocks, lgb::kCoopWarps);
    int fit, tuned, sms, hubs;
    long long units, n;
    int nsteps, vpb;
    while (std::scanf("%d %d %d %lld %d %lld %d %d", &fit, &tuned, &sms, &units, &nsteps, &n, &vpb, &hubs) == 8) {
        const int per_sm = lgb::sweep_blocks_per_sm(fit, tuned);
        std::printf("%d\n", lgb::sweep_grid(per_sm, sms, units, nsteps, n, vpb, hubs != 0));
    }
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("shape")
    (d / "main.cc").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(d / "main.cc"), "-o", str(d / "shape")],
                   check=True)

    def query(cases):
        text = "\n".join(" ".join(str(int(x)) for x in c) for c in cases)
        out = subprocess.run([str(d / "shape")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return int(out[0]), int(out[1]), [int(x) for x in out[2:]]
    return query


def test_grid_stays_within_the_scratch_of_a_launch(ask):
    """Whatever more blocks would fit, a launch has at most two per SM: the
    words of a single hub's candidates are allocated for so many."""
    cases = [(fit, tuned, sms, units, nsteps, n, vpb, hubs)
             for fit in (1, 2, 3, 4, 8) for tuned in (0, 1, 2, 3, 32) for sms in (1, 132, 152)
             for units, nsteps, n in ((0, 1, 1), (10, 5, 300), (10**6, 47, 10**7), (10**9, 1, 2**31 - 1),
                                      (1, 1000, 1))
             for vpb in (256, 2048, 65536) for hubs in (0, 1)]
    most, _, grids = ask(cases)
    assert most == 2 and len(grids) == len(cases)
    for c, g in zip(cases, grids):
        assert 1 <= g <= min(most, c[0]) * c[2], (c, g)
        if c[1] > 0:
            assert g <= c[1] * c[2], (c, g)
