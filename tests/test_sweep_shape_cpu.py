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
    int fit, tuned, sms, vpb, hubs, runs;
    long long n;
    while (std::scanf("%d %d %d %lld %d %d %d", &fit, &tuned, &sms, &n, &vpb, &hubs, &runs) == 7) {
        lgb::SweepWork w;
        for (long long steps, units; runs > 0; --runs)  // steps of units each
            if (std::scanf("%lld %lld", &steps, &units) == 2)
                while (steps-- > 0) w.step(units);
        std::printf("%d\n", lgb::sweep_grid(fit, tuned, sms, w, n, vpb, hubs != 0));
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
        text = "\n".join(" ".join(str(int(x)) for x in (*c[:6], len(c[6]), *sum(c[6], ()))) for c in cases)
        out = subprocess.run([str(d / "shape")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return int(out[0]), int(out[1]), [int(x) for x in out[2:]]
    return query


def test_grid_stays_within_the_scratch_of_a_launch(ask):
    """Whatever more blocks would fit, a launch has at most two per SM: the
    words of a single hub's candidates are allocated for so many."""
    cases = [(fit, tuned, sms, n, vpb, hubs, steps)
             for fit in (1, 2, 3, 4, 8) for tuned in (0, 1, 2, 3, 32) for sms in (1, 132, 152)
             for n, steps in ((1, []), (300, [(5, 2)]), (10**7, [(47, 30000)]), (2**31 - 1, [(1, 10**9)]),
                              (10**6, [(900, 1), (40, 900)]))
             for vpb in (256, 2048, 65536) for hubs in (0, 1)]
    most, _, grids = ask(cases)
    assert most == 2 and len(grids) == len(cases)
    for c, g in zip(cases, grids):
        assert 1 <= g <= min(most, c[0]) * c[2], (c, g)
        if c[1] > 0:
            assert g <= c[1] * c[2], (c, g)


def test_wide_steps_among_thin_ones_keep_their_blocks(ask):
    """One block takes a sweep only while its steps, one by one, fit its
    warps: the average of a thousand thin layers and a few wide steps does
    not put the wide ones on one SM."""
    full, n = 152, 300_000
    _, warps, grids = ask([
        (2, 0, full, n, 2048, 0, [(47, 16)]),            # every step in one round
        (2, 0, full, n, 2048, 0, [(47, 17)]),            # each a second round
        (2, 0, full, n, 2048, 0, [(800, 1), (10, 900)]),  # 12 units on average
        (2, 0, full, n, 2048, 0, [(800, 1), (1, 20)]),    # one extra round in 801 steps
        (2, 0, full, 1000, 2048, 0, []),
    ])
    assert warps == 16
    assert grids[0] == 1 and grids[3] == 1 and grids[4] == 1
    assert grids[1] == (n + 2047) // 2048
    assert grids[2] == (n + 2047) // 2048


@pytest.mark.parametrize("steps", [[(47, 700)], [(47, 9700)], [(47, 9800)], [(47, 10**6)]])
def test_blocks_per_sm_are_the_handle_s_choice(ask, steps):
    """coop_blocks_per_sm: 0 by a step's work, else one or two (three mean
    two) whatever the work."""
    n = 10**7  # two blocks per SM and more by its vertices
    _, warps, (rule, one, two, three) = ask([(2, t, 152, n, 2048, 0, steps) for t in (0, 1, 2, 3)])
    assert one == 152 and two == three == 304
    assert rule == (two if steps[0][1] >= 4 * warps * 152 else one)
