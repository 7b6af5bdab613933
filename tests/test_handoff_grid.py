"""Choice of the two-node hand-off kernel's build and grid (handoff_grid.h),
compiled for the host.

The launch takes the build that the grid was sized for.  Its resident blocks
per SM come from the compiler's register count and may be above the minimum
that the build was made for, so they do not name the build.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_17917_gb300", "csrc")
MAIN = """
#include <cstdio>
#include "handoff_grid.h"
int main()
{
    int sms, a, b;
    long long t;
    while (scanf("%d %d %d %lld", &sms, &a, &b, &t) == 4) {
        const dg::HandoffGrid h = dg::handoff_grid(sms, a, b, t);
        printf("%d %d %d\\n", h.minb, h.per_sm, h.grid);
    }
}
"""


@pytest.fixture(scope="module")
def pick(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("grid")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "grid")], check=True)

    def run(rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        out = subprocess.run([str(d / "grid")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]

    return run


@pytest.mark.parametrize("occ4", [4, 5, 6])
@pytest.mark.parametrize("occ5", [0, 5, 6, 7])
def test_the_build_goes_with_its_own_occupancy(pick, occ4, occ5):
    sms = 152
    tiles = sorted({1, sms, *(m * sms * o + d for m in (1, 2, 3) for o in (4, 5, 6, 7) for d in (-1, 0, 1)), 10 ** 6})
    for t, (minb, per_sm, grid) in zip(tiles, pick([(sms, occ4, occ5, t) for t in tiles])):
        assert minb in ((4, 5) if occ5 else (4,))
        assert per_sm == (occ4 if minb == 4 else occ5)          # the launch is resident as a whole
        assert grid == min(t, sms * per_sm)
        cost = {m: o * -(-t // (sms * o)) for m, o in ((4, occ4), (5, occ5)) if o}
        assert cost[minb] == min(cost.values())
        assert minb == 4 or cost[5] < cost[4]
