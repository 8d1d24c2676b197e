"""The order of the launches of a grouped compression (csrc/fa_row_groups.h), on the host: every row with moments is launched once,
a launch is chained only behind one of its own call, and no launch writes moments where the one in front of it still reads."""
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11886_b200", "csrc")
MAIN = r"""
#include "fa_row_groups.h"
#include <cstdio>
int main() {
    int B; unsigned long long fit, live;
    while (std::scanf("%d %llu %llu", &B, &fit, &live) == 3) {
        fa::for_row_groups(B, (size_t)fit, [&](int b) { return (live >> b & 1) != 0; },
                           [](const fa::RowGroup& g) { std::printf("%d,%d,%d,%d,%d ", g.b0, g.nb, g.second, g.wait_first, g.chained); return 0; });
        std::printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def groups(tmp_path_factory):
    d = tmp_path_factory.mktemp("row_groups")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    cases = [(B, fit, live) for B in range(1, 8) for fit in (1, 2, 3, 4, 5, 7, 9) for live in range(1, 1 << B)]
    text = "".join("%d %d %d\n" % c for c in cases)
    lines = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    return [(c, [tuple(int(x) for x in g.split(",")) for g in line.split()]) for c, line in zip(cases, lines)]


def test_every_row_with_moments_once_and_chained_behind_a_launch_of_the_call(groups):
    for (B, fit, live), gs in groups:
        rows = list(itertools.chain(*(range(b0, b0 + nb) for b0, nb, *_ in gs)))
        assert len(set(rows)) == len(rows) and all(b in rows for b in range(B) if live >> b & 1), (B, fit, live)
        assert [g[4] for g in gs] == [0] + [1] * (len(gs) - 1), (B, fit, live, gs)
        assert all(any(live >> b & 1 for b in range(g[0], g[0] + g[1])) for g in gs)
        assert all(g[1] <= (fit if len(gs) == 1 and fit >= B else max(1, fit // 2)) for g in gs), (B, fit, live, gs)


def test_no_launch_writes_where_the_one_in_front_reads(groups):
    """Neighbours among the launches of a call take different halves, or the later one waits."""
    for (B, fit, live), gs in groups:
        for (*_, second, _, _), (*_, second_next, wait, _) in zip(gs, gs[1:]):
            assert second != second_next or wait, (B, fit, live, gs)
        assert fit >= 2 or not any(g[2] for g in gs)
