"""The choice among the autotuner's timings (csrc/autotune.h, host code)."""
import itertools
import os
import subprocess

import pytest

from paper_1902_02999_gb300 import build

SOURCE = r"""
#include "autotune.h"
#include <cstdio>
int main()
{
    double ms[maclab::autotune::CANDIDATES], several;
    for (;;) {
        for (double& m : ms)
            if (std::scanf("%lf", &m) != 1) return 0;
        if (std::scanf("%lf", &several) != 1) return 0;
        const maclab::autotune::Choice c = maclab::autotune::choose(ms, several);
        std::printf("%d %d\n", c.shape, c.several ? 1 : 0);
    }
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("autotune")
    src, exe = str(d / "choose.cpp"), str(d / "choose")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-I" + build.CSRC, "-o", exe, src])

    def run(rows):
        out = subprocess.run([exe], input="\n".join(" ".join("%r" % x for x in r) for r in rows), text=True,
                             capture_output=True, check=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


def test_shape_and_depth_agree(choose):
    """Whatever wins: a two-step shape only where the depth is two, that is
    where several steps per launch are off."""
    inf = float("inf")
    rows = []
    for fast, second, several in itertools.product(range(9), range(9), (0.5, 2.0, inf)):
        ms = [10.0 + k for k in range(9)]
        ms[second], ms[fast] = 5.0, 1.0
        rows.append(ms + [several])
    rows.append([3.0] + [inf] * 8 + [inf])           # FP64: shapes left out
    got = choose(rows)
    assert len(got) == len(rows)
    for row, (shape, several) in zip(rows, got):
        ms = row[:9]
        assert several == (row[9] < min(ms))
        if several:
            assert shape not in (6, 8)
            assert ms[shape] == min(m for k, m in enumerate(ms) if k not in (6, 8))
        else:
            assert ms[shape] == min(ms)
