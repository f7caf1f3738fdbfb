"""The graphs that a rollout captures and launches (csrc/lc_rollout.h), compiled for the host."""
import os
import subprocess

import pytest
from conftest import ROOT

HARNESS = r"""
#include "lc_rollout.h"
#include <cstdio>
#include <cstdlib>
int main(int, char **a)
{
    const vk::RolloutPlan p = vk::rollout_plan(atoi(a[1]), atoll(a[2]), atoi(a[3]), atoi(a[4]));
    std::printf("%d %d %d %d %d\n", p.capture_one, p.capture_many, p.many, p.ones, vk::ROLL_STEPS);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "p.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2504_15574_gb300", "csrc"),
                    str(d / "p.cpp"), "-o", str(d / "p")], check=True)

    def run(*a):
        return tuple(map(int, subprocess.run([str(d / "p"), *map(str, a)], capture_output=True, text=True,
                                             check=True).stdout.split()))
    return run


@pytest.mark.parametrize("steps", [1, 7, 8, 10, 64, 95, 96, 100, 1000])
@pytest.mark.parametrize("taken", [0, 50, 400])
@pytest.mark.parametrize("one,many", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_a_rollout_captures_what_it_launches_and_no_more(plan, steps, taken, one, many):
    c1, cm, n, m, long = plan(steps, taken, one, many)
    assert n * long + m == steps
    assert c1 == (m > 0 and not one) and cm == (n > 0 and not many)
    if m >= long:                          # whole long graphs are left out only where none is captured yet
        assert n == 0 and not many


def test_a_state_that_runs_briefly_pays_for_one_small_graph(plan):
    for steps in (1, 8, 10, 16, 48):
        assert plan(steps, 0, 0, 0)[:2] == (1, 0)
    assert plan(96, 0, 0, 0)[:2] == (0, 1)          # a long one for the long graph alone, if that divides it
    assert plan(10, 90, 1, 0)[:2] == (0, 1)         # one that goes on for the long graph once it pays
