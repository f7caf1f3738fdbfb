"""The form of the FP32 stage kernel beside other solvers (csrc/stage_form.h), compiled for the host."""
import os
import subprocess

from conftest import ROOT

HARNESS = r"""
#include "stage_form.h"
#include <cstdio>
#include <thread>
#include <vector>
using namespace vk;
int main()
{
    std::printf("%d %d %d %d %d %d\n", stage_form(128, 0), stage_form(300, 0), stage_form(128, 128),
                stage_form(128, 480), stage_form(128, 481), stage_form(300, 5000));
    // handles of several threads: each sees the others' tiles while they are in flight, none are left at the end
    InFlight a, b;
    long long bad = a.enter(100) != 0;
    bad += b.enter(7) != 100;
    bad += a.enter(100) != 7;   // entered again without a wait: counted once
    a.leave();
    a.leave();
    bad += b.enter(7) != 0;
    b.leave();
    std::vector<std::thread> t;
    for (int k = 0; k < 4; ++k)
        t.emplace_back([] {
            InFlight f;
            for (int q = 0; q < 20000; ++q) {
                f.enter(3);
                f.leave();
            }
        });
    for (auto &x : t) x.join();
    std::printf("%lld %lld\n", bad, tiles_in_flight.load());
}
"""


def test_forms_and_the_count_of_tiles_in_flight(tmp_path):
    (tmp_path / "f.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I",
                    os.path.join(ROOT, "paper_2504_15574_gb300", "csrc"), str(tmp_path / "f.cpp"), "-o",
                    str(tmp_path / "f")], check=True)
    out = subprocess.run([str(tmp_path / "f")], capture_output=True, text=True, check=True).stdout.split()
    assert out[:6] == ["0", "0", "1", "1", "2", "2"]      # alone, shared, crowded
    assert out[6:] == ["0", "0"]
