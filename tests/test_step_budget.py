"""Steps per launch of the multi-step Euler kernels (csrc/step_budget.h): a
launch lasts about a millisecond in FP64 as in FP32, by the step times measured
on one GB300."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_08571_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include "step_budget.h"
int main()
{
    int f64;
    long long cells, left;
    while (std::scanf("%d %lld %lld", &f64, &cells, &left) == 3)
        std::printf("%d %lld\\n", ripple::walk_steps(f64, cells, left), ripple::solo_steps(f64, cells, left));
    return 0;
}
"""
# cells, us a step of a field's launch, us a step of a served problem's round
TIMES = {0: [(64 ** 2, 4.0, 3.4), (512 ** 2, 6.0, 5.9), (1024 ** 2, 11.2, 11.2)],
         1: [(64 ** 2, 7.4, 12.8), (128 ** 2, 8.7, 15.9), (256 ** 2, 19.7, 39.9), (512 ** 2, 64, 124), (1024 ** 2, 240, 400)]}


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("budget")
    (d / "main.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "t")], check=True)

    def ask(f64, cells, left):
        out = subprocess.run([str(d / "t")], input=f"{f64} {cells} {left}\n", capture_output=True, text=True, check=True)
        return tuple(int(x) for x in out.stdout.split())
    return ask


@pytest.mark.parametrize("f64", [0, 1])
def test_a_launch_lasts_about_a_millisecond(steps, f64):
    for cells, us_field, us_solo in TIMES[f64]:
        kf, ks = steps(f64, cells, 10 ** 6)
        assert kf >= 1 and ks >= 8
        assert kf * us_field <= 1600
        assert ks * us_solo <= 1600 or ks == 8


def test_no_more_steps_than_remain(steps):
    for f64 in (0, 1):
        for left in (1, 3, 7):
            assert steps(f64, 64 * 64, left) == (left, left)
        assert steps(f64, 1, 10 ** 6)[0] <= 256 and steps(f64, 1 << 32, 10 ** 6) == (1, 8)
