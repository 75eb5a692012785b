"""The budget of bounded device waits (csrc/wait_budget.cuh), compiled for the host: polls add up to it, one
gap in which the kernel did not run does not use it up."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#define __host__
#define __device__
#include "wait_budget.cuh"
#include <cstdio>
#include <cstdlib>
// polls at the given clock values after a start at 0: the clock value at which the budget is spent, or -1
int main(int argc, char **argv) {
    long long now = 0, step = atoll(argv[2]), gap_at = atoll(argv[3]), gap = atoll(argv[4]), end = atoll(argv[5]);
    lbm::WaitBudget wait(now, atoll(argv[1]));
    while (now < end) {
        now += now < gap_at && now + step >= gap_at ? gap : step;
        if (wait.spent(now)) return printf("%lld", now) < 0;
    }
    printf("-1");
}
"""


@pytest.fixture(scope="module")
def polls(tmp_path_factory):
    d = tmp_path_factory.mktemp("wait")
    (d / "w.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1403_3746_gb300", "csrc"), "-o", str(d / "w"),
                    str(d / "w.cpp")], check=True)
    return lambda *a: int(subprocess.run([str(d / "w"), *map(str, a)], capture_output=True, check=True).stdout)


@pytest.mark.parametrize("budget,step", [(1 << 31, 5000), (1 << 31, 1 << 20), (200000, 700), (1000, 5000)])
def test_polls_add_up_to_the_budget(polls, budget, step):
    assert budget < polls(budget, step, 0, 0, 1 << 34) <= budget + step


def test_a_gap_without_polls_counts_little(polls):
    second = 2_000_000_000
    assert polls(1 << 31, 5000, 1000000, 60 * second, 61 * second) == -1
    assert polls(1 << 31, 5000, 1000000, 60 * second, 80 * second) > 60 * second
