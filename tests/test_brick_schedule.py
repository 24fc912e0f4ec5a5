"""Tile schedules of the brickwork and HEA sweeps on the host: every gate once and in
order, exchange maps conflict-free, and no more windows than the greedy choice took at
the benchmark's depths.  CPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_09900_gb300", "csrc")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("sched") / "check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                           "-I", CSRC, os.path.join(ROOT, "tests", "cpp", "brick_schedule_check.cpp"),
                           os.path.join(CSRC, "brick_plan.cpp"), "-o", exe])

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], capture_output=True, text=True)
        assert out.returncode == 0, out.stdout
        return int(out.stdout.split()[2])
    return run


@pytest.mark.parametrize("n,l,K,low,R,kind", [(2, 8, 12, 3, 5, 0), (3, 9, 12, 3, 5, 0), (7, 8, 13, 5, 4, 0),
                                              (12, 13, 12, 2, 5, 0), (64, 8, 14, 5, 5, 0), (51, 9, 13, 4, 3, 0),
                                              (50, 7, 12, 5, 5, 0), (20, 10, 14, 5, 4, 0), (6, 8, 12, 3, 5, 1),
                                              (9, 9, 13, 5, 4, 1)])
def test_schedule_is_valid(check, n, l, K, low, R, kind):
    check(n, l, K, low, R, kind)


@pytest.mark.parametrize("l,low,greedy", [(8, 3, 65), (9, 3, 78), (10, 3, 98), (11, 2, 105)])
def test_no_more_windows_than_greedy(check, l, low, greedy):
    assert check(50, l, 12, low, 5, 0) <= greedy
