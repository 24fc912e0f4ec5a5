"""Windows of the spiral sweep on the host: maps along the window's walk, and only zeros
in the groups that a window leaves out.  CPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_09900_gb300", "csrc")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("walk") / "check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                           "-I", CSRC, "-I", "/usr/local/cuda/include",
                           os.path.join(ROOT, "tests", "cpp", "spiral_walk_check.cpp"),
                           os.path.join(CSRC, "planner.cpp"), "-o", exe])
    return exe


@pytest.mark.parametrize("n,L,R,split", [(3, 5, 4, 0), (5, 5, 5, 0), (7, 6, 4, 1), (8, 6, 5, 2), (50, 6, 4, 2),
                                         (9, 7, 5, 1), (51, 7, 4, 2), (12, 8, 5, 1), (6, 8, 5, 2)])
def test_windows_walk_and_leave_out_zeros(check, n, L, R, split):
    out = subprocess.run([check, str(n), str(L), str(R), str(split)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert L < 8 or int(out.stdout.split()[4]) > 0   # the rule is in use
