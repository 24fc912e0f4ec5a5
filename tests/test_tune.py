"""The autotuner's timing of variants on the host (tune.h): a variant's first run, which loads its
code, does not decide.  CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_09900_gb300", "csrc")


def test_first_runs_are_not_counted(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-Wall", "-Werror", "-I", CSRC,
                           os.path.join(ROOT, "tests", "cpp", "tune_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
