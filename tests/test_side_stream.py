"""A side stream exists with its event or not at all (side_stream.h, on a fake CUDA runtime).  CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_09900_gb300", "csrc")


def test_a_failed_creation_leaves_nothing(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-Wall", "-I", CSRC,
                           "-I", "/usr/local/cuda/include",
                           os.path.join(ROOT, "tests", "cpp", "side_stream_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
