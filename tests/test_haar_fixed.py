"""The fixed-point Haar sampler (haar_fixed.h), built for the host: Gaussian draws,
Gram-Schmidt columns and conversions against extended precision (long double), and
against the errors of a double-precision Householder factorisation of the same
matrices, which is the precision the gates had before.  CPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("haar") / "check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-I",
                           os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2205_09900_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cpp", "haar_fixed_check.cpp"), "-o", exe])
    out = {}
    for line in subprocess.check_output([exe, "100000"], text=True).splitlines():
        words = line.split()
        if words[0].startswith("qr"):
            out[words[0]] = {words[i]: (float(words[i + 1]), float(words[i + 3])) for i in range(1, len(words), 4)}
        else:
            out[" ".join(words[:-1])] = float(words[-1])
    return out


def test_gaussian_draws(report):
    # values up to 6.06 in units of 2^-59; the chain of truncated products is good to
    # a few units (a double holds them to 2^-53 = 1.1e-16 and more)
    assert report["gauss random"] <= 2.0 ** -54
    assert report["gauss edges"] <= 2.0 ** -54


@pytest.mark.parametrize("d", [4, 9, 16])
def test_unitary_factor(report, d):
    for name, (fixed, householder) in report[f"qr{d}"].items():
        assert fixed <= householder, name


def test_conversions_round_to_nearest(report):
    assert report["conversions"] == 0.0
