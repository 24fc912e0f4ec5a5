"""Fixed-point Haar gates: columns are neither too long nor too short on average, so that a trace's
error does not grow with its number of gates.

Tolerance: a quarter of 2^-60 per column keeps a thousand gates below 2^-52; the means are known to
0.03 units and better (rms of at most 20 units over 80,000 columns and more)."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_columns_have_length_one_on_average(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-Wno-unknown-pragmas",
                           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2205_09900_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cpp", "haar_bias_check.cpp"), "-o", exe])
    for line in subprocess.check_output([exe], text=True).splitlines():
        d, mean, rms = (float(x) for x in line.split())
        assert abs(mean) <= 0.25 and rms <= 20, line


@pytest.mark.gpu
@pytest.mark.parametrize("l", [2, 3, 4])
def test_qutrit_self_pairs_have_no_bias(fp, l):
    # Tr(U^dagger U) = 3^50; 200 pairs of rms error 2e-15 at most (FP64 sweep): the mean is known to
    # 6e-16 (4 sigma), and 200 columns' worth of a quarter of 2^-60 per qutrit pair of gates adds 1e-16
    ens = fp.Ensemble(fp.PARALLEL, 50, l, l, seed=11, q=3, flags=fp.FLAG_SELF_PAIR)
    r = ens.trace_batch(0, 200, fp.PREC_FP64)[0] / 3.0 ** 50 - 1
    assert abs(r.real.mean()) <= 8e-16 and np.sqrt(np.mean(np.abs(r) ** 2)) <= 2e-15, (r.real.mean(), np.abs(r).max())
