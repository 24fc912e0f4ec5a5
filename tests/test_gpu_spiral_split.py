"""Spiral sweep with a pair spread over 1 to 16 CTAs, and depths side by side."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fp():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_09900_gb300 import build
    build.build()
    import paper_2205_09900_gb300 as fpm
    fpm.load()
    return fpm


# counts at which the FP64 sweep takes 16, 8, 4 CTAs and 1 CTA per pair
@pytest.mark.parametrize("L,count", [(8, 1), (8, 12), (8, 30), (7, 1), (7, 5), (7, 40), (6, 1), (5, 3)])
def test_few_fp64_pairs_match_map_by_map(fp, L, count, monkeypatch):
    # FP64 to 1e-10 of max(|Tr|, 1)
    out = []
    for win in (None, "0"):
        if win:
            monkeypatch.setenv("FP_SPIRAL_WIN", win)
        e = fp.Ensemble(fp.HEA_PAULI, 50, L, seed=9 + L)
        out.append(e.trace_batch(0, count, fp.PREC_FP64)[0])
        e.close()
    assert (np.abs(out[0] - out[1]) / np.maximum(np.abs(out[1]), 1)).max() <= 1e-10


@pytest.mark.parametrize("n,lo,hi,count", [(3, 2, 9, 200), (50, 2, 8, 150), (20, 7, 8, 2)])
def test_depths_side_by_side_match_depth_by_depth(fp, n, lo, hi, count):
    # FLAG_TIMING runs one depth after another; FP32 sweeps are the same in both orders
    a = fp.Ensemble(fp.HEA_PAULI, n, lo, hi, seed=4)
    b = fp.Ensemble(fp.HEA_PAULI, n, lo, hi, seed=4, flags=fp.FLAG_TIMING)
    for _ in range(2):
        ta, _, ga = a.trace_batch(0, count, fp.PREC_FP32_RAW)
        tb, _, gb = b.trace_batch(0, count, fp.PREC_FP32_RAW)
        assert np.array_equal(ga, gb) and np.array_equal(ta, tb)
    a.close()
    b.close()
