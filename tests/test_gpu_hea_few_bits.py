"""HEA boundaries of 2 and 4 bits (L = 2, 3) in FP64, a lane per amplitude: pairs that fill a warp, a
CTA or neither, against the generic sweep, and the same bits wherever in a batch a pair falls.

Tolerance: both sweeps are FP64, each within 1e-12 of max(|Tr|, 1)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L", [(2, 2), (3, 2), (50, 2), (2, 3), (5, 3), (51, 3)])
@pytest.mark.parametrize("count", [1, 3, 8, 35])
def test_few_bits(fp, n, L, count):
    a = fp.Ensemble(fp.HEA, n, L, seed=3)
    b = fp.Ensemble(fp.HEA, n, L, seed=3, flags=fp.FLAG_GENERIC_ONLY)
    ta, ka, _ = a.trace_batch(5, count, fp.PREC_FP64)
    tb, kb, _ = b.trace_batch(5, count, fp.PREC_FP64)
    assert (np.abs(ta - tb) / np.maximum(np.abs(tb), 1)).max() <= 2e-12
    well = kb < 1e6
    assert np.allclose(ka[well], kb[well], rtol=1e-5)
    for p in {0, count - 1}:
        assert a.trace_batch(5 + p, 1, fp.PREC_FP64)[0][0] == ta[p]
    s = fp.Ensemble(fp.HEA, n, L, seed=4, flags=fp.FLAG_SELF_PAIR)
    assert np.abs(s.trace_batch(0, count, fp.PREC_FP64)[0] / 2.0 ** n - 1).max() <= 1e-13
