"""FP64 traces of the HEA sweep in 64-bit integers: at least FP64's precision."""
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


@pytest.mark.parametrize("n,L,count", [(2, 4, 3), (50, 4, 5), (50, 5, 33), (51, 6, 6), (50, 7, 3), (50, 8, 2)])
def test_self_pairs_to_a_few_ulp(fp, n, L, count):
    # Tr(U^dagger U) = 2^n; at most 4 products per qubit of error 2^-55 and 2 (L - 1) slots
    # of error 2^-57 each, all with one sign: below 2e-14
    e = fp.Ensemble(fp.HEA, n, L, seed=5 + L, flags=fp.FLAG_SELF_PAIR)
    tr = e.trace_batch(0, count, fp.PREC_FP64)[0]
    e.close()
    assert np.abs(tr / 2.0 ** n - 1).max() <= 2e-14


@pytest.mark.parametrize("n,L,count", [(3, 4, 40), (12, 5, 40), (9, 6, 20), (10, 7, 9), (12, 8, 5)])
def test_matches_the_generic_sweep(fp, n, L, count):
    # the generic sweep in FP64 arithmetic, both within 1e-12 of max(|Tr|, 1)
    a = fp.Ensemble(fp.HEA, n, L, seed=3)
    b = fp.Ensemble(fp.HEA, n, L, seed=3, flags=fp.FLAG_GENERIC_ONLY)
    ta = a.trace_batch(0, count, fp.PREC_FP64)[0]
    tb = b.trace_batch(0, count, fp.PREC_FP64)[0]
    a.close()
    b.close()
    assert (np.abs(ta - tb) / np.maximum(np.abs(tb), 1)).max() <= 2e-12
