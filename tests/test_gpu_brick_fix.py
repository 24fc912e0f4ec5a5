"""FP64 brickwork sweep in 64-bit integers: every boundary size that takes it, and the
largest one that does not (n = 50, l = 7)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2, 2, 1), (3, 2, 9), (4, 3, 40), (8, 4, 17), (9, 5, 3), (50, 5, 2), (8, 6, 3), (51, 6, 2), (8, 7, 2), (50, 7, 2)]


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


@pytest.mark.parametrize("n,l,count", SIZES)
def test_self_pairs_to_a_few_ulp(fp, n, l, count):
    # Tr(U^dagger U) = 2^n; (n - 1)(l - 1) maps of error 2^-55 each, all with one sign, are
    # 8.2e-15 at n = 50, l = 7 (which FP64 arithmetic sweeps: 1e-13)
    e = fp.Ensemble(fp.PARALLEL, n, l, seed=5 + l, flags=fp.FLAG_SELF_PAIR)
    tr = e.trace_batch(0, count, fp.PREC_FP64)[0]
    e.close()
    assert np.abs(tr / 2.0 ** n - 1).max() <= (1e-13 if (n, l) == (50, 7) else 1e-14)


@pytest.mark.parametrize("n,l,count", SIZES[:-1])
@pytest.mark.parametrize("diagonal", [False, True])
def test_matches_the_generic_sweep(fp, n, l, count, diagonal):
    # the generic sweep in FP64 arithmetic, both within 1e-12 of max(|Tr|, 1)
    flags = fp.FLAG_DIAGONAL_GATES if diagonal else 0
    a = fp.Ensemble(fp.PARALLEL, n, l, seed=3, flags=flags)
    b = fp.Ensemble(fp.PARALLEL, n, l, seed=3, flags=flags | fp.FLAG_GENERIC_ONLY)
    ta = a.trace_batch(0, count, fp.PREC_FP64)[0]
    tb = b.trace_batch(0, count, fp.PREC_FP64)[0]
    a.close()
    b.close()
    assert (np.abs(ta - tb) / np.maximum(np.abs(tb), 1)).max() <= 2e-12
