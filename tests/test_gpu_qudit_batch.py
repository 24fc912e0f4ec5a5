"""A qudit pair is fully determined by (seed, pair): its FP64 trace is the same bits wherever in a
batch the pair falls, also where its gates share a warp with those of other pairs or with none."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# gates per pair that are and are not multiples of a warp's 3 (q = 3) or 2 (q = 4)
@pytest.mark.parametrize("q,n,l", [(3, 4, 2), (3, 5, 3), (3, 8, 3), (3, 4, 4), (4, 3, 2), (4, 4, 3), (4, 6, 2)])
def test_trace_does_not_depend_on_the_batch(fp, q, n, l):
    ens = fp.Ensemble(fp.PARALLEL, n, l, l, seed=53, q=q)
    whole = ens.trace_batch(0, 60, fp.PREC_FP64)[0]
    for first, count in ((0, 1), (1, 1), (7, 1), (59, 1), (3, 2), (10, 7), (29, 31)):
        assert np.array_equal(ens.trace_batch(first, count, fp.PREC_FP64)[0], whole[first:first + count]), (first, count)
