"""Local circuits in batches of a few pairs, whose lock-step work lists have small blocks and hold
pairs of every boundary size together: traces, cancellation ratios and error estimates do not depend
on the batch, and agree with the ticket-queue sweep.

Tolerance: the two sweeps multiply and sum in different orders; 1e-11 of max(|Tr|, 1) as between any
two FP64 sweeps of these boundaries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# boundaries of a few bits beside ones of 2^14 amplitudes and more
@pytest.mark.parametrize("n,T", [(18, (20, 60, 20)), (13, (5, 45, 20)), (20, (60, 60, 1)), (10, (60, 60, 1))])
def test_few_pairs(fp, n, T, monkeypatch):
    def ens():
        return fp.Ensemble(fp.LOCAL, n, 1, 1, *T, seed=n, flags=fp.FLAG_SKIP_INFEASIBLE)
    count = 12
    for prec in (fp.PREC_FP64, fp.PREC_FP32_RAW):
        whole = ens().trace_batch(40, count, prec, with_err=True)
        for first, c in ((0, 1), (1, 2), (3, 5), (7, 5)):
            part = ens().trace_batch(40 + first, c, prec, with_err=True)
            for a, b in zip(part, whole):
                a, b = np.asarray(a), np.asarray(b)[first:first + c]
                assert np.allclose(a, b, rtol=1e-11 if prec == fp.PREC_FP64 else 1e-4, atol=1e-4 if prec else 1e-11, equal_nan=True)
        if prec == fp.PREC_FP64:
            w64 = whole
    monkeypatch.setenv("FP_SWEEP_CLUSTER", "16")
    ref = ens().trace_batch(40, count, fp.PREC_FP64, with_err=True)
    ok = ref[2] >= 0
    assert ok.sum() >= count - 2 and np.array_equal(ref[2], w64[2])
    assert np.all(np.abs(w64[0] - ref[0])[ok] <= 1e-11 * np.maximum(np.abs(ref[0][ok]), 1.0))
