"""Several host threads, an ensemble each, contract depths (or resample groups) of different sizes at
once: what one thread's kernels need must not depend on what the other launches."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def side_by_side(calls, rounds):
    """calls: functions of no argument; each thread repeats its own and compares with its first result.
    (Short calls and many rounds: what a thread sets and what it launches lie a microsecond apart.)"""
    want = [c() for c in calls]
    errors = []

    def work(c, w):
        try:
            for _ in range(rounds):
                assert np.array_equal(c(), w, equal_nan=True)
        except Exception as e:   # noqa: BLE001  (handed to the test's thread)
            errors.append(e)

    ts = [threading.Thread(target=work, args=a) for a in zip(calls, want)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors[0]


def test_bootstraps_of_different_sizes(fp):
    import torch

    def call(n):
        ens = fp.Ensemble(fp.PARALLEL, 8, 2, 2, seed=1)
        t = torch.randn(2 * n, dtype=torch.float64, device="cuda")
        g = torch.zeros(n, dtype=torch.int32, device="cuda")
        return lambda: ens.bootstrap(t, g, n, 1, 1, seed=3)

    side_by_side([call(n) for n in (50_000, 6_000, 20_000, 8_000)], 3000)


# (kind, prec, depths of one kernel, q): FP64 integers and the FP32 boundary in shared memory,
# spiral windows, qutrits
@pytest.mark.parametrize("kind,prec,depths,q", [(0, 0, (2, 5, 3, 4), 2), (0, 1, (2, 6, 3, 5), 2), (3, 0, (4, 6, 5, 4), 2),
                                                (3, 1, (5, 7, 6, 5), 2), (0, 1, (3, 4, 2, 4), 3)])
def test_depths_of_different_sizes(fp, kind, prec, depths, q):
    def call(d):
        ens = fp.Ensemble(kind, 6, d, d, seed=d, q=q)
        return lambda: ens.trace_batch(0, 1, prec)[0]

    side_by_side([call(d) for d in depths], 1500)
