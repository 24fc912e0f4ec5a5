"""Bootstrap of small batches (one CTA lists the groups), of few and of many groups, at the edges of
those three forms: members in increasing pair order, draws and sums as the oracle's.

Tolerance: |t|^2 within 2^-52 on either side gives its k-th power within 2 k 2^-52, and a sum of N
positive terms is within N 2^-53 of its value: below 1e-12 for N <= 7000."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


# (groups, pairs, k_max, B): the smallest; 4,096 pairs and one more; 16, 17, 2,048 and 2,049 groups;
# more sums than a small batch may have; 12,800 pairs, which wait for no sizes; chunks of 1,024 pairs, whole and ragged
@pytest.mark.parametrize("ng,count,k_max,B", [(1, 1, 1, 1), (3, 40, 4, 7), (9, 4096, 2, 20), (9, 4097, 2, 20), (16, 13_000, 3, 8), (17, 13_000, 3, 8),
                                              (3, 12_800, 2, 30), (3, 12_801, 2, 30), (2048, 4096, 2, 3), (2049, 4096, 2, 3), (200, 10_241, 8, 2),
                                              (2, 4096, 8, 130), (70, 4096, 8, 130), (5000, 9000, 1, 2)])
def test_groups_match_oracle(fp, ng, count, k_max, B):
    rng = np.random.default_rng(ng + count)
    grp = rng.integers(-1, ng + 1, count).astype(np.int32)     # ids outside the groups are ignored
    z = (rng.normal(size=count) + 1j * rng.normal(size=count)) * np.sqrt(0.5)
    ens = fp.Ensemble(fp.LOCAL, 8, 1, 1, 1, ng, 1, seed=1)
    t = np.ascontiguousarray(np.stack([z.real, z.imag], axis=1).reshape(-1))
    got = ens.bootstrap(t, grp, count, k_max, B, seed=9)
    keep = grp < ng
    ref = O.bootstrap(z[keep], grp[keep], ng, k_max, B, seed=9)
    assert np.allclose(got, ref, rtol=1e-12, atol=0, equal_nan=True)
    assert np.array_equal(ens.bootstrap(t, grp, count, k_max, B, seed=9), got, equal_nan=True)
