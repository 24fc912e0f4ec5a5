"""Bootstrap of groups whose members differ by many octaves, against the oracle's
draw-by-draw FP64 sums: a resample that misses the largest members has to keep its
own precision, not the group's.

Tolerance: |t|^2 within 2^-52 on either side gives its k-th power within 2 k 2^-52, and
a sum of at most 300 positive terms is within 300 2^-53 of its value: below 5e-14."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
RTOL = 5e-14


def both(fp, groups, k_max, B, seed=7):
    grp = np.repeat(np.arange(len(groups), dtype=np.int32), [len(z) for z in groups])
    z = np.concatenate(groups).astype(np.complex128)
    order = np.random.default_rng(3).permutation(len(z))
    grp, z = np.ascontiguousarray(grp[order]), z[order]
    ens = fp.Ensemble(fp.PARALLEL, 8, 2, 1 + len(groups), seed=1)
    t = np.ascontiguousarray(np.stack([z.real, z.imag], axis=1).reshape(-1))
    got = ens.bootstrap(t, grp, len(grp), k_max, B, seed=seed)
    ens.close()
    return got, O.bootstrap(z, grp, len(groups), k_max, B, seed=seed)


# two members |t|^2 = 1 and 2^r, and groups of 2 to 20 with their magnitudes spread over r octaves
@pytest.mark.parametrize("r", [10, 26, 60])
@pytest.mark.parametrize("k_max", [4, 8])
def test_small_groups_of_different_octaves(fp, r, k_max):
    rng = np.random.default_rng(r + k_max)
    groups = [np.array([1.0, 2.0 ** (r / 2)])]
    for n in (2, 3, 5, 8, 20):
        groups.append(np.exp2(rng.uniform(0, r / 2, n)) * np.exp(2j * np.pi * rng.uniform(size=n)))
    got, ref = both(fp, groups, k_max, 64)
    assert np.all(np.abs(got - ref) <= RTOL * ref), np.max(np.abs(got / ref - 1), axis=2)


# one member far above 40 of order 1; and a shallow brickwork depth: products of 25 gates' |t|^2 ~ Exp(1)
@pytest.mark.parametrize("k_max", [4, 8])
def test_outliers_and_shallow_depths(fp, k_max):
    rng = np.random.default_rng(k_max)
    groups = []
    for big in (1e3, 2e4, 1e6, 3e7, 1e12):
        groups.append(np.sqrt(np.concatenate([rng.exponential(size=40), [big]])))
    for n in (20, 100, 300):
        groups.append(np.sqrt(rng.exponential(size=(n, 25)).prod(axis=1)))
    got, ref = both(fp, groups, k_max, 100)
    assert np.all(np.abs(got - ref) <= RTOL * ref), np.max(np.abs(got / ref - 1), axis=2)
