"""Merge Peaks on lists that run out: fewer candidates than peaks asked for,
an exclusion that leaves one, equal values, and every count in between."""
import numpy as np
import pytest

from paper_2408_02398_gb300 import ttm


@pytest.mark.parametrize("n,P,dist,levels", [(1, 1, 0.0, 1), (1, 9, 3.0, 1), (7, 7, 0.0, 2), (500, 500, 0.0, 1),
                                             (500, 499, 0.0, 40), (500, 2000, 0.0, 3), (500, 2000, 6.0, 40),
                                             (500, 2000, 1e4, 3), (500, 0, 1.0, 3), (33, 12, 2.5, 5)])
def test_merge_peaks_until_the_list_ends(n, P, dist, levels):
    rng = np.random.default_rng(n + P)
    shape = (9, 14, 17)
    idx = rng.choice(int(np.prod(shape)), n, replace=False).astype(np.int64)
    val = rng.integers(-levels, levels + 1, n).astype(np.float32)
    val[rng.random(n) < 0.05] = -np.inf
    got_i, got_v = ttm.ttm_merge_peaks(idx, val, shape, P, dist)
    zyx = np.stack(np.unravel_index(idx, shape), axis=1).astype(float)
    acc = []
    for k in sorted(range(n), key=lambda k: (-float(val[k]), int(idx[k]))):
        if len(acc) < P and all(np.sum((zyx[k] - zyx[a]) ** 2) >= dist ** 2 for a in acc):
            acc.append(k)
    assert list(got_i) == [int(idx[k]) for k in acc]
    assert np.array_equal(got_v, val[acc])
