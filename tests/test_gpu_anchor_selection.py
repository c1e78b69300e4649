"""Anchors of a cluster: the lists that its warps keep (k up to 32), the search by the whole block (more), clusters that run out of
members, equal distances across warps, and blocks of every width that the assignment takes, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import anchors as oa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,d,k", [(2, 1500, 16, 32), (2, 1500, 16, 33), (3, 40, 8, 32), (1, 1024, 12, 1), (1, 1025, 12, 7), (4, 3000, 36, 10), (2, 2300, 20, 5)])
def test_selection_matches_the_oracle(n, N, d, k):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    rng = np.random.default_rng(n * N + k)
    X = (4.0 * rng.standard_normal((n, d))[rng.integers(0, n, N)] + rng.standard_normal((N, d))).astype(np.float32)
    X[N // 2:N // 2 + 4] = X[3]                       # equal distances in several warps: the lowest index first
    start = X[:n].copy()
    want = oa.build_anchors(X, start.astype(np.float64), 50, k)
    got = kb.knnssd_build_anchors(torch.tensor(X).cuda(), torch.tensor(start).cuda(), 50, k)
    assert np.array_equal(np.asarray(got["labels"]), np.asarray(want["labels"]))
    assert np.array_equal(np.asarray(got["anchors"]), np.asarray(want["anchors"]))
