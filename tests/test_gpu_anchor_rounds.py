"""Anchor construction at the edges of its kernels: widths around a step of 256 columns (16-byte rows and not), rounds past a
batch of four and a limit inside one, lists of points longer than the selection keeps in shared memory."""
import numpy as np
import pytest
import torch

import oracle.anchors as oa

pytestmark = pytest.mark.gpu


def _run(n_points, d, n, k, max_rounds, seed, spread):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    rng = np.random.default_rng(seed)
    X = rng.normal(size=(n, d)).repeat(-(-n_points // n), axis=0)[:n_points] + spread * rng.normal(size=(n_points, d))
    X = rng.permutation(X).astype(np.float32)
    start = X[:n].copy()
    want = oa.build_anchors(X, start.astype(np.float64), max_rounds, k)
    got = kb.knnssd_build_anchors(torch.from_numpy(X).cuda(), torch.from_numpy(start).cuda(), max_rounds, k)
    assert got["rounds"] == want["rounds"]
    assert np.array_equal(got["labels"], want["labels"]) and np.array_equal(got["anchors"], want["anchors"])
    # fp64 sums of at most n_points terms
    assert np.abs(got["centroids"].cpu().numpy() - want["centroids"]).max() < 1e-10
    return want["rounds"]


@pytest.mark.parametrize("d", [1, 4, 255, 256, 257, 260, 1028])
def test_widths_around_a_step(d):
    _run(203, d, 4, 3, 30, 11, 1.0)


@pytest.mark.parametrize("n", [1, 4, 5, 8, 9, 16])
def test_cluster_counts(n):
    _run(403, 132, n, 4, 30, 12, 0.9)


def test_rounds_past_a_batch_and_limits_inside_one():
    total = _run(1500, 12, 6, 5, 60, 13, 3.0)
    assert total > 5                                              # more than one batch
    for limit in (1, 3, 4, 5, total - 1, total, total + 1):
        _run(1500, 12, 6, 5, limit, 13, 3.0)


def test_more_points_than_the_selection_stages():
    _run(25600, 8, 3, 4, 6, 14, 0.4)
    _run(25601, 8, 3, 4, 6, 14, 0.4)


def test_more_results_than_are_kept_pinned():
    """Labels and anchors of 262200 points are more words than a thread keeps pinned: they come by copies, done in one batch or several."""
    for limit in (2, 6):
        _run(262200, 4, 3, 4, limit, 15, 1.5)


@pytest.mark.parametrize("n_points,d,n", [(1301, 39999, 7), (900, 16388, 16), (1301, 39999, 1)])
def test_sums_of_slices_that_are_sorted_by_cluster(n_points, d, n):
    """More blocks of sums than are resident: longer slices, taken cluster by cluster - past 256 points, with clusters that have no point
    in a slice, and all points in one."""
    _run(n_points, d, n, 3, 4, 11 + n, 3.0)


@pytest.mark.parametrize("n_points,d,n", [(1301, 3585, 3), (700, 130, 16), (1301, 20001, 3), (600, 60000, 1), (203, 230000, 4)])
def test_order_of_the_sums(n_points, d, n):
    """A centroid is the sum of its members by slices - the number of them a matter of n_points and d alone - in index order, the slices' sums
    added in their order, over the count: to the last bit.  Both forms of the sums, the smallest and the largest slices."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    rng = np.random.default_rng(d)
    X = rng.normal(size=(n_points, d)).astype(np.float32)
    got = kb.knnssd_build_anchors(torch.from_numpy(X).cuda(), torch.from_numpy(X[:n]).cuda(), 1, 1)
    slices = min(64, -(-n_points // 64), max(1, 6 * 148 // -(-d // 256)))
    per = -(-n_points // slices)
    want = np.zeros((n, d))
    for p0 in range(0, n_points, per):
        part = np.zeros((n, d))
        for p in range(p0, min(n_points, p0 + per)):
            part[got["labels"][p]] += X[p]
        want += part
    want /= np.bincount(got["labels"], minlength=n)[:, None]
    assert np.array_equal(got["centroids"].cpu().numpy(), want)
