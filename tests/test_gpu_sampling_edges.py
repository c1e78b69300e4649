"""Filtering and drawing by clusters of blocks: rows that do not divide by eight, shorter than a cluster or longer than its
shared memory, ties across the blocks' borders, rows without finite values, draws at the ends of the distribution."""
import numpy as np
import pytest
import torch

import oracle.sampling as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kb():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding
    return binding


def _rows(V, rows, seed=5):
    g = torch.Generator().manual_seed(seed)
    return 1.4 * torch.randn(rows, V, generator=g)


@pytest.mark.parametrize("V", [1, 2, 7, 8, 9, 255, 8191, 8200, 152064, 8 * 49152, 8 * 49152 + 3])
@pytest.mark.parametrize("temperature,top_p", [(0.2, 0.85), (1.0, 0.95), (1.0, 2.0)])
def test_filter_matches_oracle(kb, V, temperature, top_p):
    l = _rows(V, 2)
    got = kb.knnssd_filtered_probs(l.cuda(), temperature, top_p).cpu().numpy().astype(np.float64)
    for r in range(2):
        want = orc.filtered_distribution(l[r].numpy(), temperature, top_p)
        # a mass is a 32-bit sum in which a term meets at most V / 8192 + 30 others: 2e-6 of its size is not reached, so
        # the tokens that only one side keeps weigh less than that, and no other probability is off by more
        edge = (got[r] > 0) != (want > 0)
        assert (got[r] + want)[edge].sum() < 4e-6 and np.abs(got[r] - want).max() < 4e-6


@pytest.mark.parametrize("V,kept", [(16, 5), (1000, 333), (4096, 1024), (32000, 25600)])
def test_equal_logits_are_kept_by_lowest_id(kb, V, kept):
    """All tokens tie: the nucleus is the first ids, wherever the blocks' borders lie.  top_p half a token below the cut."""
    p = kb.knnssd_filtered_probs(torch.zeros(1, V, device="cuda"), 1.0, (kept - 0.5) / V)[0]
    assert int((p > 0).sum()) == kept and bool((p[:kept] > 0).all())
    assert torch.allclose(p[:kept], torch.full((kept,), 1.0 / kept, device="cuda"), rtol=1e-5)


@pytest.mark.parametrize("V", [1000, 32000, 65536, 152064, 400000])
def test_a_nucleus_of_everything_leaves_nothing_out(kb, V):
    """top_p = 1: less than that is ranked before every token, however small it is next to the rounding of the sums."""
    l = _rows(V, 3).cuda()
    for temperature in (0.5, 1.0):
        got = kb.knnssd_filtered_probs(l, temperature, 1.0)
        assert bool((got > 0).all()) and torch.equal(got, kb.knnssd_filtered_probs(l, temperature, 2.0))


def test_masked_and_unusable_rows(kb):
    l = _rows(1000, 4)
    l[1, 500:] = -float("inf")
    l[2, ::2] = torch.finfo(torch.float32).min
    l[3] = -float("inf")
    got = kb.knnssd_filtered_probs(l.cuda(), 0.5, 0.9).cpu()
    assert not got[1, 500:].any() and not got[2, ::2].any() and not got[3].any()
    for r in (1, 2):
        want = orc.filtered_distribution(l[r].numpy().astype(np.float64), 0.5, 0.9)
        assert np.abs(got[r].numpy() - want).max() < 2e-6


@pytest.mark.parametrize("V", [1, 5, 8, 33, 1000, 32000, 152064])
def test_draws_at_the_ends(kb, V):
    w = torch.rand(V, generator=torch.Generator().manual_seed(V)).cuda()
    w[0] = 0.25
    if V > 2:
        w[V // 2:V // 2 + 1] = 0.0
    assert kb.knnssd_sample_token(w, 0.0) == 0
    assert kb.knnssd_sample_token(w, 1.0 - 2.0 ** -24) >= V - 1 - V // 1000
    one = torch.zeros(V, device="cuda")
    one[V - 1] = 1e-30
    for u in (0.0, 0.5, 1.0 - 2.0 ** -24):
        assert kb.knnssd_sample_token(one, u) == V - 1
    cdf = w.double().cumsum(0)
    for u in (0.1, 0.37, 0.9):
        x = kb.knnssd_sample_token(w, u)
        t = u * float(cdf[-1])
        # 32-bit partial sums: within a few ulps of the total of the exact crossing
        assert float(cdf[x]) > t * (1 - 2e-6) and (x == 0 or float(cdf[x - 1]) <= t * (1 + 2e-6) + 1e-7)
        assert float(w[x]) > 0


def test_resample_falls_back_to_p_where_q_covers_it(kb):
    """max(p - q, 0) is zero everywhere: the token is drawn from p."""
    p = torch.zeros(2, 4000, device="cuda")
    p[:, 3999] = 1.0
    q = torch.zeros(1, 4000, device="cuda")
    q[0, 3999] = 1.0
    q[0, 7] = 1.0
    assert kb.knnssd_spec_accept(p, q, [7], [0.5], 0.3) == (0, 3999)


def test_a_draw_between_two_roundings_stays_in_its_block():
    """512 ids: a block has 64, its warps four each.  1 + 2^-24 + 2^-24 is 1 when added one by one and 1 + 2^-23 when block 1's
    two ids are added first, so a target of exactly 1 lies past all of the block's running sums and below its end."""
    from paper_2505_16162_b200 import binding as kb
    w = torch.zeros(512)
    w[0], w[64], w[68], w[511] = 1.0, 2.0 ** -24, 2.0 ** -24, 0.5
    total = np.float32(1.5 + 2.0 ** -23)
    us = [u for u in (np.float32(2.0 / 3.0) + np.arange(-8, 9, dtype=np.float32) * np.float32(2.0 ** -24)) if u * total == np.float32(1.0)]
    assert us
    for u in us:
        assert kb.knnssd_sample_token(w.cuda(), float(u)) in (64, 68)


@pytest.mark.parametrize("V", [9, 4100, 70000])
@pytest.mark.parametrize("top,top_p", [(1, 0.3), (1, 0.999), (3, 0.3), (3, 0.6), (3, 0.95), (3, 2.0)])
def test_largest_values_alone_among_equals_and_beside_others(kb, V, top, top_p):
    """The largest value is counted apart from the sums: the cut falls on it, among its equals, and past them."""
    g = torch.Generator().manual_seed(V + top)
    l = torch.randn(2, V, generator=g).clamp_(max=2.0) - 6.0
    at = torch.randperm(V, generator=g)[:top]
    l[:, at] = 7.0
    l[1, 0] = float("nan")
    got = kb.knnssd_filtered_probs(l.cuda(), 1.0, top_p).cpu().numpy().astype(np.float64)
    want = orc.filtered_distribution(l[0].numpy(), 1.0, top_p)
    edge = (got[0] > 0) != (want > 0)
    assert (got[0] + want)[edge].sum() < 4e-6 and np.abs(got[0] - want).max() < 2e-6
    assert not got[1].any()                                            # a NaN in the row: nothing is kept of it


@pytest.mark.parametrize("V", [8 * 16 * 2048, 8 * 16 * 2048 + 1, 600001])
def test_draws_from_runs_of_several_steps(kb, V):
    """A warp's run of more ids than the block walks at once: every draw against the exact cumulative sum."""
    w = torch.rand(V, generator=torch.Generator().manual_seed(3)).cuda()
    cdf = w.double().cumsum(0)
    for u in np.linspace(0.0005, 0.9995, 40).astype(np.float32):
        x = kb.knnssd_sample_token(w, float(u))
        t = float(u) * float(cdf[-1])
        # 32-bit partial sums: a few ulps of the total
        assert float(cdf[x]) > t * (1 - 2e-6) and (x == 0 or float(cdf[x - 1]) <= t * (1 + 2e-6))
