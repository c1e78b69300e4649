"""The nucleus filter: values so close together that more of them lie between the bounds than blocks hand to one another, until late or to
the end; rows on either side of the sizes at which a row takes sixteen slices; a row alone and in company."""
import numpy as np
import pytest
import torch

from oracle import sampling as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kb():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding
    return binding


def _compare(kb, l, temperature, top_p):
    got = kb.knnssd_filtered_probs(l.cuda(), temperature, top_p).cpu().numpy().astype(np.float64)
    for r in range(l.shape[0]):
        want = orc.filtered_distribution(l[r].numpy(), temperature, top_p)
        z = l[r].numpy().astype(np.float64) / temperature
        p = np.exp(z - z.max())
        p /= p.sum()
        # A probability carries the roundings of l - max, its product with 1 / temperature, the exponential and the quotient: a few 2^-24 of
        # its own size and as much of its exponent, so tokens that close to the smallest kept one may change places.  Beside those, the
        # masses are 32-bit sums, 2e-6 of their size (as at other sizes): the two sides' kept masses differ by no more than twice
        # that and the token that the nucleus ends on, and so do the other tokens that one side alone keeps.
        x0 = p[want > 0].min()
        near = 2.0 * (1e-6 + 2.0 ** -23 * (z.max() - z[want > 0].min()))
        edge = (got[r] > 0) != (want > 0)
        assert p[edge & (np.abs(p / x0 - 1.0) > near)].sum() < 4e-6 + x0
        assert abs(p[got[r] > 0].sum() - p[want > 0].sum()) < 4e-6 + x0
        assert np.abs(got[r] - want)[~edge].max() < 4e-6


@pytest.mark.parametrize("V", [300, 4097, 40000, 70000])
@pytest.mark.parametrize("ulps", [1, 40, 3000])
def test_values_close_together(kb, V, ulps):
    g = torch.Generator().manual_seed(V + ulps)
    step = torch.randint(0, ulps + 1, (2, V), generator=g).float() * 2.0 ** -23
    l = 1.0 + step                                        # neighbouring floats, many of them equal
    l[:, 0] = 1.5
    _compare(kb, l, 1.0, 0.6)
    _compare(kb, l, 0.7, 0.97)


@pytest.mark.parametrize("V", [65535, 65536, 65537, 8 * 24576, 8 * 24576 + 1])
@pytest.mark.parametrize("rows", [5, 6])
def test_rows_at_the_line_between_eight_and_sixteen_blocks(kb, V, rows):
    l = 1.4 * torch.randn(rows, V, generator=torch.Generator().manual_seed(V + rows))
    _compare(kb, l, 0.5, 0.9)


@pytest.mark.parametrize("V", [65536, 80000, 100003, 152064, 8 * 24576])
@pytest.mark.parametrize("top_p", [0.8, 0.95])
def test_flat_rows_of_sixteen_slices(kb, V, top_p):
    """No block has more values left between the bounds than it may hand over, all of them together have more than are gone through."""
    l = 1.4 * torch.randn(3, V, generator=torch.Generator().manual_seed(V))
    _compare(kb, l, 1.0, top_p)


@pytest.mark.parametrize("V", [32000, 65535, 65536, 100003, 152064, 8 * 24576, 8 * 24576 + 1])
def test_a_row_does_not_depend_on_its_company(kb, V):
    """A row by itself, among five and among nine: the blocks that share it are not the same, its bits are.  Rows with nothing special
    about them, with many equal values at the cut, and with more values between the bounds than blocks hand to one another."""
    g = torch.Generator().manual_seed(V)
    l = 1.4 * torch.randn(9, V, generator=g)
    l[1] = torch.round(4 * l[1]) / 4
    l[2] = 1.0 + torch.randint(0, 41, (V,), generator=g).float() * 2.0 ** -23
    l[3] = 0.0
    l[4, V // 2:] = -float("inf")
    l = l.cuda()
    for temperature, top_p in ((0.2, 0.85), (1.0, 0.95), (0.7, 2.0)):
        nine = kb.knnssd_filtered_probs(l, temperature, top_p)
        five = kb.knnssd_filtered_probs(l[:5].contiguous(), temperature, top_p)
        assert torch.equal(five, nine[:5])
        for r in range(9):
            assert torch.equal(kb.knnssd_filtered_probs(l[r:r + 1].contiguous(), temperature, top_p)[0], nine[r]), r
