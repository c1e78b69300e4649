"""Cosine top-1 over more anchors than blocks are resident, rows that one warp holds and rows that it does not: the best anchor and its
cosine against 64 bits, and an anchor's cosine the same bits in a small set and in a large one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 1183, 1184, 1185, 5000, 30011])
@pytest.mark.parametrize("d", [1, 3, 31, 33, 64, 128, 132, 640])
def test_the_best_of_many(n, d):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    g = torch.Generator().manual_seed(n * 1000 + d)
    a = torch.randn(n, d, generator=g).cuda()
    q = torch.randn(d, generator=g).cuda()
    for best in (n - 1, n // 2, 0):                              # the query itself, scaled: one anchor is well ahead of the others
        keep = a[best].clone()
        a[best] = 3.0 * q + (0.01 * q.norm() / d ** 0.5) * torch.randn(d, generator=g).cuda() if d > 3 else 3.0 * q
        got = kb.knnssd_cosine_top1(q, a)
        cos = (a.double() @ q.double()) / a.double().norm(dim=1) / q.double().norm()
        # in one to three dimensions others may be as near: any of those that 32-bit sums of d squares cannot tell apart, 2e-6 of 1
        assert float(cos[got[0]]) > float(cos.max()) - 2e-6
        assert abs(got[1] - float(cos[got[0]])) < 2e-6
        if d > 3:
            assert got[0] == best
            assert kb.knnssd_cosine_top1(q, a[best:best + 1].contiguous())[1] == got[1]
            few = torch.cat([a[best:best + 1], -a[:6]]).contiguous()
            assert kb.knnssd_cosine_top1(q, few) == (0, got[1])
        a[best] = keep
    q0 = torch.zeros(d, device="cuda")
    with pytest.raises(kb.KnnssdError) as e:
        kb.knnssd_cosine_top1(q0, a)
    assert e.value.status == 5
    assert kb.knnssd_cosine_top1(q, a)[0] >= 0                   # the failed call left the counters at zero
