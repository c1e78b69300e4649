"""Weights written by the kernel that comes right before the linear map on the stream, with nothing in between: a library kernel that lets
its successor be set up early, in eager launches and in a captured graph, and in-place updates before a session's pass."""
import numpy as np
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu

# rows of the filter = outputs of the map, values a row (each of them two bf16 weights): one slice of ids a block and more, several batches of groups
SIZES = [(148, 1024), (700, 2048), (301, 65536)]


def _library():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    return kb


def _case(rows, vocab, seed):
    """Logits of which 2^j are equal and the others far below, in row r (j = 1 .. 8): probabilities 2^-j, whose low half-words are zero."""
    g = torch.Generator().manual_seed(seed)
    logits = torch.full((rows, vocab), -1e4)
    for r in range(rows):
        logits[r, torch.randperm(vocab, generator=g)[:2 << (r + seed) % 8]] = 1.0
    x = torch.randn(5, 2 * vocab, generator=g)
    return logits.cuda(), x.cuda()


def _pair(kb, logits, probs, x, y):
    s = torch.cuda.current_stream().cuda_stream
    rows, vocab = logits.shape
    assert kb._lib.knnssd_filtered_probs(logits.data_ptr(), rows, vocab, 1.0, 1.5, probs.data_ptr(), s) == 0
    assert kb._lib.knnssd_linear(probs.data_ptr(), 1, rows, 2 * vocab, x.data_ptr(), x.shape[0], y.data_ptr(), s) == 0


def _separate(kb, logits, x):
    """The same with a wait between the two."""
    probs = kb.knnssd_filtered_probs(logits, 1.0, 1.5)
    torch.cuda.synchronize()
    y = kb.knnssd_linear(probs.view(torch.bfloat16), x)
    torch.cuda.synchronize()
    # every product is exact; sums of 256 and fewer terms in another order
    want = x.double() @ torch.where(logits == 1.0, 1.0 / (logits == 1.0).sum(dim=1, keepdim=True), 0.0).double().repeat_interleave(2, dim=1).mul(
        torch.tensor([0.0, 1.0], dtype=torch.float64, device="cuda").repeat(logits.shape[1])).T
    assert (y.double() - want).abs().max() < 1e-5
    return y


@pytest.mark.parametrize("rows,vocab", SIZES)
def test_weights_from_the_kernel_before(rows, vocab):
    kb = _library()
    probs, y = torch.empty(rows, vocab, device="cuda"), torch.empty(5, rows, device="cuda")
    for seed in range(3):
        logits, x = _case(rows, vocab, seed)
        want = _separate(kb, logits, x)
        probs.zero_()
        y.fill_(-7.0)
        torch.cuda.synchronize()
        _pair(kb, logits, probs, x, y)
        assert torch.equal(y, want)


def test_captured_and_replayed():
    kb = _library()
    rows, vocab = SIZES[1]
    logits, x = _case(rows, vocab, 0)
    probs, y = torch.zeros(rows, vocab, device="cuda"), torch.empty(5, rows, device="cuda")
    _separate(kb, logits, x)                                        # before the capture: attributes and device properties are looked up
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        probs.zero_()
        _pair(kb, logits, probs, x, y)
        y.mul_(2.0)
    for seed in range(1, 4):
        for buf, new in zip((logits, x), _case(rows, vocab, seed)):
            buf.copy_(new)
        graph.replay()
        torch.cuda.synchronize()
        got = y.clone()
        assert torch.equal(got, 2.0 * _separate(kb, logits, x))


def test_weights_updated_in_place_before_a_pass():
    """A model whose passes run kernel by kernel, with maps of the streaming kernel (100 MB a layer)."""
    kb = _library()
    shape = si.ModelShape("op-stream", 1, 2048, 16, 16, 128, 5448, 997, "bf16", 1e-5, 10000.0)
    old, new = (si.make_model_weights(shape, seed, device="cuda", gain_spread=0.1) for seed in (3, 4))
    stream = torch.cuda.Stream()
    sess = kb.Session.from_shape(shape, old, 96, max_draft=4, stream=stream)
    rows = si.uniform_tokens(3, 1, 4, shape.vocab).numpy()
    sess.prefill(si.uniform_tokens(3, 0, 30, shape.vocab).numpy())
    before = sess.launch_count

    def verify():
        sess.set_length(30)
        sess.set_pending(int(rows[0]))
        return sess.verify(rows[1:], want_logits=True)["logits"].clone()

    was = verify()
    assert sess.launch_count - before > 9
    weights = [(old[k], new[k]) for k in ("lm_head",)] + [(old[k][0], new[k][0]) for k in ("wq", "wk", "wv", "wo", "w_gate", "w_up", "w_down")]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for a, b in weights:
            a.copy_(b)
    got = verify()
    torch.cuda.synchronize()
    want = verify()
    assert torch.equal(got, want) and not torch.equal(got, was)
    assert np.isfinite(got.cpu().numpy()).all()
