"""Device times of a session's calls: stamped by the first and the last kernel of a call, whichever kernels run its passes."""
import numpy as np
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu

SHAPES = [si.SHAPES["stream-bf16"], si.SHAPES["tiny"], si.ModelShape("op-fp32", 1, 1536, 12, 4, 128, 4096, 997, "fp32", 1e-5, 10000.0)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: s.name)
def test_calls_report_their_device_time(shape):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    w = si.make_model_weights(shape, 3, device="cuda")
    anchors = torch.nn.functional.normalize(torch.randn(6, shape.d_model, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1)), dim=1)
    mask = np.zeros((2, 2 * shape.n_layers), np.uint8)
    mask[:, 1] = 1
    s = kb.Session.from_shape(shape, w, 96, max_draft=15, anchors=anchors, skip_masks=mask, anchors_per_domain=3)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    drafts = si.uniform_tokens(3, 1, 4, shape.vocab).numpy()
    calls = [("ms_prefill", lambda: s.prefill(si.uniform_tokens(3, 0, 40, shape.vocab).numpy())), ("ms_select", s.select_skipset),
             ("ms_draft", lambda: s.draft(3, want_logits=True)), ("ms_verify", lambda: s.verify(drafts, want_logits=True)), ("ms_verify", lambda: s.verify(drafts[:0]))]
    for name, call in calls:
        call()
        before = s.get_stats()[name] if name in ("ms_draft", "ms_verify") else 0.0       # these add up since the prompt
        torch.cuda.synchronize()
        e[0].record()
        call()
        e[1].record()
        torch.cuda.synchronize()
        took = s.get_stats()[name] - before
        assert 0.0 < took < e[0].elapsed_time(e[1]), name


def test_the_time_of_a_call_has_the_hand_over_in_it():
    """16 rows of 10^6 logits to the caller's buffer: 128 MB read and written, 16 us at 8 TB/s, which is more than
    the memory gives.  Half of that, for what L2 still holds; the call without logits runs the same pass."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.ModelShape("wide-head", 1, 128, 2, 2, 64, 256, 1000000, "bf16", 1e-5, 10000.0)
    w = si.make_model_weights(shape, 3, device="cuda")
    s = kb.Session.from_shape(shape, w, 64, max_draft=15)
    drafts = si.uniform_tokens(3, 1, 15, shape.vocab).numpy()
    s.prefill(si.uniform_tokens(3, 0, 20, shape.vocab).numpy())

    spoiled = torch.empty(16, shape.vocab, device="cuda")

    def took(want_logits):
        before = s.get_stats()["ms_verify"]
        s.set_length(20)
        spoiled.fill_(0.0)                                           # L2 holds the same kind of lines before either call
        torch.cuda.synchronize()
        s.verify(drafts, want_logits=want_logits)
        return s.get_stats()["ms_verify"] - before

    times = {want: [took(want) for _ in range(24)][4:] for want in (True, False)}
    assert np.median(times[True]) - np.median(times[False]) > 0.008
