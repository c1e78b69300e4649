"""Session calls while the session's stream is being captured: refused before anything has moved, the capture goes on, and the next call
equals one from a session that never saw a capture."""
import gc

import numpy as np
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "stream-bf16"])
def test_calls_are_refused_while_the_stream_is_captured(name):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.SHAPES[name]
    w = si.make_model_weights(shape, 3, device="cuda", gain_spread=0.1)
    mask = si.skip_mask(3, 2 * shape.n_layers, 2)
    prompt = si.uniform_tokens(3, 0, 30, shape.vocab).numpy()
    rows = si.uniform_tokens(3, 1, 4, shape.vocab).numpy()
    anchors = torch.randn(2, shape.d_model, generator=torch.Generator().manual_seed(0)).cuda()
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    sess = [kb.Session.from_shape(shape, w, 96, max_draft=4, anchors=anchors, skip_masks=np.stack([mask, mask]), anchors_per_domain=1,
                                  stream=stream if captured else torch.cuda.Stream()) for captured in (True, False)]
    for s in sess:
        s.set_skipmask(mask)
        s.prefill(prompt)
    s = sess[0]
    calls = [lambda: s.draft(1), lambda: s.verify(rows[1:]), lambda: s.prefill(prompt), lambda: s.select_skipset(), lambda: s.generate(prompt, 8, 2),
             lambda: s.decode(8, 2), lambda: s.decode_sampled(3, 1, 1.0, 0.9, np.zeros(6, np.float32)), lambda: s.time_pass(0, 0, 1), lambda: s.set_length(10),
             lambda: s.set_pending(1)]
    launches = s.launch_count
    graph, kept = torch.cuda.CUDAGraph(), torch.zeros(4, device="cuda")
    gc.collect()
    gc.disable()                                                     # a session of another test that goes away now would end the capture
    try:
        with torch.cuda.graph(graph, stream=stream):
            kept.add_(1)
            for call in calls:                                       # an odd number of passes each, for the first two
                with pytest.raises(kb.KnnssdError) as e:
                    call()
                assert e.value.status == 6
    finally:
        gc.enable()
    graph.replay()
    torch.cuda.synchronize()
    assert kept.tolist() == [1.0] * 4                                # the capture was not spoiled
    assert s.launch_count == launches and s.length == len(prompt)
    for s in sess:
        s.set_pending(int(rows[0]))
    drafted = [s.draft(1, want_logits=True) for s in sess]
    assert torch.equal(drafted[0][1], drafted[1][1]) and np.array_equal(drafted[0][0], drafted[1][0])
    verified = [s.verify(rows[1:], want_logits=True, want_hidden=True) for s in sess]
    assert torch.equal(verified[0]["logits"], verified[1]["logits"]) and torch.equal(verified[0]["hidden"], verified[1]["hidden"])
