"""What a session takes on the device follows its model and its length, and holds what its kernels put there."""
import numpy as np
import pytest
import torch

import oracle
import synthetic_inputs as si

pytestmark = pytest.mark.gpu


def test_a_small_session_takes_little_memory():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.SHAPES["stream-bf16"]
    w = si.make_model_weights(shape, 0, device="cuda")
    kb.Session.from_shape(shape, w, 64, max_draft=4).close()     # the kernels are loaded
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sess = [kb.Session.from_shape(shape, w, 64, max_draft=4) for _ in range(4)]
    # weights aside, buffers of 64 rows x at most 1920 values: a few MB with what allocations are rounded up to
    assert free - torch.cuda.mem_get_info()[0] < 4 * (16 << 20)
    for s in sess:
        s.close()


def test_pooled_state_of_a_wide_model_with_few_heads():
    """16 times the q, k and v values of a row are fewer than the model's width here: the slices of the pooled sum are what sizes the
    buffer that both share."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.ModelShape("wide", 1, 6272, 4, 1, 64, 256, 512, "bf16", 1e-5, 10000.0)
    w = si.make_model_weights(shape, 9, gain_spread=0.1)
    sess = kb.Session.from_shape(shape, {k: ([t.cuda() for t in v] if isinstance(v, list) else v.cuda()) for k, v in w.items()}, 128, max_draft=4)
    om = oracle.OracleModel(shape, w, 128)
    for n in (127, 97):
        prompt = si.uniform_tokens(9, n, n, shape.vocab).numpy()
        want, first, _ = om.prefill(prompt)
        got_first, got = sess.prefill(prompt, want_pooled=True)
        # K and V in bf16: as the other prompt passes against the oracle
        assert got_first == first and np.abs(got.cpu().numpy() - want).max() < 2e-3
