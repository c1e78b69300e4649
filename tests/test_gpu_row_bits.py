"""What a prompt leaves in the K/V cache for a position must not depend on how many tokens follow it: the launches of a prompt pass
take other tiles, and do the heads' rotary embedding in other places, from length to length."""
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu


# lengths at which the q / k / v launch of these widths takes 128 or 256 columns, whole tiles or pieces, one row tile or several
@pytest.mark.parametrize("name", ["llama7b", "llama13b", "qwen14b"])
def test_cache_rows_are_the_same_bits_whatever_follows_them(name):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.SHAPES[name].with_layers(2)
    w = si.make_model_weights(shape, 7, device="cuda", gain_spread=0.1)
    sess = kb.Session.from_shape(shape, w, 1100, max_draft=4)
    tokens = si.uniform_tokens(7, 0, 1029, shape.vocab).numpy()
    rows = si.uniform_tokens(7, 1, 4, shape.vocab).numpy()
    common, want = 20, None
    for n in (1029, 20, 77, 128, 129, 256, 300, 640, 1000):
        sess.prefill(tokens[:n])
        sess.set_length(common)
        sess.set_pending(int(rows[0]))
        got = sess.verify(rows[1:], want_logits=True)["logits"]
        want = got if want is None else want
        assert torch.equal(got, want), n
