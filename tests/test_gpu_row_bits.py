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


@pytest.mark.parametrize("rows", [20, 77, 300])
def test_a_norm_is_the_same_bits_whichever_kernel_sums_it(rows):
    """A layer whose maps back into the residual stream are zero changes nothing: the layer behind it finds the rows that the embedding left.
    Its norms come from squares that the zero maps' epilogues left, those of the same layer at the bottom of a model from the rows."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    two = si.ModelShape("norms", 2, 1536, 12, 4, 128, 2048, 1003, "bf16", 1e-5, 10000.0)
    one = two.with_layers(1)
    w = si.make_model_weights(two, 9, device="cuda", gain_spread=0.1)
    w["wo"][0].zero_()
    w["w_down"][0].zero_()
    w1 = {k: (v[1:] if isinstance(v, list) else v) for k, v in w.items()}
    prompt = si.uniform_tokens(9, 0, rows, two.vocab).numpy()
    got = []
    for shape, weights in ((two, w), (one, w1)):
        sess = kb.Session.from_shape(shape, weights, 400, max_draft=4)
        got.append(sess.prefill(prompt, want_pooled=True))
    assert got[0][0] == got[1][0] and torch.equal(got[0][1], got[1][1])
