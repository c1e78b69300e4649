"""Passes of 13..16 rows on models whose d_model-wide maps give every CTA more than two groups of units run an instance of
their own: a row's numbers must not depend on it (the same check on narrower models is in test_gpu_parity.py)."""
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,heads", [(128, 4), (64, 4)])
def test_rows_of_wide_passes_on_a_wide_model(head_dim, heads):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    d = (32 * n_sms // 128 + 1) * 128                            # the first width past the rule's border
    shape = si.ModelShape("wide", 2, d, heads, heads // 2, head_dim, 384, 1001, "bf16", 1e-5, 10000.0)
    w = si.make_model_weights(shape, 3, device="cuda", gain_spread=0.1)
    sess = kb.Session.from_shape(shape, w, 160, max_draft=15)
    first = sess.prefill(si.uniform_tokens(5, 0, 70, shape.vocab).numpy())
    rows = si.uniform_tokens(6, 1, 15, shape.vocab).numpy()
    got = {}
    for k in (15, 12, 13, 0, 3, 11):
        sess.set_length(70)
        sess.set_pending(first)
        g = sess.verify(rows[:k], want_logits=True, want_hidden=True)
        got[k] = (g["logits"], g["hidden"])
        assert torch.equal(got[k][0], got[15][0][:k + 1]) and torch.equal(got[k][1], got[15][1][:k + 1]), k
