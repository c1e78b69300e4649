"""Passes of models whose decoder pass is one cooperative launch (small fp32 and bf16 shapes): rows around the borders of an
attention split (256 positions), every row count that has an instance of its own and its neighbours, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synthetic_inputs as si

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "bf16": 2e-2}


@pytest.mark.parametrize("name", ["tiny", "gqa-fp32", "ragged-bf16"])
def test_rows_around_the_borders_of_a_split_match_the_oracle(name):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.SHAPES[name].with_layers(2)
    w = si.make_model_weights(shape, 4, gain_spread=0.1)
    om = oracle.OracleModel(shape, w, 600)
    sess = kb.Session.from_shape(shape, {k: ([t.cuda() for t in v] if isinstance(v, list) else v.cuda()) for k, v in w.items()}, 600, max_draft=15)
    prompt = si.uniform_tokens(4, 0, 540, shape.vocab).numpy()
    om.prefill(prompt)
    sess.prefill(prompt)
    mask = si.skip_mask(4, 2 * shape.n_layers, 2)
    # from the longest context down: a pass writes the rows it adds
    for n, k in ((540, 4), (512, 0), (511, 3), (506, 15), (300, 8), (257, 1), (256, 5), (255, 9), (254, 2), (245, 10), (17, 4), (1, 15)):
        rows = si.uniform_tokens(4, 100 + n, k + 1, shape.vocab).numpy()
        want = om.forward(rows, n, want_hidden=True)
        sess.set_length(n)
        sess.set_pending(int(rows[0]))
        got = sess.verify(rows[1:], want_logits=True, want_hidden=True)
        assert np.abs(got["logits"].cpu().numpy() - want["logits"]).max() < TOL[shape.dtype], (n, k)
        assert np.abs(got["hidden"].cpu().numpy() - want["hidden"]).max() < TOL[shape.dtype], (n, k)
        # one row with sublayers left out; its K and V are written again by the next pass
        sess.set_length(n)
        sess.set_skipmask(mask)
        sess.set_pending(int(rows[0]))
        logits = sess.draft(1, want_logits=True)[1]
        assert np.abs(logits.cpu().numpy() - om.forward(rows[:1], n, skip_mask=mask)["logits"]).max() < TOL[shape.dtype], n
        om.forward(rows, n)
