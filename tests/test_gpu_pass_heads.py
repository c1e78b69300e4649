"""Attention of the persistent pass kernel where the q / k / v map leaves its heads: rows before, on and past the border of a 64-position
segment, blocks of eight (query head, row) pairs that are full, begun and spread over several heads of a group."""
import numpy as np
import pytest
import torch

import oracle
import synthetic_inputs as si

pytestmark = pytest.mark.gpu

SHAPES = {"group5-128": si.ModelShape("group5-128", 2, 256, 5, 1, 128, 512, 515, "bf16", 1e-5, 10000.0),
          "single-64": si.ModelShape("single-64", 2, 256, 6, 6, 64, 512, 101, "bf16", 1e-6, 1000000.0)}      # fewer ids than blocks: some have no units
# two layers leave 7e-5 .. 4e-4 on logits of a few tenths: a few K / V entries round to the other neighbour, 2^-8 of themselves
TOL = 2e-3


@pytest.mark.parametrize("name", list(SHAPES))
def test_passes_across_segment_borders_match_the_oracle(name):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = SHAPES[name]
    w = si.make_model_weights(shape, 9, gain_spread=0.1)
    om = oracle.OracleModel(shape, w, 160)
    sess = kb.Session.from_shape(shape, {k: ([t.cuda() for t in v] if isinstance(v, list) else v.cuda()) for k, v in w.items()}, 160, max_draft=15)
    prompt = si.uniform_tokens(9, 0, 130, shape.vocab).numpy()
    om.prefill(prompt)
    sess.prefill(prompt)
    for n, k in ((130, 0), (128, 1), (127, 2), (121, 7), (120, 8), (113, 15), (65, 3), (64, 4), (63, 0), (1, 11)):
        rows = si.uniform_tokens(9, 100 + n, k + 1, shape.vocab).numpy()
        want = om.forward(rows, n, want_hidden=True)
        sess.set_length(n)
        sess.set_pending(int(rows[0]))
        got = sess.verify(rows[1:], want_logits=True, want_hidden=True)
        assert np.abs(got["logits"].cpu().numpy() - want["logits"]).max() < TOL, (n, k)
        assert np.abs(got["hidden"].cpu().numpy() - want["hidden"]).max() < 5 * TOL, (n, k)      # hidden states are of size one
        # one row that leaves its K / V at a border of the cache, and another behind it
        sess.set_length(n)
        sess.set_skipmask(np.array([0, 0, 0, 1], np.uint8))
        sess.set_pending(int(rows[0]))
        logits = sess.draft(1, want_logits=True)[1]
        assert np.abs(logits.cpu().numpy() - om.forward(rows[:1], n, skip_mask=np.array([0, 0, 0, 1], np.uint8))["logits"]).max() < TOL, (n, k)
        om.forward(rows, n)
        sess.set_length(n)
        sess.set_pending(int(rows[0]))
        sess.verify(rows[1:])
