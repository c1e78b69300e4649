"""Passes of models that run kernel by kernel: more weights a layer than the one-launch pass takes, and widths or a type that the
streaming pass does not.  Rows and contexts around the borders of an attention split, every result against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synthetic_inputs as si

pytestmark = pytest.mark.gpu

SHAPES = {"fp32": si.ModelShape("op-fp32", 1, 1536, 12, 4, 128, 4096, 997, "fp32", 1e-5, 10000.0),          # 101 MB a layer
          "bf16": si.ModelShape("op-bf16", 1, 1536, 24, 24, 64, 4104, 1000, "bf16", 1e-5, 10000.0)}         # 57 MB
TOL = {"fp32": 1e-4, "bf16": 2e-2}


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_kernel_by_kernel_passes_match_the_oracle(dtype):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = SHAPES[dtype]
    w = si.make_model_weights(shape, 4, gain_spread=0.1)
    om = oracle.OracleModel(shape, w, 340)
    sess = kb.Session.from_shape(shape, {k: ([t.cuda() for t in v] if isinstance(v, list) else v.cuda()) for k, v in w.items()}, 340, max_draft=15)
    prompt = si.uniform_tokens(4, 0, 290, shape.vocab).numpy()
    want_pooled, want_first, _ = om.prefill(prompt)
    before = sess.launch_count
    first, pooled = sess.prefill(prompt, want_pooled=True)
    assert sess.launch_count - before > 9 * ((len(prompt) + 15) // 16)                   # nine kernels a layer of each chunk of 16 rows
    mask = np.zeros(2, np.uint8)
    for n, k in ((290, 4), (256, 0), (255, 9), (241, 15), (100, 7), (1, 2)):
        rows = si.uniform_tokens(4, 100 + n, k + 1, shape.vocab).numpy()
        want = om.forward(rows, n, want_hidden=True)
        sess.set_length(n)
        sess.set_pending(int(rows[0]))
        got = sess.verify(rows[1:], want_logits=True, want_hidden=True)
        assert np.abs(got["logits"].cpu().numpy() - want["logits"]).max() < TOL[dtype], (n, k)
        assert np.abs(got["hidden"].cpu().numpy() - want["hidden"]).max() < TOL[dtype], (n, k)
        for mask in (np.array([1, 0], np.uint8), np.array([0, 1], np.uint8)):            # one row with a sublayer left out
            sess.set_length(n)
            sess.set_skipmask(mask)
            sess.set_pending(int(rows[0]))
            logits = sess.draft(1, want_logits=True)[1]
            assert np.abs(logits.cpu().numpy() - om.forward(rows[:1], n, skip_mask=mask)["logits"]).max() < TOL[dtype], (n, mask)
            om.forward(rows, n)
