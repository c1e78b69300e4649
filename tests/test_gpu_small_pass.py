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


def _session(kb, shape, w, max_seq):
    return kb.Session.from_shape(shape, {k: ([t.cuda() for t in v] if isinstance(v, list) else v.cuda()) for k, v in w.items()}, max_seq, max_draft=15)


def _launches(sess, call):
    before = sess.launch_count
    call()
    return sess.launch_count - before


@pytest.mark.parametrize("name,own_head", [("tiny", False), ("ragged-bf16", False), ("gqa-fp32", False), ("wide-head", True)])
def test_a_pass_is_one_launch(name, own_head):
    """And what hands its results back; a large head takes three launches behind it, the arg-max among them."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    # 61 MB of head
    shape = si.SHAPES[name] if name in si.SHAPES else si.ModelShape(name, 2, 512, 8, 2, 64, 512, 30011, "fp32", 1e-5, 10000.0)
    w = si.make_model_weights(shape, 6, gain_spread=0.1)
    sess = _session(kb, shape, w, 64)
    prompt = si.uniform_tokens(6, 0, 20, shape.vocab).numpy()
    sess.prefill(prompt)
    sess.set_skipmask(si.skip_mask(6, 2 * shape.n_layers, 2))
    each = 4 if own_head else 1
    assert _launches(sess, lambda: sess.draft(1)) == each + 1
    assert _launches(sess, lambda: sess.draft(3)) == 3 * each + 1
    rows = si.uniform_tokens(6, 1, 5, shape.vocab).numpy()
    om = oracle.OracleModel(shape, w, 64)
    om.prefill(prompt)
    want = om.forward(rows, len(prompt), want_hidden=True)
    sess.set_pending(int(rows[0]))
    got = {}
    assert _launches(sess, lambda: got.update(sess.verify(rows[1:], want_logits=True, want_hidden=True))) == each + 1
    assert np.abs(got["logits"].cpu().numpy() - want["logits"]).max() < TOL[shape.dtype]
    assert np.abs(got["hidden"].cpu().numpy() - want["hidden"]).max() < TOL[shape.dtype]
    timed = sess.time_pass(1, 4, 2)
    assert timed["launches"] == each
    assert timed["linear_launches"] == 4 * shape.n_layers + 1 and timed["ms_linear"] > 0        # replayed kernel by kernel


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_attention_launches_of_its_own_leave_the_same(dtype):
    """Ten splits of context for 16 rows of 16 heads are more attention tasks than the one launch takes, for one row they are not: the
    first row of either has the same bits, and all agree with the oracle."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.ModelShape("long", 2, 264, 16, 4, 64, 264, 515, dtype, 1e-5, 10000.0)
    w = si.make_model_weights(shape, 8, gain_spread=0.1)
    om = oracle.OracleModel(shape, w, 2600)
    sess = _session(kb, shape, w, 2600)
    prompt = si.uniform_tokens(8, 0, 2500, shape.vocab).numpy()
    want_pooled = om.prefill(prompt)[0]
    first, pooled = sess.prefill(prompt, want_pooled=True)
    assert np.abs(pooled.cpu().numpy() - want_pooled).max() < TOL[dtype]
    for n in (2500, 2304, 2303, 300):
        rows = si.uniform_tokens(8, 100 + n, 16, shape.vocab).numpy()
        want = om.forward(rows, n, want_hidden=True)
        one = {}
        for k in (15, 0):
            sess.set_length(n)
            sess.set_pending(int(rows[0]))
            got = {}
            n_launches = _launches(sess, lambda: got.update(sess.verify(rows[1:k + 1], want_logits=True, want_hidden=True)))
            assert n_launches == (2 + 2 * shape.n_layers if k and n > 300 else 2), (n, k)
            assert np.abs(got["logits"].cpu().numpy() - want["logits"][:k + 1]).max() < TOL[dtype], (n, k)
            assert np.abs(got["hidden"].cpu().numpy() - want["hidden"][:k + 1]).max() < TOL[dtype], (n, k)
            one[k] = got
        assert torch.equal(one[15]["logits"][:1], one[0]["logits"]) and torch.equal(one[15]["hidden"][:1], one[0]["hidden"])


def test_sublayers_left_out_of_a_pass_in_parts():
    """120 heads: a draft step of one row at 1100 positions comes in parts too, whichever of its sublayers are left out."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.ModelShape("heads", 3, 136, 120, 4, 64, 136, 301, "fp32", 1e-5, 10000.0)
    w = si.make_model_weights(shape, 9, gain_spread=0.1)
    om = oracle.OracleModel(shape, w, 1160)
    sess = _session(kb, shape, w, 1160)
    prompt = si.uniform_tokens(9, 0, 1100, shape.vocab).numpy()
    om.prefill(prompt)
    sess.prefill(prompt)
    rows = si.uniform_tokens(9, 1, 2, shape.vocab).numpy()
    for mask in ([0, 0, 0, 0, 0, 0], [1, 0, 0, 1, 0, 0], [0, 1, 1, 0, 1, 0], [1, 1, 1, 1, 1, 1], [0, 0, 0, 0, 1, 1]):
        mask = np.array(mask, np.uint8)
        sess.set_skipmask(mask)
        sess.set_pending(int(rows[0]))
        got = []
        n_launches = _launches(sess, lambda: got.append(sess.draft(1, want_logits=True)[1]))
        assert n_launches == 2 + 2 * int((mask[::2] == 0).sum())
        assert np.abs(got[0].cpu().numpy() - om.forward(rows[:1], len(prompt), skip_mask=mask)["logits"]).max() < TOL["fp32"], mask


@pytest.mark.parametrize("shape", [si.ModelShape("wide-bf16", 2, 2056, 8, 2, 64, 1032, 515, "bf16", 1e-5, 10000.0),
                                   si.ModelShape("wide-fp32", 2, 1032, 4, 4, 64, 2056, 515, "fp32", 1e-5, 10000.0)], ids=lambda s: s.name)
def test_widths_that_shared_memory_does_not_hold(shape):
    """Weight rows, gains and (from some row count on) the rows of a map one step longer than what a block keeps of them."""
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    w = si.make_model_weights(shape, 6, gain_spread=0.1)
    om = oracle.OracleModel(shape, w, 64)
    sess = kb.Session.from_shape(shape, {k: ([t.cuda() for t in v] if isinstance(v, list) else v.cuda()) for k, v in w.items()}, 64, max_draft=15)
    prompt = si.uniform_tokens(6, 0, 30, shape.vocab).numpy()
    om.prefill(prompt)
    sess.prefill(prompt)
    for mask in ([0, 1, 0, 0], [1, 0, 0, 1], [0, 0, 1, 1], [1, 1, 1, 1]):
        sess.set_length(30)
        sess.set_skipmask(np.array(mask, np.uint8))
        sess.set_pending(int(prompt[3]))
        logits = sess.draft(1, want_logits=True)[1]
        want = om.forward(prompt[3:4], 30, skip_mask=np.array(mask, np.uint8))["logits"]
        assert np.abs(logits.cpu().numpy() - want).max() < TOL[shape.dtype], mask
    for k in (0, 4, 10, 11, 12, 15):
        rows = si.uniform_tokens(6, 100 + k, k + 1, shape.vocab).numpy()
        want = om.forward(rows, 30, want_hidden=True)
        sess.set_length(30)
        sess.set_pending(int(rows[0]))
        got = sess.verify(rows[1:], want_logits=True, want_hidden=True)
        assert np.abs(got["logits"].cpu().numpy() - want["logits"]).max() < TOL[shape.dtype], k
        assert np.abs(got["hidden"].cpu().numpy() - want["hidden"]).max() < TOL[shape.dtype], k
