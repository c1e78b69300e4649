"""Results that a kernel may not store straight to the caller's buffer (managed memory, which another device or the host may hold at the
time) are copied there: the same bits as in device memory."""
import ctypes as C

import numpy as np
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu


class Managed:
    """`shape` values of managed memory."""

    def __init__(self, shape, dtype=np.float32):
        self.rt = C.CDLL("libcudart.so.12")                       # the one torch has loaded
        self.p = C.c_void_p()
        n = int(np.prod(shape)) * np.dtype(dtype).itemsize
        assert self.rt.cudaMallocManaged(C.byref(self.p), C.c_size_t(n), C.c_uint(1)) == 0
        self.array = np.frombuffer((C.c_char * n).from_address(self.p.value), dtype=dtype).reshape(shape)
        self.array[:] = -7

    def close(self):
        torch.cuda.synchronize()
        self.rt.cudaFree(self.p)


@pytest.mark.parametrize("name", ["tiny", "stream-bf16"])
def test_session_results_in_managed_memory(name):
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    shape = si.SHAPES[name]
    w = si.make_model_weights(shape, 5, device="cuda", gain_spread=0.1)
    prompt = np.ascontiguousarray(si.uniform_tokens(5, 0, 40, shape.vocab).numpy(), dtype=np.int32)
    rows = si.uniform_tokens(5, 1, 4, shape.vocab).numpy()
    sess = kb.Session.from_shape(shape, w, 96, max_draft=4)
    sess.set_skipmask(si.skip_mask(5, 2 * shape.n_layers, 2))
    bufs = [Managed(shape.d_model), Managed((2, shape.vocab)), Managed((4, shape.vocab)), Managed((4, shape.d_model))]
    first, a, nx, drafted = C.c_int(), C.c_int(), C.c_int(), np.zeros(2, np.int32)
    want_first, want_pooled = sess.prefill(prompt, want_pooled=True)
    want_drafted, want_draft = sess.draft(2, want_logits=True)
    sess.set_pending(int(rows[0]))
    want = sess.verify(rows[1:], want_logits=True, want_hidden=True)
    sess._check(kb._lib.knnssd_prefill(sess.h, prompt.ctypes.data, len(prompt), bufs[0].p, C.byref(first)))
    sess._check(kb._lib.knnssd_draft(sess.h, 2, drafted.ctypes.data, bufs[1].p))
    sess.set_pending(int(rows[0]))
    drafts = np.ascontiguousarray(rows[1:], dtype=np.int32)
    sess._check(kb._lib.knnssd_verify(sess.h, drafts.ctypes.data, 3, C.byref(a), C.byref(nx), bufs[2].p, bufs[3].p))
    assert first.value == want_first and np.array_equal(drafted, want_drafted) and (a.value, nx.value) == (want["n_accepted"], want["next_token"])
    for buf, t in zip(bufs, (want_pooled, want_draft, want["logits"], want["hidden"])):
        assert np.array_equal(buf.array, t.cpu().numpy())
        buf.close()


def test_centroids_in_managed_memory():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding as kb
    x = torch.randn(900, 36, generator=torch.Generator().manual_seed(1)).cuda()
    start = x[:3].contiguous()
    for limit in (3, 40):
        want = kb.knnssd_build_anchors(x, start, limit, 4)
        mu, labels, anchors = Managed((3, 36), np.float64), np.zeros(900, np.int32), np.zeros((3, 4), np.int32)
        rounds, ms = C.c_int(), C.c_float()
        assert kb._lib.knnssd_build_anchors(x.data_ptr(), 900, 36, 3, start.data_ptr(), limit, 4, labels.ctypes.data, mu.p, anchors.ctypes.data, C.byref(rounds),
                                            C.byref(ms), torch.cuda.current_stream().cuda_stream) == 0
        assert rounds.value == want["rounds"] and np.array_equal(labels, want["labels"]) and np.array_equal(anchors, want["anchors"])
        assert np.array_equal(mu.array, want["centroids"].cpu().numpy())
        mu.close()
