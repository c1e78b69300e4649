"""The prompt pass's contraction deals its tiles out whole or in pieces, with 128 to 256 columns, by the sizes of the launch.
A row's sum is the same chunk sums added in the same order either way, so its bits must not depend on the rows it is
launched with.  (The values themselves are compared with the oracle in test_gpu_prefill.py.)"""
import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kb():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding
    return binding


def _inputs(n_out, n_in, T):
    W = si.normal_weight(21, 7, n_out, n_in, 0.02, "bf16", device="cuda")
    x = si.normal_f32(21, 8, torch.arange(T * n_in, device="cuda"), 1.0).view(T, n_in).contiguous()
    return W, x


# 27 and 8.6 chunks of columns (a short last one), ragged last column tiles, one chunk only, more tiles than SMs + a few
@pytest.mark.parametrize("n_out,n_in", [(5120, 13824), (1032, 4416), (4936, 5120), (264, 512), (5000, 320)])
def test_rows_are_the_same_bits_however_the_launch_is_dealt_out(kb, n_out, n_in):
    W, x = _inputs(n_out, n_in, 1024)
    y0 = si.normal_f32(21, 10, torch.arange(1024 * n_out, device="cuda"), 1.0).view(1024, n_out)
    full = {0: kb.knnssd_gemm_split(W, x, 0), 1: kb.knnssd_gemm_split(W, x, 1, y=y0.clone()), 2: kb.knnssd_gemm_split(W, x, 2, W1=W)}
    for T in (1, 77, 128, 129, 300, 1000):
        for mode, want in full.items():
            got = kb.knnssd_gemm_split(W, x[1024 - T:].contiguous(), mode, W1=W if mode == 2 else None, y=y0[1024 - T:].clone() if mode == 1 else None)
            assert torch.equal(got, want[1024 - T:]), (T, mode)


@pytest.mark.parametrize("T", [5, 300])
def test_add_to_rows_that_are_16_byte_aligned_only(kb, T):
    """The add epilogue works in 32-byte accesses where the rows allow it, and must not where they do not."""
    W, x = _inputs(520, 640, T)
    y0 = si.normal_f32(21, 9, torch.arange(T * 520, device="cuda"), 1.0).view(T, 520)
    want = kb.knnssd_gemm_split(W, x, 1, y=y0.clone())
    buf = torch.zeros(T * 520 + 8, device="cuda")
    y = buf[4:4 + T * 520].view(T, 520)
    assert y.data_ptr() % 32 == 16
    y.copy_(y0)
    kb.knnssd_gemm_split(W, x, 1, y=y)
    assert torch.equal(y, want) and not buf[:4].any() and not buf[-4:].any()
