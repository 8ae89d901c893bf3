"""The default output of attention_prefill: zero outside every sequence, attention
inside, and all zero for a bad sequence table."""
import pytest
import torch

from paper_2608_30877_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("starts", [[0, 100, 300, 700], [5, 5, 260, 261, 699], [700, 700], [0, 0],
                                    [130, 131]])
def test_default_output_is_zero_outside(starts):
    from paper_2608_30877_gb300 import w4a16 as W
    H, M = 3, 700
    qkv = S.make_x(M, 3 * H * 128, 5, "cuda")
    st = torch.tensor(starts, dtype=torch.int32, device="cuda")
    want = W.attention_prefill(qkv, st, H, 200, out=torch.zeros((M, H * 128), dtype=torch.bfloat16,
                                                                device="cuda"))
    torch.full((M, H * 128), 7.0, dtype=torch.bfloat16, device="cuda")  # dirty the allocator's block
    got = W.attention_prefill(qkv, st, H, 200)
    assert torch.equal(got, want)
    assert not got[:starts[0]].any() and not got[starts[-1]:].any()
    assert W.get_device_error() == W.OK


def test_bad_table_gives_zeros_and_the_status():
    from paper_2608_30877_gb300 import w4a16 as W
    H, M = 2, 300
    qkv = S.make_x(M, 3 * H * 128, 6, "cuda")
    st = torch.tensor([0, 200, 100, 300], dtype=torch.int32, device="cuda")
    got = W.attention_prefill(qkv, st, H, 64)
    assert W.get_device_error() == W.ERR_INVALID_ARG
    assert not got.any()


@pytest.mark.parametrize("limit_ns", [1, 2000, 20000])
def test_rows_that_a_timed_out_call_did_not_finish_are_zero(limit_ns):
    """The kernel stores a (16 rows, head) piece whole or leaves it, so in every piece
    the output is the attention's or zero, never what the memory held before."""
    from paper_2608_30877_gb300 import w4a16 as W
    H, M = 4, 3000
    qkv = S.make_x(M, 3 * H * 128, 8, "cuda")
    st = torch.tensor([3, 900, 901, 2500, 2990], dtype=torch.int32, device="cuda")
    want = W.attention_prefill(qkv, st, H, 32768)
    dirty = torch.full((M, H * 128), 7.0, dtype=torch.bfloat16, device="cuda")
    at = dirty.data_ptr()
    del dirty
    W.set_wait_limit(limit_ns)
    try:
        got = W.attention_prefill(qkv, st, H, 32768)
        status = W.get_device_error()
    finally:
        W.set_wait_limit(0)
    assert got.data_ptr() == at  # the dirtied memory
    assert status in (W.OK, W.ERR_TIMEOUT)
    if limit_ns == 1:
        assert status == W.ERR_TIMEOUT
    rows = lambda t: t.view(M, H, 128)
    same = (rows(got) == rows(want)).all(-1)
    zero = (rows(got) == 0).all(-1)
    assert (same | zero).all()
    assert status == W.ERR_TIMEOUT or same.all()
    assert torch.equal(W.attention_prefill(qkv, st, H, 32768), want)
    assert W.get_device_error() == W.OK
