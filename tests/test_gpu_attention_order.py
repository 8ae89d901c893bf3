"""The two orders of attention's jobs: a sequence that is most of a batch has its heads
fastest, others go head by head.  A job computes the same either way, so a sequence
gives the same bits alone and as one of several."""
import pytest
import torch

from paper_2608_30877_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length,H,window", [(1, 3, 100), (129, 1, 32768), (700, 5, 32768),
                                             (2049, 16, 300), (5000, 2, 32768)])
def test_sequence_alone_and_among_others(length, H, window):
    from paper_2608_30877_gb300 import w4a16 as W
    qkv = S.make_x(3 * length + 40, 3 * H * 128, length + H, "cuda")
    table = lambda *s: torch.tensor(s, dtype=torch.int32, device="cuda")
    three = W.attention_prefill(qkv, table(0, length, 2 * length, 3 * length), H, window)
    for i in range(3):
        a = i * length
        alone = W.attention_prefill(qkv[a:a + length].contiguous(), table(0, length), H, window)
        assert torch.equal(alone, three[a:a + length])
    # most of a batch that has empty and short sequences next to it
    mixed = W.attention_prefill(qkv[:length + 3].contiguous(), table(0, 0, length, length + 2, length + 2),
                                H, window)
    assert torch.equal(mixed[:length], three[:length]) and not mixed[length + 2:].any()
    assert W.get_device_error() == W.OK
