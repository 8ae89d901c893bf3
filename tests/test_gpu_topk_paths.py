"""Top-k beyond what 8 CTAs keep in shared memory (16 CTAs, keys kept or read
again), slices that end inside a 16-byte load, and equal keys across slices."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,ties,bf16", [
    (320000, 1024, False, False), (320001, 7, False, False),   # the last size on 8 CTAs, 16 CTAs
    (640003, 1000, False, False), (700001, 1024, True, False), (700001, 513, False, True),
    (33, 33, True, False), (63, 1, False, True), (5, 5, True, True),
])
def test_topk_sizes_match_the_oracle(n, k, ties, bf16):
    from paper_2608_30877_gb300 import w4a16 as W
    rng = np.random.default_rng(n + k)
    s = (rng.normal(size=n) * 3 - 8).astype(np.float32)
    if ties:  # the k-th falls inside a long run of equal scores, spread over every slice
        s = np.round(s / 4).astype(np.float32)
    t = torch.from_numpy(s)
    if bf16:
        t = t.to(torch.bfloat16)
    want_i, want_v = O.topk_smallest(t.float().numpy(), k)
    idx, val = W.topk_smallest(t.cuda(), k)
    torch.cuda.synchronize()
    assert idx.cpu().numpy().tolist() == want_i.tolist()
    assert val.cpu().numpy().tobytes() == want_v.tobytes()


@pytest.mark.parametrize("n", [2, 3, 1024, 1025, 2048, 2049, 4097, 70000, 4194305])
@pytest.mark.parametrize("kind", ["equal", "two"])
def test_topk_among_equal_scores(n, kind):
    """The k-th falls among equal scores, so the search goes on to the index: sizes around
    the powers of two where its digits change."""
    from paper_2608_30877_gb300 import w4a16 as W
    s = np.full(n, -7.25, dtype=np.float32)
    if kind == "two":
        s[np.random.default_rng(n).random(n) < 0.5] = np.nan
    for k in [777] if n > 1000000 else sorted({1, min(n, 2), min(n, 777), min(n, 1024)}):
        want_i, want_v = O.topk_smallest(s, k)
        idx, val = W.topk_smallest(torch.from_numpy(s).cuda(), k)
        assert idx.cpu().numpy().tolist() == want_i.tolist()
        assert val.cpu().numpy().tobytes() == want_v.tobytes()
