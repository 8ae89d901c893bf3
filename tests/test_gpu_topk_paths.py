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
