"""Linear layers of at most 8 weight rows (the affinity head's kernel) against
the oracle: one and four tokens per CTA, K down to one scale group, every
activation with bias and residual."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2608_30877_gb300 import synthetic as S
from tests.gpu_helpers import assert_close, assert_close_fused, bf16_to_f64, host_case, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,g", [
    (1, 1, 64, 64), (64, 2, 12288, 128), (5, 3, 1024, 256), (130, 8, 512, 128), (9, 7, 192, 192),
    (700, 4, 640, 64), (1501, 1, 2112, 64), (611, 6, 256, 128),  # four tokens per CTA
])
def test_few_rows_match_the_oracle(M, N, K, g):
    from paper_2608_30877_gb300 import w4a16 as W
    x, xb, packed, scales = host_case(M, N, K, g, 7 * M + N, K)
    xd, wd, sd = to_device(x, packed, scales)
    y = O.linear_rows(xb, packed, scales, N, K, g, nthreads=O.max_threads())
    assert_close(bf16_to_f64(W.linear(xd, wd, sd, g)), y, f"{M}x{K}x{N} g{g}")
    rng = np.random.default_rng(M + N)
    bf16 = lambda a: S.bf16_bits(torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16))
    dev = lambda b: torch.from_numpy(b.view(np.int16)).view(torch.bfloat16).cuda()
    for act in (W.ACT_NONE, W.ACT_SWIGLU, W.ACT_GELU):
        if act == W.ACT_SWIGLU and N % 2:
            continue
        n_out = N // 2 if act == W.ACT_SWIGLU else N
        bias, res = bf16(0.5 * rng.normal(size=N)), bf16(0.5 * rng.normal(size=(M, n_out)))
        buf = dev(res)
        W.linear_fused(xd, wd, sd, g, act=act, bias=dev(bias), residual=buf, out=buf)
        ref = O.epilogue_rows(y, act, bias=bias, residual=res)
        assert_close_fused(bf16_to_f64(buf), y, ref, act, bias, f"{M}x{K}x{N} act{act}")
    assert W.get_device_error() == W.OK
