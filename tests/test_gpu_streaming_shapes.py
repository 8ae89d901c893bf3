"""The tensor-core streaming kernel's choices by shape, against the oracle:
K whole and split over clusters of 2, 4 and 8 CTAs (narrow layers), every group size
with K ending inside a 128-k stage, token tiles beyond 128 tokens, ragged rows."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2608_30877_gb300 import synthetic as S
from tests.gpu_helpers import assert_close, assert_close_fused, bf16_to_f64, host_case, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,g", [
    (17, 257, 4096, 128), (32, 1001, 2048, 128), (33, 4100, 2048, 128), (64, 12290, 1024, 128),
    (100, 2000, 4096, 128), (128, 12288, 1152, 128),                        # split or not
    (24, 999, 1088, 64), (40, 1000, 64, 64), (128, 513, 960, 192), (20, 640, 4160, 320),
    (1, 300, 576, 64), (16, 10, 2112, 64),                                  # K % 128 = 64
    (96, 1500, 1024, 128), (97, 4200, 640, 128), (112, 49000, 256, 128),    # 96 and 112 columns
    (129, 1000, 1024, 128), (333, 4100, 1088, 64), (500, 300, 2048, 256),   # token tiles
])
def test_streaming_shapes_match_the_oracle(M, N, K, g):
    from paper_2608_30877_gb300 import w4a16 as W
    assert W.route(M, N, K, g)[0] == "stream"
    x, xb, packed, scales = host_case(M, N, K, g, 31 * M + N, K)
    xd, wd, sd = to_device(x, packed, scales)
    out = W.linear(xd, wd, sd, g)
    again = W.linear(xd, wd, sd, g)
    torch.cuda.synchronize()
    ref = O.linear_rows(xb, packed, scales, N, K, g, nthreads=O.max_threads())
    assert_close(bf16_to_f64(out), ref, f"{M}x{K}x{N} g{g}")
    assert torch.equal(out, again)          # the split sums in a fixed order
    assert W.get_device_error() == W.OK


@pytest.mark.parametrize("M,N,K", [(24, 1000, 4096), (100, 4100, 2048), (333, 1002, 2048)])
@pytest.mark.parametrize("act", [0, 1, 2])
def test_split_sums_through_the_fused_epilogue(M, N, K, act):
    from paper_2608_30877_gb300 import w4a16 as W
    x, xb, packed, scales = host_case(M, N, K, 128, M + N, K + act)
    xd, wd, sd = to_device(x, packed, scales)
    n_out = N // 2 if act == W.ACT_SWIGLU else N
    rng = np.random.default_rng(M + act)
    bf16 = lambda a: S.bf16_bits(torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16))
    dev = lambda b: torch.from_numpy(b.view(np.int16)).view(torch.bfloat16).cuda()
    bias, res = bf16(0.5 * rng.normal(size=N)), bf16(0.5 * rng.normal(size=(M, n_out)))
    buf = dev(res)
    W.linear_fused(xd, wd, sd, 128, act=act, bias=dev(bias), residual=buf, out=buf)
    torch.cuda.synchronize()
    y = O.linear_rows(xb, packed, scales, N, K, 128, nthreads=O.max_threads())
    ref = O.epilogue_rows(y, act, bias=bias, residual=res)
    assert_close_fused(bf16_to_f64(buf), y, ref, act, bias, f"{M}x{K}x{N} act{act}")
    assert W.get_device_error() == W.OK


# (split, M, N, K, g): stages that the ranks share unevenly, a last slice of tokens that is
# not whole, odd rows, token tiles
SPLITS = [(1, 24, 40001, 640, 128), (2, 23, 20001, 8320, 128), (2, 97, 20001, 8320, 128),
          (4, 24, 8191, 4224, 128), (4, 101, 8192, 4160, 64), (4, 65, 7002, 4096, 256),
          (8, 17, 2001, 4992, 128), (8, 128, 3000, 5056, 64), (2, 200, 10002, 8320, 128)]


@pytest.mark.parametrize("split,M,N,K,g", SPLITS)
@pytest.mark.parametrize("act", [0, 1, 2])
def test_every_split_plain_and_fused(split, M, N, K, g, act):
    from paper_2608_30877_gb300 import w4a16 as W
    if act == W.ACT_SWIGLU and N % 2:
        N += 1
    assert W.route(M, N, K, g)[::2] == ("stream", split)
    assert W.route(M, N, K, g, act, True)[::2] == ("stream", split)
    x, xb, packed, scales = host_case(M, N, K, g, M + N, K + act)
    xd, wd, sd = to_device(x, packed, scales)
    y = O.linear_rows(xb, packed, scales, N, K, g, nthreads=O.max_threads())
    if act == 0:
        assert_close(bf16_to_f64(W.linear(xd, wd, sd, g)), y, f"split {split} {M}x{K}x{N} g{g}")
    n_out = N // 2 if act == W.ACT_SWIGLU else N
    rng = np.random.default_rng(M + act)
    bf16 = lambda a: S.bf16_bits(torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16))
    dev = lambda b: torch.from_numpy(b.view(np.int16)).view(torch.bfloat16).cuda()
    bias, res = bf16(0.5 * rng.normal(size=N)), bf16(0.5 * rng.normal(size=(M, n_out)))
    buf = dev(res)
    W.linear_fused(xd, wd, sd, g, act=act, bias=dev(bias), residual=buf, out=buf)
    ref = O.epilogue_rows(y, act, bias=bias, residual=res)
    assert_close_fused(bf16_to_f64(buf), y, ref, act, bias, f"split {split} {M}x{K}x{N} act{act}")
    assert W.get_device_error() == W.OK
