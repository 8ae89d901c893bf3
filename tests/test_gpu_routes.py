"""Which kernel the dispatch gives a linear layer, by size, through the test hook that
names it (w4a16_selftest_route)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,g,kernel", [
    (64, 2, 12288, 128, "head"), (8, 30000, 12288, 128, "rows"), (24, 49152, 12288, 128, "stream"),
    (333, 12288, 12288, 128, "stream"), (4096, 36864, 12288, 128, "gemm"),
])
def test_kernel_by_size(M, N, K, g, kernel):
    from paper_2608_30877_gb300 import w4a16 as W
    name, tokens, ctas, rows = W.route(M, N, K, g)
    assert name == kernel
    assert tokens in {"stream": (32, 64, 96, 112, 128), "gemm": (256, 384)}.get(kernel, (0,))
    assert ctas in {"stream": (1, 2, 4, 8), "gemm": (2,)}.get(kernel, (1,))
    assert (rows > 0) == (kernel == "stream")


# layers that a kernel with a higher rate, but more to start or to finish, had taken
@pytest.mark.parametrize("M,N,K,g,act,residual,kernel", [
    (1, 98304, 1024, 128, 1, False, "rows"), (8, 49152, 256, 128, 2, False, "rows"),
    (1, 49152, 1024, 128, 0, False, "rows"), (8, 98304, 12288, 128, 1, False, "stream"),
    (1, 36864, 12288, 128, 1, False, "stream"), (1, 36864, 1024, 128, 1, False, "rows"),
    (8, 30000, 12288, 128, 1, True, "rows"),
    (8, 98304, 12288, 128, 0, False, "stream"), (16, 49152, 1024, 128, 1, False, "stream"),
    (1, 49152, 12288, 128, 0, False, "stream"),
    (129, 36864, 12288, 64, 0, False, "gemm"), (129, 36864, 12288, 128, 0, False, "stream"),
    (65536, 101, 256, 64, 2, True, "gemm"), (65536, 100, 256, 64, 2, True, "stream"),
])
def test_kernel_by_output_stage_waves_and_scales(M, N, K, g, act, residual, kernel):
    from paper_2608_30877_gb300 import w4a16 as W
    assert W.route(M, N, K, g, act, residual)[0] == kernel


# few rows: the sums over a CTA's threads cost more than the products where K is short
@pytest.mark.parametrize("M,N,K,head", [
    (128, 8, 64, True), (1000, 8, 64, True), (16384, 8, 64, False), (65536, 4, 64, False),
    (65536, 3, 256, False), (65536, 2, 64, False), (8000, 5, 512, False), (65536, 2, 12288, True),
    (65536, 8, 12288, False),
])
def test_few_rows_by_tokens_and_length(M, N, K, head):
    from paper_2608_30877_gb300 import w4a16 as W
    assert (W.route(M, N, K, 64)[0] == "head") == head
