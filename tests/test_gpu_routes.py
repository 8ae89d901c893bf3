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
