"""The output stage that the GEMM and the tensor-core streaming kernel share, where
its pairing of columns and tokens can go wrong: odd and even widths, odd token counts,
slices that end past the last token, the residual in place."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,split,M,N,K", [
    ("stream", 8, 23, 513, 4096), ("stream", 8, 101, 514, 4096), ("stream", 8, 33, 1001, 4224),
    ("stream", 1, 23, 513, 1024), ("stream", 1, 101, 514, 1024),
    ("stream", 1, 40, 40001, 256), ("stream", 1, 127, 40002, 256),   # whole K per CTA
    ("gemm", 2, 2047, 8193, 256), ("gemm", 2, 2049, 8194, 256),
])
@pytest.mark.parametrize("act", [0, 2])
def test_in_place_residual_at_every_width(kernel, split, M, N, K, act):
    from paper_2608_30877_gb300 import w4a16 as W
    assert W.route(M, N, K, 128, act, True)[::2] == (kernel, split)
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    x = rnd(M, K).bfloat16()
    packed, scales = W.quantize(0.02 * rnd(N, K), 128)
    bias, buf = rnd(N).bfloat16(), rnd(M, N).bfloat16()
    y = x.double() @ W.dequant(packed, scales, 128).double().t()
    z = y + bias.double()
    ref = (torch.nn.functional.gelu(z) if act == W.ACT_GELU else z) + buf.double()
    W.linear_fused(x, packed, scales, 128, act=act, bias=bias, residual=buf, out=buf)
    # one bf16 rounding of the output, and the sums' own error: 2e-2 of rms(y) bounds
    # every kernel's plain output, times the activation's slope (at most 1.13)
    bound = 2.0 ** -8 * ref.abs() + 2e-2 * 1.13 * y.square().mean().sqrt()
    assert ((buf.double() - ref).abs() <= bound).all()
