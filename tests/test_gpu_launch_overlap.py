"""Linears launched while the one before still runs: each reads what that one wrote, so
a chain without a synchronisation in between, from the host and as a captured graph,
has to give the bits of the chain that synchronises after every call."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(1, 2048), (8, 4096), (24, 4096), (100, 2048), (300, 2048)])
def test_chain_without_synchronisation(M, N):
    from paper_2608_30877_gb300 import w4a16 as W
    gen = torch.Generator(device="cuda").manual_seed(M)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    # weights of unit gain; a residual of its input in every layer keeps the chain from dying
    layers = [W.quantize(rnd(N, N) / N ** 0.5, 128) for _ in range(2)]
    x = rnd(M, N).bfloat16()
    bufs = [torch.empty_like(x) for _ in range(2)]

    def chain(sync):
        bufs[1].copy_(x)
        for i in range(12):
            W.linear_fused(bufs[1 - i % 2], *layers[i % 2], 128, residual=x, out=bufs[i % 2])
            if sync:
                torch.cuda.synchronize()
        return bufs[1].clone()

    ref = chain(True)
    for _ in range(5):
        assert torch.equal(chain(False), ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = chain(False)
    for _ in range(3):
        captured.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(captured, ref)
