"""The weights the linears multiply by, value for value: one-hot activations
make out[m, n] the dequantised weight wd[n, m] itself (one exact product, every
other term zero), which must equal the oracle's dequantisation for every code
and for scales on both sides of the single-FMA path's range |s| < 2^-2."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from tests.gpu_helpers import GEMM_ENVS, assert_gemm, run_in_child

pytestmark = pytest.mark.gpu

# zero, the range's edge from both sides and signs, subnormals, tiny, large
EDGE_SCALES = [0.0, 0.25, 0.2490234375, -0.25, -0.2490234375, 9.2e-41, -1e-38, 3e-39, 1e-30,
               -7.25e-3, 0.0014982223510742188, 1.5, 250.0, -3e30, 1e37]


STREAM_CASES = [(20, 66, 64, 64), (64, 300, 128, 128), (128, 400, 192, 64), (100, 130, 256, 256),
                (300, 300, 320, 64), (700, 40, 384, 128)]
# every form of the GEMM's scale index: one per stage, two stages per scale, a shift, a division
GEMM_CASES = [(300, 300, 320, 64), (300, 257, 256, 128), (700, 40, 512, 256), (200, 130, 576, 192)]


def check_values(M, N, K, g):
    from paper_2608_30877_gb300 import w4a16 as W
    rng = np.random.default_rng(M + N + K)
    packed = rng.integers(0, 256, size=(N, K // 2), dtype=np.uint8)
    scales_f = rng.uniform(-0.3, 0.3, size=(N, K // g))
    # whole warps of rows inside the range, warps with one row outside it
    scales_f[64:192] *= 0.5
    scales_f[:len(EDGE_SCALES), 0] = EDGE_SCALES
    scales_f[N - 1] = 31.0
    bits = torch.from_numpy(scales_f.astype(np.float32)).to(torch.bfloat16)
    scales = bits.view(torch.int16).numpy().view(np.uint16)
    x = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    n = min(M, K)
    x[torch.arange(n), torch.arange(n)] = 1.0
    out = W.linear(x, torch.from_numpy(packed).cuda(), bits.cuda(), g)
    torch.cuda.synchronize()
    want = O.bf16_bits_to_f32(O.dequant(packed, scales, N, K, g).reshape(-1)).reshape(N, K)
    got = out.float().cpu().numpy()[:n].T
    # equal as numbers: the sign of a zero is not kept through the accumulation
    assert np.array_equal(got, want[:, :n])
    assert W.get_device_error() == W.OK


def check_gemm_values(variant):
    from paper_2608_30877_gb300 import w4a16 as W
    for case in GEMM_CASES:
        assert_gemm(W, variant, *case)
        check_values(*case)


@pytest.mark.parametrize("M,N,K,g", STREAM_CASES)
def test_one_hot_activations_give_the_dequantised_weights(M, N, K, g):
    from paper_2608_30877_gb300 import w4a16 as W
    assert W.route(M, N, K, g)[0] == "stream"
    check_values(M, N, K, g)


@pytest.mark.parametrize("variant", GEMM_ENVS)
def test_one_hot_activations_on_the_gemm(variant):
    run_in_child(GEMM_ENVS[variant][0], "test_gpu_dequant_values", "check_gemm_values", variant)
