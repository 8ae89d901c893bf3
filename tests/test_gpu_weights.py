"""Quantise and dequantise byte for byte on the per-lane path (g = 64, 128, 256)
and the general one (other g): quotients at and next to rounding ties, scales that
are zero, subnormal or rounded a long way, blocks that end inside a CTA."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,g", [(1, 64, 64), (37, 192, 64), (129, 384, 128), (3, 128, 128),
                                   (65, 512, 256), (1, 256, 256), (7, 384, 192), (5, 640, 320)])
def test_quantise_and_dequantise_bytes(N, K, g):
    from paper_2608_30877_gb300 import w4a16 as W
    rng = np.random.default_rng(N + K + g)
    w = (0.02 * rng.normal(size=(N, K))).astype(np.float32)
    rows = w.reshape(N * K // g, g)
    for i, row in enumerate(rows):
        kind = i % 6
        if kind == 1:    # ties of w / s and their neighbours: s = 2^-6 exactly
            q = rng.integers(-7, 7, size=g) + 0.5
            row[:] = (q * 2.0 ** -6).astype(np.float32)
            row[1::3] = np.nextafter(row[1::3], np.float32(1))
            row[2::3] = np.nextafter(row[2::3], np.float32(-1))
            row[0] = 7 * 2.0 ** -6
        elif kind == 2:  # the same for a scale that is no power of two
            s = O.bf16_bits_to_f32(np.array([O.bf16_rne(0.013)], np.uint16))[0]
            q = (rng.integers(-7, 7, size=g) + 0.5).astype(np.float32)
            row[:] = q * s
            row[::2] = np.nextafter(row[::2], np.float32(0))
            row[0] = np.float32(7) * s
        elif kind == 3:
            row[:] = 0.0
        elif kind == 4:  # the scale is a subnormal with few bits, or rounds to zero
            row[:] = (rng.integers(-9, 10, size=g) * (1e-40 if i % 4 else 1e-42)).astype(np.float32)
        elif kind == 5:
            row[:] *= np.float32(1e30 if i % 4 else 1e-32)
    packed, scales = O.quantize(w, g)
    got_p, got_s = W.quantize(torch.from_numpy(w).cuda(), g)
    torch.cuda.synchronize()
    assert np.array_equal(got_s.cpu().view(torch.int16).numpy().view(np.uint16), scales)
    assert np.array_equal(got_p.cpu().numpy(), packed)
    want = O.dequant(packed, scales, N, K, g)
    got = W.dequant(got_p, got_s, g)
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().view(torch.int16).numpy().view(np.uint16), want)
