"""Gather of rows at widths on both sides of its two copies' lines: rows of no whole 16-byte
units, rows shorter than a CTA's threads, one row and more rows than the CTAs take at
once, bad indices among good ones."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 7, 8, 100, 255, 2040, 2047, 2048, 2056, 4097])
@pytest.mark.parametrize("P", [1, 5, 3001])
def test_rows_of_every_width(D, P):
    from paper_2608_30877_gb300 import w4a16 as W
    gen = torch.Generator(device="cuda").manual_seed(D + P)
    src = torch.randint(-32768, 32767, (77, D), dtype=torch.int16, device="cuda", generator=gen)
    idx = torch.randint(0, 77, (P,), dtype=torch.int32, device="cuda", generator=gen)
    guard = torch.full((P * D + 64,), 3, dtype=torch.int16, device="cuda")
    out = guard[:P * D].view(P, D)
    W.gather_rows(src.view(torch.bfloat16), idx, out=out.view(torch.bfloat16))
    assert torch.equal(out, src[idx.long()]) and (guard[P * D:] == 3).all()
    assert W.get_device_error() == W.OK
    idx[P // 2] = 77
    idx[P - 1] = -1
    W.gather_rows(src.view(torch.bfloat16), idx, out=out.view(torch.bfloat16))
    assert W.get_device_error() == W.ERR_INVALID_ARG
    good = (idx >= 0) & (idx < 77)
    assert torch.equal(out[good], src[idx[good].long()]) and not out[~good].any()
