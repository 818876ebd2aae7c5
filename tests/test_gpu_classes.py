"""The residue classes of a strided backward pass in one launch of the general kernel, against 64-bit sums: classes without taps, odd
extents, channels that fill no tile, codes on every boundary, more taps than the table of code offsets holds, both code widths, a
residual in place and one that gates."""
import pytest
import torch

from paper_1605_04711_b200 import twn
from _gpu_util import kernel_launches
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k,kernels", [
    (50, 28, 192, 384, 3, 1), (20, 56, 64, 128, 3, 1), (64, 28, 128, 256, 1, 1), (24, 25, 704, 384, 3, 1), (128, 19, 608, 368, 1, 1),
    (6, 66, 544, 240, 3, 4), (17, 35, 448, 320, 3, 1), (15, 41, 72, 1472, 3, 1), (49, 42, 128, 128, 5, 1)])
@pytest.mark.parametrize("epilogue", ["plain", "add", "gate"])
def test_against_64_bits(B, H, Cin, Cout, k, kernels, epilogue):
    d = twn.conv_desc(B, H, H, Cin, Cout, k, 2, k // 2)
    T, packed, ld = packed_codes(Cin, k * k * Cout, 2, 0, 0)           # rows: input channels, columns: taps, output channels
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    dZ = torch.randn((B, d.Ho, d.Wo, Cout), generator=g, device="cuda").bfloat16()
    R = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    scale, shift = torch.randn(Cin, generator=g, device="cuda"), torch.randn(Cin, generator=g, device="cuda")
    dX = R.clone() if epilogue == "add" else torch.full((B, H, H, Cin), 7.0, dtype=torch.bfloat16, device="cuda")
    epi = {"plain": lambda: twn.epilogue(scale, shift, relu=True, out_dtype=twn.BF16),
           "add": lambda: twn.epilogue(None, None, dX, out_dtype=twn.BF16),
           "gate": lambda: twn.epilogue(scale, None, R, out_dtype=twn.BF16, residual_op=twn.RESIDUAL_GATE)}[epilogue]()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    call = lambda: twn.conv2d_bwd_data(d, dZ, packed, ld, None, epi, dX, status)     # noqa: E731
    if epilogue == "plain":
        assert kernel_launches(call) == kernels
    call()
    # [Cin][kh][kw][Cout] -> the filter of the forward pass [Cout][Cin][kh][kw]
    w = T.reshape(Cin, k, k, Cout).permute(3, 0, 1, 2)
    z = dZ.double().permute(0, 3, 1, 2)
    back = lambda a, b: torch.nn.grad.conv2d_input((B, Cin, H, H), b, a, stride=2, padding=k // 2).permute(0, 2, 3, 1)     # noqa: E731
    want, size = back(z, w), back(z.abs(), w.abs())
    if epilogue == "plain":
        want, size = (want * scale.double() + shift.double()).relu(), size * scale.double().abs() + shift.double().abs()
    elif epilogue == "add":
        want, size = want + R.double(), size + R.double().abs()
    else:
        want, size = torch.where(R > 0, want * scale.double(), 0.0), size * scale.double().abs()
    assert twn.read_status(status) == 0
    # half a unit of bf16, and the roundings of 32 bits of a sum of k * k * Cout / 4 and more products in any order
    assert ((dX.double() - want).abs() <= want.abs() * 2.0 ** -8 + size * (k * k * Cout + 3) * 2.0 ** -23).all()


def test_binary_codes():
    B, H, Cin, Cout, k = 50, 28, 192, 384, 3
    d = twn.conv_desc(B, H, H, Cin, Cout, k, 2, 1)
    T, packed, ld = packed_codes(Cin, k * k * Cout, 1, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    dZ = torch.randn((B, d.Ho, d.Wo, Cout), generator=g, device="cuda").bfloat16()
    dX = torch.full((B, H, H, Cin), 7.0, dtype=torch.bfloat16, device="cuda")
    call = lambda: twn.conv2d_bwd_data_b1(d, dZ, packed, ld, None, twn.epilogue(out_dtype=twn.BF16), dX)     # noqa: E731
    assert kernel_launches(call) == 1
    call()
    w = T.reshape(Cin, k, k, Cout).permute(3, 0, 1, 2)
    want = torch.nn.grad.conv2d_input((B, Cin, H, H), w, dZ.double().permute(0, 3, 1, 2), stride=2, padding=1).permute(0, 2, 3, 1)
    assert ((dX.double() - want).abs() <= want.abs() * 2.0 ** -8 + k * k * Cout * 2.0 ** -20).all()
