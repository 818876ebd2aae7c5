"""A small convolution with the 2x2 pooling of its output where its sums may be split: one kernel (a sweep of its own where that is
modelled faster), the output against 64-bit sums, the pooled values those of the sweep over that output to the bit.  Windows that end with the image, shares of a tile that hold few
of them, channels that fill no tile, a residual, NaN."""
import pytest
import torch

from paper_1605_04711_b200 import twn
from _gpu_util import kernel_launches
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k,stride,residual,kernels", [
    (100, 12, 32, 64, 5, 1, False, 1), (1, 12, 32, 64, 5, 1, True, 2), (8, 12, 32, 64, 5, 1, False, 1), (2, 9, 64, 24, 3, 1, True, 1),
    (5, 7, 256, 56, 3, 1, False, 1), (1, 33, 64, 64, 3, 2, False, 1), (3, 2, 512, 64, 3, 1, True, 2), (16, 14, 128, 40, 3, 1, False, 1),
    (1, 64, 16, 8, 1, 1, False, 1)])
def test_pooled_output(B, H, Cin, Cout, k, stride, residual, kernels):
    K = k * k * Cin
    T, packed, ld = packed_codes(Cout, K, 2, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(H)
    d = twn.conv_desc(B, H, H, Cin, Cout, k, stride, k // 2)
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    R = torch.randn((B, d.Ho, d.Wo, Cout), generator=g, device="cuda").bfloat16() if residual else None
    scale, shift = torch.randn(Cout, generator=g, device="cuda"), torch.randn(Cout, generator=g, device="cuda")
    epi = twn.epilogue(scale, shift, R, relu=not residual, out_dtype=twn.BF16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y = torch.full((B, d.Ho, d.Wo, Cout), 7.0, dtype=torch.bfloat16, device="cuda")
    P, P2 = (torch.full((B, d.Ho // 2, d.Wo // 2, Cout), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    call = lambda: twn.conv2d_fwd_maxpool(d, X, packed, ld, None, epi, Y, P, status)     # noqa: E731
    assert kernel_launches(call) == kernels
    Y.fill_(7.0), P.fill_(7.0)
    call()
    x, w = X.double().permute(0, 3, 1, 2), T.reshape(Cout, k, k, Cin).permute(0, 3, 1, 2)
    conv = lambda a, b: torch.nn.functional.conv2d(a, b, stride=stride, padding=k // 2).permute(0, 2, 3, 1)     # noqa: E731
    want = conv(x, w) * scale.double() + shift.double() + (R.double() if residual else 0.0)
    size = conv(x.abs(), w.abs()) * scale.double().abs() + shift.double().abs() + (R.double().abs() if residual else 0.0)
    want = want if residual else want.relu()
    # half a unit of bf16, and the roundings of 32 bits of a sum in any order: K at most, of its magnitudes
    assert ((Y.double() - want).abs() <= want.abs() * 2.0 ** -8 + size * (K + 3) * 2.0 ** -23).all()
    twn.maxpool2d_fwd(Y, B, d.Ho, d.Wo, Cout, 2, 2, 0, P2)
    assert torch.equal(P.view(torch.int16), P2.view(torch.int16))
    X[0, 1, 1, 3] = float("nan")
    call()
    twn.maxpool2d_fwd(Y, B, d.Ho, d.Wo, Cout, 2, 2, 0, P2)
    assert Y.isnan().any() and torch.equal(P.view(torch.int16), P2.view(torch.int16))
    assert twn.read_status(status) == 0
