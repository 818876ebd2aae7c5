"""Filters without padding whose rows are taken as one run of elements: with the sums in order the outputs have the bits of the same
layer on an image that carries its padding (a column of zeros around it, where every tap is taken by itself), strides, both code
widths, a pooled output."""
import pytest
import torch

from paper_1605_04711_b200 import twn
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k,stride", [
    (100, 12, 32, 64, 5, 1), (3, 12, 32, 64, 5, 1), (64, 28, 96, 192, 3, 1), (2, 9, 160, 72, 3, 2), (40, 30, 16, 128, 5, 1), (50, 57, 32, 64, 3, 2),
    (1, 3, 224, 24, 3, 1)])
@pytest.mark.parametrize("bits", [2, 1])
def test_bits(B, H, Cin, Cout, k, stride, bits):
    if bits == 1 and Cin % 32:
        pytest.skip("binary codes of several taps start on whole words")
    _, packed, ld = packed_codes(Cout, k * k * Cin, bits, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(H)
    # the image and, on its right, columns that no output reads: the padded layer's outputs there are left out
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    d = twn.conv_desc(B, H, H, Cin, Cout, k, stride, 0)
    wide = twn.ConvDesc(B, H, H, Cin, Cout, k, k, stride, stride, 0, stride)       # one more output on the left
    call = twn.conv2d_fwd if bits == 2 else twn.conv2d_fwd_b1
    epi = twn.epilogue(out_dtype=twn.F32, residual_op=twn.SUM_IN_ORDER)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y = torch.full((B, d.Ho, d.Wo, Cout), 7.0, device="cuda")
    Y2 = torch.full((B, wide.Ho, wide.Wo, Cout), 7.0, device="cuda")
    call(d, X, packed, ld, None, epi, Y, status)
    call(wide, X, packed, ld, None, epi, Y2, status)
    assert twn.read_status(status) == 0
    assert torch.equal(Y, Y2[:, :, 1:1 + d.Wo])
    if bits == 2 and d.Ho >= 2 and Cout % 8 == 0:
        Z, P, P2 = (torch.zeros((B, h, w, Cout), dtype=torch.bfloat16, device="cuda")
                    for h, w in ((d.Ho, d.Wo), (d.Ho // 2, d.Wo // 2), (d.Ho // 2, d.Wo // 2)))
        twn.conv2d_fwd_maxpool(d, X, packed, ld, None, twn.epilogue(relu=True, out_dtype=twn.BF16), Z, P, status)
        twn.maxpool2d_fwd(Z, B, d.Ho, d.Wo, Cout, 2, 2, 0, P2)
        assert torch.equal(P, P2)
        # a split sum is another order: as far from the sums in order as k * k * Cin roundings
        assert ((Z.float() - Y.relu()).abs() <= Y.abs() * 2.0 ** -7 + k * k * Cin * 2.0 ** -20).all()
