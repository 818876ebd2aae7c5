"""The convolution from the image at its limits of size: many small images, whose outputs are far from 2^32 although each with a unit's
worth of pixels around it would not be, and an image wider than the kernel takes, which a network gives to the product."""
import pytest
import torch

from paper_1605_04711_b200 import nets, twn
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


def test_many_small_images():
    B, Cout = 420000, 32                         # 53.8 million outputs; 18 x 18 pixels an image would make 2^32.02
    T, packed, ld = packed_codes(Cout, 1, 2, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    X = torch.randn((B, 2, 2, 1), generator=g, device="cuda").bfloat16()
    Y, Yp = (torch.full((B, n, n, Cout), 7.0, dtype=torch.bfloat16, device="cuda") for n in (2, 1))
    twn.conv2d_fwd_image(twn.conv_desc(B, 2, 2, 1, Cout, 1, 1, 0), X, packed, ld, None, twn.epilogue(out_dtype=twn.BF16), Y, Yp)
    want = X * T.view(Cout).bfloat16()           # one product by -1, 0 or 1: exact
    assert torch.equal(Y, want)
    assert torch.equal(Yp, want.amax((1, 2), keepdim=True))


def test_a_wide_image():
    W = 2 ** 24
    net = nets.TernaryNet("wide", 1, (1, W, 1), [("layer", nets.Layer("conv", 1, 8, H=1, W=W, src="input"))])
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    net.act["input"].copy_(torch.randn((1, 1, W, 1), generator=g, device="cuda"))
    net.ternarize_all()
    net.forward()
    L = net.layers["conv"]
    e, y = L.extra, net.act["conv"]
    columns, want = torch.zeros((W, L.ldk), dtype=torch.bfloat16, device="cuda"), torch.full_like(y, 7.0)
    twn.im2col(L.desc, net.act["input"], columns, L.ldk)
    twn.gemm(columns, L.ldk, e["packed"], e["ld"], e["stats"], W, 8, 1, e["epi"], want, 8)
    assert torch.equal(y.view(torch.int16), want.view(torch.int16)) and bool((y != 0).any())
