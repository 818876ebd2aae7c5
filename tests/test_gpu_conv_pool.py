"""A convolution with the 2x2 pooling of its output: output and pooled values are those of the convolution and the pooling sweep
to the bit, whether the call is one kernel or two (and it is the one where the case says so); odd extents, several images in a
tile, channels that fill no store, every tile shape, NaN."""
import pytest
import torch

from paper_1605_04711_b200 import nets, twn
from _gpu_util import kernel_launches
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k,stride,relu,affine,kernels", [
    # pooled in the epilogue
    (40, 32, 64, 128, 3, 1, True, True, 1), (33, 15, 128, 136, 3, 1, True, False, 1), (200, 6, 96, 48, 3, 1, False, False, 1),
    (64, 28, 64, 256, 5, 2, True, True, 1), (100, 12, 32, 64, 5, 1, True, False, 1), (128, 8, 512, 512, 3, 1, True, True, 1),
    # by a sweep: faster so, or (20 channels) nothing that the epilogue can store
    (128, 8, 256, 264, 3, 1, False, True, 2), (100, 7, 512, 512, 3, 1, True, True, 2), (500, 2, 64, 96, 1, 1, False, True, 2),
    (2, 9, 64, 24, 3, 1, True, True, 2), (3, 11, 64, 20, 3, 1, True, True, 2)])
def test_pooled_output(B, H, Cin, Cout, k, stride, relu, affine, kernels):
    _, packed, ld = packed_codes(Cout, k * k * Cin, 2, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(H)
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    X[0, 1, 1, 3] = float("nan")
    d = twn.conv_desc(B, H, H, Cin, Cout, k, stride, k // 2)
    scale, shift = (torch.randn(Cout, generator=g, device="cuda"), torch.randn(Cout, generator=g, device="cuda")) if affine else (None, None)
    epi = twn.epilogue(scale, shift, relu=relu, out_dtype=twn.BF16, residual_op=twn.SUM_IN_ORDER)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y, Y2 = (torch.full((B, d.Ho, d.Wo, Cout), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    P, P2 = (torch.full((B, d.Ho // 2, d.Wo // 2, Cout), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    assert kernel_launches(lambda: twn.conv2d_fwd_maxpool(d, X, packed, ld, None, epi, Y, P, status)) == kernels
    Y.fill_(7.0), P.fill_(7.0)
    twn.conv2d_fwd_maxpool(d, X, packed, ld, None, epi, Y, P, status)
    twn.conv2d_fwd(d, X, packed, ld, None, epi, Y2, status)
    twn.maxpool2d_fwd(Y, B, d.Ho, d.Wo, Cout, 2, 2, 0, P2)
    assert twn.read_status(status) == 0
    assert torch.equal(Y.view(torch.int16), Y2.view(torch.int16))      # the sums in order, in every kernel
    assert torch.equal(P.view(torch.int16), P2.view(torch.int16))


def test_what_is_refused():
    _, packed, ld = packed_codes(16, 64, 2, 0, 0)
    X = torch.zeros((2, 1, 4, 64), dtype=torch.bfloat16, device="cuda")
    Y, P = torch.zeros((2, 1, 4, 16), dtype=torch.bfloat16, device="cuda"), torch.zeros(64, dtype=torch.bfloat16, device="cuda")
    d = twn.conv_desc(2, 1, 4, 64, 16, 1, 1, 0)
    with pytest.raises(twn.TwnError):                      # one row: no window
        twn.conv2d_fwd_maxpool(d, X, packed, ld, None, twn.epilogue(out_dtype=twn.BF16), Y, P)
    d = twn.conv_desc(2, 4, 1, 64, 16, 1, 1, 0)
    with pytest.raises(twn.TwnError):
        twn.conv2d_fwd_maxpool(d, X, packed, ld, None, None, Y, P)


def test_network_with_and_without():
    """A VGG-7's activations and pooled activations are those of the calls apart, layer by layer, with the sums in order: at 24
    images every pooled layer runs in the kernel that pools, which never splits them."""
    net = nets.vgg7(batch=24)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    net.act["input"].copy_(torch.randn(net.act["input"].shape, generator=g, device="cuda"))
    net.ternarize_all()
    assert kernel_launches(net.forward) == 9           # patch matrix, six convolutions, two inner products
    net.forward()
    pools = [op for op in net.ops if op[0] == "maxpool"]
    assert len(pools) == 3
    for _, name, src, *_ in pools:
        L = net.layers[src]
        e, y = L.extra, net.act[src]
        apart, want = torch.empty_like(y), torch.empty_like(net.act[name])
        epi = twn.epilogue(e["scale"], e["shift"], relu=True, out_dtype=twn.BF16, residual_op=twn.SUM_IN_ORDER)
        twn.conv2d_fwd(L.desc, net.act[L.src], e["packed"], e["ld"], e["stats"], epi, apart)
        twn.maxpool2d_fwd(apart, *apart.shape, 2, 2, 0, want)
        assert torch.equal(y.view(torch.int16), apart.view(torch.int16))
        assert torch.equal(net.act[name].view(torch.int16), want.view(torch.int16))
