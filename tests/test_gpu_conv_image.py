"""A layer on few channels taken straight from the image: against 64-bit sums over the same codes; its pooled output is the pooling
sweep's to the bit; pieces that end inside the image, odd extents, filters that fill no step of 16, strides, channels past a group."""
import pytest
import torch

from paper_1605_04711_b200 import nets, twn
from _gpu_util import kernel_launches
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,W,Cin,Cout,k,stride,pad,affine", [
    (3, 28, 28, 1, 32, 5, 1, 0, False), (2, 32, 32, 3, 128, 3, 1, 1, True), (1, 2, 3, 1, 8, 2, 1, 1, True), (2, 9, 301, 3, 72, 3, 1, 2, True),
    (2, 15, 17, 2, 40, 4, 2, 3, True), (1, 70, 5, 7, 96, 3, 2, 0, False), (4, 5, 5, 8, 24, 1, 1, 0, True), (300, 6, 6, 4, 264, 4, 1, 1, True),
    (1, 1, 1, 5, 16, 1, 2, 0, True), (3, 40, 31, 8, 48, (8, 1), 2, 0, True), (2, 600, 400, 1, 16, 8, 2, 7, True)])
@pytest.mark.parametrize("relu", [False, True])
def test_against_64_bits(B, H, W, Cin, Cout, k, stride, pad, affine, relu):
    kh, kw = k if isinstance(k, tuple) else (k, k)
    K = kh * kw * Cin
    codes, packed, ld = packed_codes(Cout, K, 2, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(H * W)
    X = torch.randn((B, H, W, Cin), generator=g, device="cuda").bfloat16()
    d = twn.conv_desc(B, H, W, Cin, Cout, k, stride, pad)
    scale, shift = (torch.randn(Cout, generator=g, device="cuda"), torch.randn(Cout, generator=g, device="cuda")) if affine else (None, None)
    epi = twn.epilogue(scale, shift, relu=relu, out_dtype=twn.BF16)
    pool = d.Ho >= 2 and d.Wo >= 2
    Y = torch.full((B, d.Ho, d.Wo, Cout), 7.0, dtype=torch.bfloat16, device="cuda")
    Yp, want_p = (torch.full((B, d.Ho // 2, d.Wo // 2, Cout), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    twn.conv2d_fwd_image(d, X, packed, ld, None, epi, Y, Yp if pool else None)
    T = torch.as_tensor(codes, dtype=torch.float64, device="cuda").reshape(Cout, kh, kw, Cin).permute(0, 3, 1, 2)
    x = X.double().permute(0, 3, 1, 2)
    s, f = (v.double() if v is not None else u for v, u in ((scale, 1.0), (shift, 0.0)))
    want = torch.nn.functional.conv2d(x, T, stride=stride, padding=pad).permute(0, 2, 3, 1) * s + f
    size = torch.nn.functional.conv2d(x.abs(), T.abs(), stride=stride, padding=pad).permute(0, 2, 3, 1) * (abs(s)) + abs(f)
    want = want.relu() if relu else want
    # half a unit of bf16, and (K + 2) roundings of 32 bits on the sum of the magnitudes
    assert ((Y.double() - want).abs() <= want.abs() * 2.0 ** -8 + size * (K + 2) * 2.0 ** -23).all()
    if pool:
        twn.maxpool2d_fwd(Y, B, d.Ho, d.Wo, Cout, 2, 2, 0, want_p)
        assert torch.equal(Yp.view(torch.int16), want_p.view(torch.int16))


def test_not_a_number():
    """It stays one in every output that reads it, past the ReLU, and never wins a window."""
    _, packed, ld = packed_codes(32, 25, 2, 0, 0)
    X = torch.ones((1, 28, 28, 1), dtype=torch.bfloat16, device="cuda")
    X[0, 10, 11, 0] = float("nan")
    d = twn.conv_desc(1, 28, 28, 1, 32, 5, 1, 0)
    Y, P, want = (torch.zeros((1, n, n, 32), dtype=torch.bfloat16, device="cuda") for n in (24, 12, 12))
    twn.conv2d_fwd_image(d, X, packed, ld, None, twn.epilogue(relu=True, out_dtype=twn.BF16), Y, P)
    nan = torch.zeros((24, 24), dtype=torch.bool, device="cuda")
    nan[6:11, 7:12] = True
    assert torch.equal(Y[0].isnan(), nan[:, :, None].expand(24, 24, 32))
    twn.maxpool2d_fwd(Y, 1, 24, 24, 32, 2, 2, 0, want)
    assert torch.equal(P.view(torch.int16), want.view(torch.int16))


@pytest.mark.parametrize("kw", [dict(k=9), dict(stride=3), dict(pad=5), dict(Cout=36), dict(out_dtype=twn.F32), dict(H=1, W=1, k=1, pool=True)])
def test_what_is_refused(kw):
    c = {"H": 16, "W": 16, "k": 5, "stride": 1, "pad": 0, "Cout": 32, "out_dtype": twn.BF16, "pool": False, **kw}
    buf = torch.zeros(1 << 16, dtype=torch.bfloat16, device="cuda")
    T = torch.zeros((64, 8), dtype=torch.int32, device="cuda")
    d = twn.conv_desc(1, c["H"], c["W"], 1, c["Cout"], c["k"], c["stride"], c["pad"])
    with pytest.raises(twn.TwnError):
        twn.conv2d_fwd_image(d, buf, T, 128, None, twn.epilogue(out_dtype=c["out_dtype"]), buf, buf if c["pool"] else None)


def test_network():
    """LeNet-5 runs its first layer with the pooling in one launch, and a buffer that replaces one of its activations is written."""
    net = nets.lenet5(batch=7)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    net.act["input"].copy_(torch.randn(net.act["input"].shape, generator=g, device="cuda"))
    net.ternarize_all()
    first = net.forward().clone()
    conv1, pool1 = net.act["conv1"].clone(), net.act["pool1"].clone()
    L = net.layers["conv1"]
    assert kernel_launches(lambda: twn.conv2d_fwd_image(L.desc, net.act["input"], L.extra["packed"], L.extra["ld"], L.extra["stats"],
                                                        L.extra["epi"], net.act["conv1"], net.act["pool1"])) == 1
    # a buffer that 16-byte stores cannot reach goes the way of the patch matrix
    odd = torch.zeros(net.act["conv1"].numel() + 2, dtype=torch.bfloat16, device="cuda")[2:].view(net.act["conv1"].shape)
    net.act["conv1"] = odd
    net.act["pool1"].zero_()
    second = net.forward()
    # two orders of 25 products apart
    assert ((odd.float() - conv1.float()).abs() <= conv1.float().abs() * 2.0 ** -7 + 1e-5).all()
    assert ((net.act["pool1"].float() - pool1.float()).abs() <= pool1.float().abs() * 2.0 ** -7 + 1e-5).all()
    assert torch.allclose(first, second, rtol=2e-2, atol=2e-2 * float(first.abs().max()))
