"""Weight gradients whose partial sums are added four outputs at a time: fewer splits than are in flight at once, more, and the
smallest gradient that goes this way with the largest that does not, against 64-bit sums; the same bits on every run."""
import pytest
import torch

from paper_1605_04711_b200 import twn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k,stride", [
    (50, 28, 192, 384, 3, 2), (45, 12, 128, 480, 5, 1), (64, 28, 400, 384, 1, 1), (64, 28, 128, 1184, 1, 1), (64, 28, 128, 1192, 1, 1), (64, 28, 136, 1120, 1, 1),
    (9, 20, 72, 264, 3, 1)])
def test_against_64_bits(B, H, Cin, Cout, k, stride):
    d = twn.conv_desc(B, H, H, Cin, Cout, k, stride, k // 2)
    g = torch.Generator(device="cuda")
    g.manual_seed(Cin)
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    dZ = torch.randn((B, d.Ho, d.Wo, Cout), generator=g, device="cuda").bfloat16()
    dW, again = (torch.full((Cout, k * k * Cin), 7.0, device="cuda") for _ in range(2))
    ws = torch.empty(max(16, twn.conv2d_bwd_weight_workspace_bytes(d)), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    twn.conv2d_bwd_weight(d, X, dZ, dW, ws, status)
    twn.conv2d_bwd_weight(d, X, dZ, again, ws, status)
    assert twn.read_status(status) == 0 and torch.equal(dW, again)
    grad = lambda x, z: torch.nn.grad.conv2d_weight(x.permute(0, 3, 1, 2), (Cout, Cin, k, k), z.permute(0, 3, 1, 2), stride=stride,     # noqa: E731
                                                    padding=k // 2).permute(0, 2, 3, 1).reshape(Cout, -1)
    want, size = grad(X.double(), dZ.double()), grad(X.double().abs(), dZ.double().abs())
    # roundings of 32 bits along the longest chain of additions: a split's pixels, then the splits; a fifth of the pixels is above both
    assert ((dW.double() - want).abs() <= size * max(64, B * d.Ho * d.Wo / 5) * 2.0 ** -24).all()
