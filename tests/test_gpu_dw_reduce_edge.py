"""Weight gradients on both sides of the size from which their partial sums are added four outputs at a time (a block of 256 threads for
every SM), and one with more splits than are in flight at once just below it, against 64-bit sums; the same bits on every run."""
import pytest
import torch

from paper_1605_04711_b200 import twn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [-8, 0, 8])
def test_around_the_limit(side):
    edge = torch.cuda.get_device_properties(0).multi_processor_count * 256 * 4           # outputs
    check(64, 28, 128, edge // 128 // 8 * 8 + side, 1)


def test_many_splits_below():
    check(64, 28, 128, 128, 3)


def check(B, H, Cin, Cout, k):
    d = twn.conv_desc(B, H, H, Cin, Cout, k, 1, k // 2)
    g = torch.Generator(device="cuda")
    g.manual_seed(Cout)
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    dZ = torch.randn((B, d.Ho, d.Wo, Cout), generator=g, device="cuda").bfloat16()
    dW, again = (torch.full((Cout, k * k * Cin), 7.0, device="cuda") for _ in range(2))
    size = twn.conv2d_bwd_weight_workspace_bytes(d)
    assert size > Cout * k * k * Cin * 4                   # more than one split
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    twn.conv2d_bwd_weight(d, X, dZ, dW, ws, status)
    twn.conv2d_bwd_weight(d, X, dZ, again, ws, status)
    assert twn.read_status(status) == 0 and torch.equal(dW, again)
    grad = lambda x, z: torch.nn.grad.conv2d_weight(x.permute(0, 3, 1, 2), (Cout, Cin, k, k), z.permute(0, 3, 1, 2),     # noqa: E731
                                                    padding=k // 2).permute(0, 2, 3, 1).reshape(Cout, -1)
    want, size = grad(X.double(), dZ.double()), grad(X.double().abs(), dZ.double().abs())
    # roundings of 32 bits along the longest chain of additions: a split's pixels, then the splits; a fifth of the pixels is above both
    assert ((dW.double() - want).abs() <= size * max(64, B * d.Ho * d.Wo / 5) * 2.0 ** -24).all()
