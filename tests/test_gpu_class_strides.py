"""The residue classes of a backward pass whose strides differ in h and w, two to four of them in one launch of the general kernel,
against 64-bit sums: extents that end inside a class, classes without taps, a residual in place and one that gates."""
import pytest
import torch

from paper_1605_04711_b200 import twn
from test_gpu_class_choice import kernel_names
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k,strides", [
    (20, 32, 256, 256, 3, (1, 2)), (59, 35, 112, 64, 3, (1, 2)), (12, 20, 352, 384, 3, (2, 1)), (18, 42, 128, 128, 5, (2, 1)),
    (19, 44, 224, 208, 1, (1, 3)), (39, 36, 64, 96, 3, (1, 3)), (41, 29, 72, 128, 3, (3, 1)), (43, 36, 248, 384, 1, (3, 1)),
    (37, 25, 152, 64, 1, (1, 4)), (35, 26, 232, 128, 5, (1, 4)), (23, 38, 160, 64, 5, (4, 1)), (30, 26, 432, 256, 1, (4, 1))])
@pytest.mark.parametrize("epilogue", ["plain", "add", "gate"])
def test_against_64_bits(B, H, Cin, Cout, k, strides, epilogue):
    d = twn.ConvDesc(B, H, H, Cin, Cout, k, k, *strides, k // 2, k // 2)
    T, packed, ld = packed_codes(Cin, k * k * Cout, 2, 0, 0)
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
        names = kernel_names(call)
        assert len(names) == 1 and "tconv_kernel" in names[0]
    call()
    w, z = T.reshape(Cin, k, k, Cout).permute(3, 0, 1, 2), dZ.double().permute(0, 3, 1, 2)
    back = lambda a, b: torch.nn.grad.conv2d_input((B, Cin, H, H), b, a, stride=strides, padding=k // 2).permute(0, 2, 3, 1)     # noqa: E731
    want, size = back(z, w), back(z.abs(), w.abs())
    if epilogue == "plain":
        want, size = (want * scale.double() + shift.double()).relu(), size * scale.double().abs() + shift.double().abs()
    elif epilogue == "add":
        want, size = want + R.double(), size + R.double().abs()
    else:
        want, size = torch.where(R > 0, want * scale.double(), 0.0), size * scale.double().abs()
    assert twn.read_status(status) == 0
    # half a unit of bf16, and the roundings of 32 bits of a sum of at most k * k * Cout products in any order
    assert ((dX.double() - want).abs() <= want.abs() * 2.0 ** -8 + size * (k * k * Cout + 3) * 2.0 ** -23).all()
