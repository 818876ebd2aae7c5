"""Strided backward for data where the choice lies between one launch of all residue classes and a launch per class: shapes
on both sides, with every kernel that a class may run."""
import pytest
import torch

from paper_1605_04711_b200 import twn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Cin,Cout,k", [
    (5, 76, 640, 32, 3), (10, 100, 48, 64, 3), (8, 112, 32, 64, 3), (31, 68, 96, 160, 3), (64, 56, 64, 128, 1),      # near the line
    (64, 56, 64, 128, 3), (20, 56, 64, 128, 3), (8, 31, 512, 192, 5), (1, 16, 64, 64, 3), (3, 7, 96, 96, 5)])
@pytest.mark.parametrize("op", ["plain", "gate", "add"])
def test_against_fp64(B, H, Cin, Cout, k, op):
    g = torch.Generator(device="cuda").manual_seed(B + H)
    K, Ho = k * k * Cin, (H + 2 * (k // 2) - k) // 2 + 1
    d = twn.conv_desc(B, H, H, Cin, Cout, k, 2, k // 2)
    codes = torch.randint(-1, 2, (Cout, K), dtype=torch.int8, device="cuda", generator=g)
    ld, ld_b = twn.ld_for(K), twn.ld_for(k * k * Cout)
    packed = torch.zeros((Cout, ld // 16), dtype=torch.int32, device="cuda")
    packed_b = torch.zeros((Cin, ld_b // 16), dtype=torch.int32, device="cuda")
    twn.pack(codes, Cout, K, packed, ld)
    twn.transpose_codes(packed, ld, d, packed_b, ld_b)
    dZ = torch.randn(B, Ho, Ho, Cout, device="cuda", generator=g).bfloat16()
    other = torch.randn(B, H, H, Cin, device="cuda", generator=g).bfloat16()
    dX = other.clone() if op == "add" else torch.full((B, H, H, Cin), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    e = {"plain": lambda: twn.epilogue(out_dtype=twn.BF16), "add": lambda: twn.epilogue(residual=dX, out_dtype=twn.BF16),
         "gate": lambda: twn.epilogue(residual=other, out_dtype=twn.BF16, residual_op=twn.RESIDUAL_GATE)}[op]()
    twn.conv2d_bwd_data(d, dZ, packed_b, ld_b, None, e, dX, status)
    assert twn.read_status(status) == 0
    T = codes.view(Cout, k, k, Cin).permute(0, 3, 1, 2).double()
    pick = sorted({0, B // 2, B - 1})
    z = dZ[pick].double().permute(0, 3, 1, 2)
    want, size = (torch.nn.grad.conv2d_input((len(pick), Cin, H, H), t, y, stride=2, padding=k // 2).permute(0, 2, 3, 1)
                  for t, y in ((T, z), (T.abs(), z.abs())))
    o = other[pick].double()
    want = torch.where(o > 0, want, 0.0) if op == "gate" else want + o if op == "add" else want
    # fp32 sums of at most k * k * Cout terms, then one rounding to bf16
    tol = 2.0 ** -24 * k * k * Cout * (size + o.abs()) + 1e-6
    assert bool(((dX[pick].double() - want).abs() <= tol + 2.0 ** -8 * (want.abs() + tol)).all())
