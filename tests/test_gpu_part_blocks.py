"""Channel counts that are no multiple of 64: the codes of a k-block lie on 16, 8 or 4-byte boundaries.  With the sums in order the result has the bits of the same layer whose channels are filled up with zeros to a multiple of 64,
in the general kernel (many pixels) and in the split one (few), for both code widths."""
import pytest
import torch

import oracle
from paper_1605_04711_b200 import twn
from _gpu_util import dev_u32
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Cin", [32, 96, 160, 224, 16, 80, 176])
@pytest.mark.parametrize("B,H,Cout", [(40, 28, 192), (3, 9, 72), (64, 7, 520)])
@pytest.mark.parametrize("bits", [2, 1])
def test_against_filled_channels(B, H, Cin, Cout, bits):
    if bits == 1 and Cin % 32:
        pytest.skip("binary codes of several taps start on whole words")
    k, full = 3, (Cin + 63) // 64 * 64
    codes, packed, ld = packed_codes(Cout, k * k * Cin, bits, 0, 0)
    filled = torch.ones((Cout, k * k, full), dtype=torch.int8)          # binary codes have no zero; their channels are zero
    if bits == 2:
        filled.zero_()
    filled[:, :, :Cin] = codes.cpu().reshape(Cout, k * k, Cin).to(torch.int8)
    filled = filled.reshape(Cout, -1).numpy()
    ld2 = twn.ld_for(k * k * full) if bits == 2 else twn.ld_for_b1(k * k * full)
    packed2 = dev_u32(oracle.pack(filled, ld2) if bits == 2 else oracle.pack1(filled, ld2)).reshape(Cout, -1)
    g = torch.Generator(device="cuda")
    g.manual_seed(Cin)
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    X2 = torch.zeros((B, H, H, full), dtype=torch.bfloat16, device="cuda")
    X2[..., :Cin] = X
    epi = twn.epilogue(out_dtype=twn.F32, residual_op=twn.SUM_IN_ORDER)
    call = twn.conv2d_fwd if bits == 2 else twn.conv2d_fwd_b1
    Y, Y2 = (torch.full((B, H, H, Cout), 7.0, device="cuda") for _ in range(2))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    call(twn.conv_desc(B, H, H, Cin, Cout, k, 1, 1), X, packed, ld, None, epi, Y, status)
    call(twn.conv_desc(B, H, H, full, Cout, k, 1, 1), X2, packed2, ld2, None, epi, Y2, status)
    assert twn.read_status(status) == 0
    assert torch.equal(Y.view(torch.int32), Y2.view(torch.int32))
