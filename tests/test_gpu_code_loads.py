"""The general contraction's three tile shapes and the ways it fetches codes: two k-blocks at once (even and odd counts, a row
pitch with room behind the last), 16 bytes at once (odd pitch, a matrix off the 32-byte boundaries), single words (channel counts
that are no multiple of 64), both code widths.  The oracle is the product in 64 bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_04711_b200 import twn
from _gpu_util import dev_u32

pytestmark = pytest.mark.gpu


def packed_codes(rows, cols, bits, extra, offset):
    c = np.random.default_rng(rows + cols).integers(-1, 2, (rows, cols)).astype(np.int8)
    c = c if bits == 2 else np.where(c < 0, -1, 1).astype(np.int8)
    ld = (twn.ld_for(cols) if bits == 2 else twn.ld_for_b1(cols)) + extra
    words = dev_u32(oracle.pack(c, ld) if bits == 2 else oracle.pack1(c, ld)).reshape(-1)
    buf = torch.zeros(words.numel() + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = words
    return torch.from_numpy(c).cuda().double(), buf[offset:].view(rows, -1), ld


@pytest.mark.parametrize("M,N,K,bits,extra,offset", [
    (4001, 512, 1152, 2, 0, 0), (4001, 512, 1216, 2, 64, 0), (4001, 512, 1984, 2, 0, 0), (4001, 500, 1152, 2, 0, 4),
    (4001, 512, 1984, 1, 0, 0), (4001, 512, 1100, 1, 128, 0), (4001, 512, 9000, 2, 0, 0), (9472, 512, 12288, 2, 0, 0)])
def test_inner_product(M, N, K, bits, extra, offset):
    T, packed, ld = packed_codes(N, K, bits, extra, offset)
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    X = torch.zeros((M, (K + 7) // 8 * 8), dtype=torch.bfloat16, device="cuda")
    X[:, :K] = torch.randn((M, K), generator=g, device="cuda").bfloat16()
    Y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    (twn.gemm if bits == 2 else twn.gemm_b1)(X, X.shape[1], packed, ld, None, M, N, K, None, Y, N, status)
    Xd = X[:, :K].double()
    assert twn.read_status(status) == 0
    assert bool(((Y.double() - Xd @ T.T).abs() <= 1e-4 * (Xd.abs() @ T.abs().T) + 1e-6).all())


@pytest.mark.parametrize("B,H,Cin,Cout,k,stride,bits", [
    (100, 7, 512, 512, 3, 1, 2), (40, 14, 224, 512, 3, 1, 2), (70, 28, 96, 272, 5, 2, 2), (64, 14, 192, 250, 3, 1, 2), (64, 14, 96, 256, 5, 1, 1)])
def test_convolution(B, H, Cin, Cout, k, stride, bits):
    T, packed, ld = packed_codes(Cout, k * k * Cin, bits, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(Cin)
    X = torch.randn((B, H, H, Cin), generator=g, device="cuda").bfloat16()
    d = twn.conv_desc(B, H, H, Cin, Cout, k, stride, k // 2)
    Y = torch.full((B, d.Ho, d.Wo, Cout), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    (twn.conv2d_fwd if bits == 2 else twn.conv2d_fwd_b1)(d, X, packed, ld, None, twn.epilogue(out_dtype=twn.F32), Y, status)
    x, w = X.double().permute(0, 3, 1, 2), T.view(Cout, k, k, Cin).permute(0, 3, 1, 2)
    conv = lambda x, w: torch.nn.functional.conv2d(x, w, stride=stride, padding=k // 2).permute(0, 2, 3, 1)     # noqa: E731
    assert twn.read_status(status) == 0
    assert bool(((Y.double() - conv(x, w)).abs() <= 1e-4 * conv(x.abs(), w.abs()) + 1e-6).all())
