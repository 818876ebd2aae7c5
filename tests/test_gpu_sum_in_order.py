"""TWN_SUM_IN_ORDER: an output's bits depend neither on the batch nor on the kernel that the batch leads to.

Batches from one image to a full GPU take a call through the split, the resident-weight and the general kernel; with one
and several channel blocks and taps, every epilogue path (fp32, bf16, residual), both directions and both code widths."""
import pytest
import torch

from paper_1605_04711_b200 import twn

pytestmark = pytest.mark.gpu


def packed_codes(rows, cols, bits, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = torch.randn(rows, cols, device="cuda", generator=g)
    ld = twn.ld_for(cols) if bits == 2 else twn.ld_for_b1(cols)
    packed, stats = torch.zeros((rows, ld * bits // 32), dtype=torch.int32, device="cuda"), twn.new_stats()
    if bits == 2:
        twn.ternarize(W, 0.7, stats, packed, ld, None, torch.empty(twn.ternarize_workspace_bytes(), dtype=torch.uint8, device="cuda"))
    else:
        twn.binarize(W, stats, packed, ld, torch.empty(twn.binarize_workspace_bytes(), dtype=torch.uint8, device="cuda"))
    return packed, ld, stats


def bits_of(t):
    return t.view(torch.int32 if t.dtype == torch.float32 else torch.int16)


def same_bits_over_batches(batches, X, shape_of, call, epi):
    """call(batch, input, epilogue, output) for each batch; the outputs of the images they share are compared."""
    g = torch.Generator(device="cuda").manual_seed(9)
    most, dtype = max(batches), torch.float32 if epi == "f32" else torch.bfloat16
    C = shape_of(1)[-1]
    scale, shift = torch.randn(C, device="cuda", generator=g), torch.randn(C, device="cuda", generator=g)
    res = torch.randn(shape_of(most), device="cuda", generator=g).bfloat16() if epi == "residual" else None
    outs = {}
    for b in batches:
        Y = torch.full(shape_of(b), float("nan"), dtype=dtype, device="cuda")
        r = None if res is None else res[:b].contiguous()
        e = (twn.epilogue(out_dtype=twn.F32, residual_op=twn.SUM_IN_ORDER) if epi == "f32" else
             twn.epilogue(scale, shift, r, relu=True, out_dtype=twn.BF16, residual_op=twn.SUM_IN_ORDER))
        x = X[:b].contiguous()
        call(b, x, e, Y)
        torch.cuda.synchronize()
        outs[b] = Y
    for b in batches:
        assert torch.equal(bits_of(outs[b]), bits_of(outs[most][:b])), f"batch {b} against {most}"


FORWARD = [
    # H, Cin, Cout, k, stride, batches: at one of them the resident-weight kernel would be the fastest
    (28, 128, 64, 3, 1, (1, 4, 16, 64)), (28, 96, 64, 3, 1, (1, 8, 32)), (56, 160, 32, 3, 1, (1, 8)), (32, 96, 192, 3, 1, (1, 64, 128)),
    # one channel block, or one tap: its order is that of the others
    (28, 64, 64, 3, 1, (1, 8, 64)), (20, 32, 272, 3, 1, (1, 16, 64)), (56, 160, 80, 1, 1, (1, 8, 64)),
    # general and split kernel
    (14, 256, 256, 3, 1, (1, 8, 64)), (28, 64, 128, 3, 2, (1, 8, 64)), (12, 128, 64, 5, 1, (1, 16, 64)),
]


@pytest.mark.parametrize("epi", ["f32", "affine", "residual"])
@pytest.mark.parametrize("H,Cin,Cout,k,stride,batches", FORWARD)
def test_forward(H, Cin, Cout, k, stride, batches, epi, bits=2):
    packed, ld, stats = packed_codes(Cout, k * k * Cin, bits, 1)
    X = torch.randn(max(batches), H, H, Cin, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2)).bfloat16()
    Ho = (H + 2 * (k // 2) - k) // stride + 1
    fwd = twn.conv2d_fwd if bits == 2 else twn.conv2d_fwd_b1
    same_bits_over_batches(batches, X, lambda b: (b, Ho, Ho, Cout), lambda b, x, e, Y:
                           fwd(twn.conv_desc(b, H, H, Cin, Cout, k, stride, k // 2), x, packed, ld, stats, e, Y), epi)


def test_forward_of_binary_weights():
    test_forward(28, 128, 64, 3, 1, (1, 4, 16), "f32", bits=1)


@pytest.mark.parametrize("epi", ["f32", "residual"])
@pytest.mark.parametrize("H,Cin,Cout,k,stride,batches", [(28, 192, 384, 3, 2, (1, 50)), (28, 64, 128, 3, 2, (1, 20, 200)),
                                                          (28, 64, 128, 3, 1, (1, 16, 64)), (14, 256, 256, 3, 1, (1, 64))])
def test_backward_for_data(H, Cin, Cout, k, stride, batches, epi):
    packed, ld, stats = packed_codes(Cout, k * k * Cin, 2, 3)
    ld_b = twn.ld_for(k * k * Cout)
    packed_b = torch.zeros((Cin, ld_b // 16), dtype=torch.int32, device="cuda")
    twn.transpose_codes(packed, ld, twn.conv_desc(1, H, H, Cin, Cout, k, stride, k // 2), packed_b, ld_b)
    Ho = (H + 2 * (k // 2) - k) // stride + 1
    dZ = torch.randn(max(batches), Ho, Ho, Cout, device="cuda", generator=torch.Generator(device="cuda").manual_seed(4)).bfloat16()
    same_bits_over_batches(batches, dZ, lambda b: (b, H, H, Cin), lambda b, x, e, Y:
                           twn.conv2d_bwd_data(twn.conv_desc(b, H, H, Cin, Cout, k, stride, k // 2), x, packed_b, ld_b, stats, e, Y), epi)


@pytest.mark.parametrize("K,N,rows", [(4608, 512, (1, 300, 4001)), (1024, 10, (1, 70, 30000)), (176, 960, (1, 14704))])
def test_inner_product(K, N, rows):
    packed, ld, stats = packed_codes(N, K, 2, 5)
    X = torch.randn(max(rows), K, device="cuda", generator=torch.Generator(device="cuda").manual_seed(6)).bfloat16()
    same_bits_over_batches(rows, X, lambda m: (m, N), lambda m, x, e, Y: twn.gemm(x, K, packed, ld, stats, m, N, K, e, Y, N), "f32")
