"""The contraction that splits its reduction over a cluster, at its edges: one pixel, reductions shorter and longer than the
split, channels that fill no tile, strides, both code widths, every epilogue, and the outputs of which no four are aligned."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_04711_b200 import datagen as dg
from paper_1605_04711_b200 import twn
from _gpu_util import dev_bf16, dev_f32, dev_u32

pytestmark = pytest.mark.gpu


def codes_of(n, seed, bits):
    c = np.random.default_rng(seed).integers(-1, 2, n).astype(np.int8)
    return c if bits == 2 else np.where(c < 0, -1, 1).astype(np.int8)


@pytest.mark.parametrize("B,H,Cin,Cout,k,stride,bits,epi", [
    (1, 1, 64, 8, 1, 1, 2, "plain"), (1, 1, 1024, 512, 1, 1, 2, "plain"), (33, 1, 200, 10, 1, 1, 2, "f32res"),
    (2, 8, 160, 400, 3, 2, 2, "affine"), (3, 9, 96, 272, 3, 1, 2, "residual"), (1, 15, 256, 129, 3, 1, 2, "affine"),
    (1, 7, 768, 48, 5, 1, 1, "gate"), (5, 14, 64, 131, 3, 2, 1, "residual"), (2, 13, 512, 640, 1, 1, 1, "affine")])
def test_forward(B, H, Cin, Cout, k, stride, bits, epi):
    K = k * k * Cin
    d = twn.conv_desc(B, H, H, Cin, Cout, k, stride, k // 2)
    od = oracle.conv_desc(B, H, H, Cin, Cout, k, stride, k // 2)
    codes = codes_of(Cout * K, 3, bits).reshape(Cout, K)
    ld = twn.ld_for(K) if bits == 2 else twn.ld_for_b1(K)
    packed = dev_u32(oracle.pack(codes, ld) if bits == 2 else oracle.pack1(codes, ld))
    X = dg.draw_bf16(1, "split-x", B * H * H * Cin, "normal").reshape(B, H, H, Cin)
    shape = (B, d.Ho, d.Wo, Cout)
    n = int(np.prod(shape))
    scale = shift = res = None
    res_host = None
    if epi in ("affine", "residual", "gate"):
        scale, shift = dg.draw(1, "split-s", Cout, "normal", 1.0, 0.3), dg.draw(1, "split-b", Cout, "normal")
    if epi in ("residual", "gate"):
        bits16 = dg.draw_bf16(1, "split-r", n, "normal").reshape(shape)
        res, res_host = dev_bf16(bits16), dg.bf16_bits_to_f64(bits16)
    if epi == "f32res":
        r = dg.draw(1, "split-r", n, "normal").reshape(shape)
        res, res_host = dev_f32(r), r.astype(np.float64)
    relu = epi in ("affine", "residual")
    bf16 = epi != "f32res" and epi != "plain"
    sd, bd = (dev_f32(scale), dev_f32(shift)) if scale is not None else (None, None)
    e = twn.epilogue(sd, bd, res, relu, twn.BF16 if bf16 else twn.F32, twn.RESIDUAL_GATE if epi == "gate" else twn.RESIDUAL_ADD)
    Y = torch.full(shape, float("nan"), dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    (twn.conv2d_fwd if bits == 2 else twn.conv2d_fwd_b1)(d, dev_bf16(X), packed, ld, None, e, Y, status)
    assert twn.read_status(status) == 0
    gate = epi == "gate"
    want, A = oracle.conv2d_fwd(od, X, codes.reshape(Cout, k, k, Cin), 1.0, scale, shift, None if gate else res_host, relu)
    want = np.asarray(want).reshape(shape)
    if gate:
        want = np.where(res_host > 0, want, 0.0)
    tol = 1e-4 * np.asarray(A).reshape(shape) * (np.abs(scale) if scale is not None else 1.0) + 1e-6
    got = Y.float().cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - want) <= tol + (2.0 ** -8 * (np.abs(want) + tol) if bf16 else 0.0))
