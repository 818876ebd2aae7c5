"""A NaN stays a NaN through the ReLU of the epilogue, in every kernel and output type (as y < 0 ? 0 : y leaves it)."""
import pytest
import torch

from paper_1605_04711_b200 import twn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("M,K,N", [
    (70, 1024, 96),          # split kernel
    (30000, 64, 64),         # resident weights
    (30000, 1024, 512),      # general kernel
    (30000, 1024, 509),      # general kernel, outputs that TMA cannot store
])
def test_nan_through_relu(M, K, N, dtype):
    codes = torch.ones((N, K), dtype=torch.int8, device="cuda")
    ld = twn.ld_for(K)
    packed = torch.zeros((N, ld // 16), dtype=torch.int32, device="cuda")
    twn.pack(codes, N, K, packed, ld)
    X = torch.full((M, K), -1.0, dtype=torch.bfloat16, device="cuda")
    rows = torch.tensor([0, 33, M - 1], device="cuda")
    X[rows, 5] = float("nan")
    Y = torch.full((M, N), 7.0, dtype=dtype, device="cuda")
    twn.gemm(X, K, packed, ld, None, M, N, K, twn.epilogue(relu=True, out_dtype=twn.F32 if dtype == torch.float32 else twn.BF16), Y, N)
    assert Y[rows].isnan().all()
    keep = torch.ones(M, dtype=torch.bool, device="cuda")
    keep[rows] = False
    assert (Y[keep] == 0).all()
