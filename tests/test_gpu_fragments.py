"""The general contraction's bf16 epilogue, which drains the accumulator as matrix fragments: channels that end eight past a
warp's thirty-two or a tile's 128, ragged pixels, residual, gate, ReLU, all three tile shapes, strided backward for data."""
import pytest

import test_gpu_narrow as narrow

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [
    (32, 28, 28, 128, 136, 3, 1, "add", True, True, True),
    (64, 14, 13, 192, 264, 3, 1, "gate", False, True, True),
    (128, 8, 8, 256, 488, 3, 1, None, True, True, True),
    (100, 15, 15, 576, 168, 1, 0, "add", True, False, True),
    (33, 31, 29, 320, 200, 3, 1, None, False, False, True),
])
def test_forward(case):
    narrow.test_narrow_conv_fwd_matches_oracle(case)


@pytest.mark.parametrize("case", [(32, 28, 28, 136, 256, 3, 1, 1, "add", True), (64, 28, 28, 200, 256, 3, 2, 1, "gate", True)])
def test_bwd_data(case):
    narrow.test_narrow_conv_bwd_data_matches_oracle(case)


@pytest.mark.parametrize("M,N,K", [(16385, 520, 1024), (30001, 152, 2048)])
def test_gemm(M, N, K):
    narrow.test_narrow_gemm_matches_oracle(M, N, K, True)
