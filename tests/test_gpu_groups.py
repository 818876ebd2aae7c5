"""Layers of more than 64 output channels whose short reductions run in the resident-weight kernel, 64 channels per block:
the last group full, one channel above the first, short of half; every epilogue; both output types; backward for data."""
import pytest

import test_gpu_narrow as narrow

pytestmark = pytest.mark.gpu


# enough pixel tiles for that kernel to be the choice
@pytest.mark.parametrize("case", [
    (40, 28, 28, 16, 136, 1, 0, None, True, True, False),
    (24, 56, 50, 32, 72, 3, 1, "add", True, True, True),
    (24, 40, 40, 16, 200, 3, 1, "gate", False, True, True),
    (30, 33, 31, 64, 128, 1, 0, "add", True, True, False),
    (30, 33, 31, 16, 96, 1, 0, None, False, False, True),
    (100, 16, 16, 32, 352, 3, 1, None, True, True, False),
])
def test_forward(case):
    narrow.test_narrow_conv_fwd_matches_oracle(case)


@pytest.mark.parametrize("case", [(24, 40, 44, 72, 32, 3, 1, 1, "add", True), (30, 34, 34, 256, 64, 1, 1, 0, "gate", True),
                                  (24, 56, 56, 128, 64, 1, 2, 0, "add", True)])
def test_bwd_data(case):
    narrow.test_narrow_conv_bwd_data_matches_oracle(case)


@pytest.mark.parametrize("M,N,K,out_bf16", [(14705, 960, 176, False), (40001, 72, 64, False), (16385, 1032, 64, True)])
def test_gemm(M, N, K, out_bf16):
    narrow.test_narrow_gemm_matches_oracle(M, N, K, out_bf16)
