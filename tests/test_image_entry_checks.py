"""twn_conv2d_fwd_image refuses an epilogue that the other contractions refuse, on the host, before any CUDA call."""
import ctypes as C

import pytest

from paper_1605_04711_b200 import build, twn


@pytest.mark.parametrize("field,value", [("residual_dtype", 7), ("residual_dtype", -1), ("residual_op", 4), ("residual_op", -1), ("relu", 2),
                                         ("out_dtype", 2)])
def test_epilogue(field, value):
    lib, fake = C.CDLL(build.build()), C.c_void_p(4096)          # never dereferenced: a host check comes first
    d = twn.conv_desc(2, 8, 8, 1, 16, 3, 1, 1)
    epi = twn.Epilogue(out_dtype=twn.BF16)
    setattr(epi, field, value)
    size = C.c_int64
    calls = [lib.twn_conv2d_fwd_image(C.byref(d), fake, fake, size(64), None, C.byref(epi), fake, None, None),
             lib.twn_gemm(fake, size(64), fake, size(64), None, size(4), size(8), size(64), C.byref(epi), fake, size(8), None, None)]
    assert calls == [-1, -1]                                     # TWN_ERR_INVALID_ARG
