"""Python binding of libtwn.so: the same entry points as include/twn.h.

Argument marshalling only: the compute calls go through the native module _twn (csrc/binding.cpp), the size
queries and the status read-back through ctypes.  Tensors are torch tensors on the current CUDA
device (torch provides memory and streams); every step of the computation runs
in the library's kernels.  There is no fallback: if the library is missing or
the device is not sm_100 the calls raise.
"""
from __future__ import annotations

import ctypes as C
import os

import torch

try:
    from . import _twn as _C
except ImportError as e:
    class _Missing:
        """Stands in for the native module where it is not built: every call says so."""
        reason = str(e)

        def __getattr__(self, name):
            raise FileNotFoundError(f"the native binding does not load ({self.reason}): build it with "
                                    "`python -m paper_1605_04711_b200.build`")
    _C = _Missing()

_PKG = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_PKG, "libtwn.so")

OK = 0
F32, BF16 = 0, 1
STATS_BYTES = 64


class TwnError(RuntimeError):
    def __init__(self, code: int, where: str):
        self.code = code
        super().__init__(f"{where}: {strerror(code)} ({code})")


class ConvDesc(C.Structure):
    _fields_ = [("B", C.c_int64), ("H", C.c_int64), ("W", C.c_int64), ("Cin", C.c_int64),
                ("Cout", C.c_int64), ("kh", C.c_int32), ("kw", C.c_int32),
                ("stride_h", C.c_int32), ("stride_w", C.c_int32),
                ("pad_h", C.c_int32), ("pad_w", C.c_int32)]

    @property
    def Ho(self):
        return (self.H + 2 * self.pad_h - self.kh) // self.stride_h + 1

    @property
    def Wo(self):
        return (self.W + 2 * self.pad_w - self.kw) // self.stride_w + 1


def conv_desc(B, H, W, Cin, Cout, k, stride=1, pad=0) -> ConvDesc:
    kh, kw = (k, k) if isinstance(k, int) else k
    return ConvDesc(B, H, W, Cin, Cout, kh, kw, stride, stride, pad, pad)


class Epilogue(C.Structure):
    _fields_ = [("scale", C.c_void_p), ("shift", C.c_void_p), ("residual", C.c_void_p),
                ("residual_dtype", C.c_int32), ("relu", C.c_int32), ("out_dtype", C.c_int32),
                ("residual_op", C.c_int32)]


_lib = None


def lib() -> C.CDLL:
    """Opens libtwn.so (built by paper_1605_04711_b200/build.py).  Raises if absent."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise FileNotFoundError(
                f"{LIB_PATH} not found: build it with `python -m paper_1605_04711_b200.build`")
        l = C.CDLL(LIB_PATH)
        l.twn_strerror.restype = C.c_char_p
        l.twn_ternarize_workspace_bytes.restype = C.c_size_t
        l.twn_ternarize_batch_workspace_bytes.restype = C.c_size_t
        l.twn_conv2d_bwd_weight_workspace_bytes.restype = C.c_size_t
        l.twn_conv2d_bwd_weight_folded_workspace_bytes.restype = C.c_size_t
        l.twn_binarize_workspace_bytes.restype = C.c_size_t
        l.twn_conv2d_fwd_bn_workspace_bytes.restype = C.c_size_t
        _lib = l
    return _lib


def strerror(code: int) -> str:
    return lib().twn_strerror(C.c_int(code)).decode()


def _check(code: int, where: str) -> None:
    if code != OK:
        raise TwnError(code, where)


def _ptr(t) -> C.c_void_p:
    if t is None:
        return C.c_void_p(0)
    assert t.is_cuda and t.is_contiguous(), "device tensors must be contiguous CUDA tensors"
    return C.c_void_p(t.data_ptr())


def _stream(stream=None) -> C.c_void_p:
    s = torch.cuda.current_stream() if stream is None else stream
    return C.c_void_p(s.cuda_stream)


def ld_for(cols: int) -> int:
    """Smallest legal row pitch (in codes) for rows of `cols` codes."""
    return (cols + 63) // 64 * 64


def new_stats(device="cuda") -> torch.Tensor:
    """A zeroed device twn_stats_t (64 bytes, as 8 int64 words)."""
    return torch.zeros(8, dtype=torch.int64, device=device)


def stats_to_host(stats: torch.Tensor) -> dict:
    """Synchronises and decodes a device twn_stats_t."""
    h = stats.cpu()
    d = h.view(torch.float64)
    return {"delta": float(d[0]), "alpha": float(d[1]), "sum_abs": float(d[2]),
            "sum_abs_kept": float(d[3]), "n_neg": int(h[4]), "n_zero": int(h[5]),
            "n_pos": int(h[6]), "status": int(h.view(torch.int32)[14])}


def read_status(dev_status: torch.Tensor, stream=None) -> int:
    out = C.c_int32(0)
    _check(lib().twn_read_status(_ptr(dev_status), C.byref(out), _stream(stream)), "twn_read_status")
    return out.value


def ternarize_workspace_bytes() -> int:
    return int(lib().twn_ternarize_workspace_bytes())


def ternarize(W: torch.Tensor, delta_factor: float, stats: torch.Tensor, packed: torch.Tensor,
              ld_codes: int, codes_i8, workspace: torch.Tensor, stream=None,
              rows: int | None = None, cols: int | None = None) -> None:
    """twn_ternarize.  W fp32 [rows, cols] (or any shape with rows/cols given)."""
    if rows is None:
        rows, cols = (W.shape[0], W.numel() // W.shape[0]) if W.dim() > 1 else (1, W.numel())
    _check(_C.ternarize(W, rows, cols, delta_factor, stats, packed, ld_codes, codes_i8, workspace, stream),
           "twn_ternarize")


def sgd_update(W: torch.Tensor, dW: torch.Tensor, V: torch.Tensor, lr: float, momentum: float,
               weight_decay: float, delta_factor: float, stats_next, workspace: torch.Tensor, stream=None) -> None:
    """twn_sgd_update: in-place SGD step on the fp32 master weights; stats_next (optional) receives
    the threshold of the updated weights."""
    _check(_C.sgd_update(W, dW, V, W.numel(), lr, momentum, weight_decay, delta_factor, stats_next, workspace, stream),
           "twn_sgd_update")


def ternarize_codes(W: torch.Tensor, rows: int, cols: int, stats: torch.Tensor, packed: torch.Tensor,
                    ld_codes: int, codes_i8, workspace: torch.Tensor, stream=None) -> None:
    """twn_ternarize_codes: the coding sweep alone, against the threshold already in `stats`."""
    _check(_C.ternarize_codes(W, rows, cols, stats, packed, ld_codes, codes_i8, workspace, stream),
           "twn_ternarize_codes")


def ternarize_batch_workspace_bytes(count: int) -> int:
    return int(lib().twn_ternarize_batch_workspace_bytes(C.c_int(count)))


def ternarize_batch(items, delta_factor: float, workspace: torch.Tensor, stream=None) -> None:
    """twn_ternarize_batch.  items: list of (W, rows, cols, stats, packed, ld_codes, codes_i8 or None)."""
    _check(_C.ternarize_batch(items, delta_factor, workspace, stream), "twn_ternarize_batch")


def sgd_update_batch(items, lr: float, momentum: float, weight_decay: float, delta_factor: float,
                     workspace: torch.Tensor, stream=None) -> None:
    """twn_sgd_update_batch.  items: list of (W, dW, V, stats_next or None)."""
    _check(_C.sgd_update_batch(items, lr, momentum, weight_decay, delta_factor, workspace, stream),
           "twn_sgd_update_batch")


def ternarize_codes_batch(items, workspace: torch.Tensor, stream=None) -> None:
    """twn_ternarize_codes_batch.  items as for ternarize_batch; every stats holds its threshold already."""
    _check(_C.ternarize_codes_batch(items, workspace, stream), "twn_ternarize_codes_batch")


def transpose_codes_batch(items, stream=None) -> None:
    """twn_transpose_codes_batch.  items: list of (packed_fwd, ld_fwd, desc, packed_bwd, ld_bwd)."""
    _check(_C.transpose_codes_batch(items, stream), "twn_transpose_codes_batch")


def ternarize_rows(W: torch.Tensor, delta_factor: float, stats: torch.Tensor, packed: torch.Tensor,
                   ld_codes: int, codes_i8=None, stream=None) -> None:
    """twn_ternarize_rows: one threshold and one scale per filter.  W fp32 [rows, cols];
    stats int64 [rows, 8] (one twn_stats_t per row)."""
    rows, cols = W.shape[0], W.numel() // max(W.shape[0], 1)
    assert stats.numel() * stats.element_size() >= 64 * rows
    _check(_C.ternarize_rows(W, rows, cols, delta_factor, stats, packed, ld_codes, codes_i8, stream),
           "twn_ternarize_rows")


def rows_scale(stats: torch.Tensor, rows: int, scale_in, scale_out: torch.Tensor, dev_status=None,
               stream=None) -> None:
    """twn_rows_scale: scale_out[r] = alpha_r * scale_in[r]."""
    _check(_C.rows_scale(stats, rows, scale_in, scale_out, dev_status, stream), "twn_rows_scale")


def new_stats_rows(rows: int, device="cuda") -> torch.Tensor:
    """Zeroed device array of `rows` twn_stats_t."""
    return torch.zeros((rows, 8), dtype=torch.int64, device=device)


def stats_rows_to_host(stats: torch.Tensor) -> list:
    h = stats.cpu().contiguous()
    d = h.view(torch.float64)
    i32 = h.view(torch.int32)
    return [{"delta": float(d[r, 0]), "alpha": float(d[r, 1]), "sum_abs": float(d[r, 2]),
             "sum_abs_kept": float(d[r, 3]), "n_neg": int(h[r, 4]), "n_zero": int(h[r, 5]),
             "n_pos": int(h[r, 6]), "status": int(i32[r, 14])} for r in range(h.shape[0])]


TERNARIZE_STATIC_MAX_WEIGHTS = 1 << 31


def ternarize_static(W: torch.Tensor, delta_factor: float, stats: torch.Tensor, packed: torch.Tensor,
                     ld_codes: int, codes_i8, stream=None, rows: int | None = None,
                     cols: int | None = None) -> None:
    """twn_ternarize_static: the same ternarization with the scratch held inside the library,
    for callers that cannot allocate device memory.  Calls on one device must not overlap."""
    if rows is None:
        rows, cols = (W.shape[0], W.numel() // W.shape[0]) if W.dim() > 1 else (1, W.numel())
    _check(_C.ternarize_static(W, rows, cols, delta_factor, stats, packed, ld_codes, codes_i8, stream),
           "twn_ternarize_static")


def pack(codes: torch.Tensor, rows: int, cols: int, packed: torch.Tensor, ld_codes: int,
         counts=None, stream=None) -> None:
    _check(_C.pack(codes, rows, cols, packed, ld_codes, counts, stream), "twn_pack")


def unpack(packed: torch.Tensor, rows: int, cols: int, ld_codes: int, codes: torch.Tensor,
           dev_status=None, stream=None) -> None:
    _check(_C.unpack(packed, rows, cols, ld_codes, codes, dev_status, stream), "twn_unpack")


def transpose_codes(packed_fwd: torch.Tensor, ld_fwd: int, desc: ConvDesc, packed_bwd: torch.Tensor,
                    ld_bwd: int, stream=None) -> None:
    _check(_C.transpose_codes(packed_fwd, ld_fwd, desc, packed_bwd, ld_bwd, stream), "twn_transpose_codes")


RESIDUAL_ADD, RESIDUAL_GATE = 0, 1
SUM_IN_ORDER = 2          # or-ed into residual_op


def epilogue(scale=None, shift=None, residual=None, relu=False, out_dtype=F32, residual_op=RESIDUAL_ADD):
    """Builds a twn_epilogue_t; keeps no reference, the caller keeps the tensors alive.

    The sums of a contraction may be split over blocks as its sizes suggest, so an image's outputs can be rounded
    differently in batches of different size; SUM_IN_ORDER in residual_op makes them the same bits in every batch."""
    e = Epilogue(_ptr(scale).value, _ptr(shift).value, _ptr(residual).value,
                 BF16 if (residual is not None and residual.dtype == torch.bfloat16) else F32,
                 int(bool(relu)), out_dtype, residual_op)
    return e


def gemm(X: torch.Tensor, ldx: int, T_packed: torch.Tensor, ld_codes: int, stats, M: int, N: int,
         K: int, epi, Y: torch.Tensor, ldy: int, dev_status=None, stream=None) -> None:
    _check(_C.gemm(X, ldx, T_packed, ld_codes, stats, M, N, K, epi, Y, ldy, dev_status, stream), "twn_gemm")


def conv2d_fwd(desc: ConvDesc, X: torch.Tensor, T_fwd: torch.Tensor, ld_codes: int, stats, epi,
               Y: torch.Tensor, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_fwd(desc, X, T_fwd, ld_codes, stats, epi, Y, dev_status, stream), "twn_conv2d_fwd")


def conv2d_fwd_maxpool(desc: ConvDesc, X: torch.Tensor, T_fwd: torch.Tensor, ld_codes: int, stats, epi,
                       Y: torch.Tensor, Yp: torch.Tensor, dev_status=None, stream=None) -> None:
    """conv2d_fwd, and the 2x2 max pooling of its output into Yp (inference)."""
    _check(_C.conv2d_fwd_maxpool(desc, X, T_fwd, ld_codes, stats, epi, Y, Yp, dev_status, stream), "twn_conv2d_fwd_maxpool")


def conv2d_fwd_bn_workspace_bytes(desc: ConvDesc) -> int:
    return int(lib().twn_conv2d_fwd_bn_workspace_bytes(C.byref(desc)))


def conv2d_fwd_bn(desc: ConvDesc, X: torch.Tensor, T_fwd: torch.Tensor, ld_codes: int, stats, epi, Y: torch.Tensor,
                  bn_sum: torch.Tensor, bn_sumsq: torch.Tensor, workspace: torch.Tensor, dev_status=None,
                  stream=None) -> None:
    _check(_C.conv2d_fwd_bn(desc, X, T_fwd, ld_codes, stats, epi, Y, bn_sum, bn_sumsq, workspace, dev_status, stream),
           "twn_conv2d_fwd_bn")


def bn_finalize(bn_sum: torch.Tensor, bn_sumsq: torch.Tensor, n: int, C_: int, gamma, beta, eps: float, scale, shift,
                mean=None, var=None, stream=None) -> None:
    _check(_C.bn_finalize(bn_sum, bn_sumsq, n, C_, gamma, beta, eps, scale, shift, mean, var, stream),
           "twn_bn_finalize")


def conv2d_bwd_data(desc: ConvDesc, dZ: torch.Tensor, T_bwd: torch.Tensor, ld_codes: int, stats, epi,
                    dX: torch.Tensor, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_bwd_data(desc, dZ, T_bwd, ld_codes, stats, epi, dX, dev_status, stream), "twn_conv2d_bwd_data")


# ---- binary precision weights: the same calls on 1-bit codes
def ld_for_b1(cols: int) -> int:
    """Smallest legal row pitch (in codes) for 1-bit rows of `cols` codes."""
    return (cols + 127) // 128 * 128


def binarize_workspace_bytes() -> int:
    return int(lib().twn_binarize_workspace_bytes())


def binarize(W: torch.Tensor, stats: torch.Tensor, packed: torch.Tensor, ld_codes: int, workspace: torch.Tensor,
             stream=None, rows: int | None = None, cols: int | None = None) -> None:
    if rows is None:
        rows, cols = (W.shape[0], W.numel() // W.shape[0]) if W.dim() > 1 else (1, W.numel())
    _check(_C.binarize(W, rows, cols, stats, packed, ld_codes, workspace, stream), "twn_binarize")


def unpack_b1(packed: torch.Tensor, rows: int, cols: int, ld_codes: int, codes: torch.Tensor, stream=None) -> None:
    _check(_C.unpack_b1(packed, rows, cols, ld_codes, codes, stream), "twn_unpack_b1")


def transpose_codes_b1(packed_fwd: torch.Tensor, ld_fwd: int, desc: ConvDesc, packed_bwd: torch.Tensor, ld_bwd: int,
                       stream=None) -> None:
    _check(_C.transpose_codes_b1(packed_fwd, ld_fwd, desc, packed_bwd, ld_bwd, stream), "twn_transpose_codes_b1")


def gemm_b1(X: torch.Tensor, ldx: int, B_packed: torch.Tensor, ld_codes: int, stats, M: int, N: int,
            K: int, epi, Y: torch.Tensor, ldy: int, dev_status=None, stream=None) -> None:
    _check(_C.gemm_b1(X, ldx, B_packed, ld_codes, stats, M, N, K, epi, Y, ldy, dev_status, stream), "twn_gemm_b1")


def conv2d_fwd_b1(desc: ConvDesc, X: torch.Tensor, B_fwd: torch.Tensor, ld_codes: int, stats, epi,
                  Y: torch.Tensor, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_fwd_b1(desc, X, B_fwd, ld_codes, stats, epi, Y, dev_status, stream), "twn_conv2d_fwd_b1")


def conv2d_bwd_data_b1(desc: ConvDesc, dZ: torch.Tensor, B_bwd: torch.Tensor, ld_codes: int, stats, epi,
                       dX: torch.Tensor, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_bwd_data_b1(desc, dZ, B_bwd, ld_codes, stats, epi, dX, dev_status, stream),
           "twn_conv2d_bwd_data_b1")


def im2col(desc: ConvDesc, X: torch.Tensor, Xcol: torch.Tensor, ldk: int, stream=None) -> None:
    _check(_C.im2col(desc, X, Xcol, ldk, stream), "twn_im2col")


def conv2d_fwd_image(desc: ConvDesc, X: torch.Tensor, T_fwd: torch.Tensor, ld_codes: int, stats, epi, Y: torch.Tensor, Yp=None,
                     stream=None) -> None:
    _check(_C.conv2d_fwd_image(desc, X, T_fwd, ld_codes, stats, epi, Y, Yp, stream), "twn_conv2d_fwd_image")


def fold_dims(desc: ConvDesc):
    """(Hf, Wf, ldf) of the folded form of a stride-2 layer with few channels, or None if the
    layer cannot be folded."""
    hf, wf, ldf = C.c_int64(0), C.c_int64(0), C.c_int64(0)
    rc = lib().twn_fold_dims(C.byref(desc), C.byref(hf), C.byref(wf), C.byref(ldf))
    return (hf.value, wf.value, ldf.value) if rc == 0 else None


def fold_input(desc: ConvDesc, X, Xf, stream=None) -> None:
    _check(_C.fold_input(desc, X, Xf, stream), "twn_fold_input")


def fold_codes(desc: ConvDesc, packed, ld_codes: int, packed_folded, ld_folded: int, stream=None) -> None:
    _check(_C.fold_codes(desc, packed, ld_codes, packed_folded, ld_folded, stream), "twn_fold_codes")


def conv2d_fwd_folded(desc: ConvDesc, Xf, Tf, ld_folded: int, stats, epi, Y, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_fwd_folded(desc, Xf, Tf, ld_folded, stats, epi, Y, dev_status, stream), "twn_conv2d_fwd_folded")


def conv2d_bwd_weight_folded_workspace_bytes(desc: ConvDesc) -> int:
    return int(lib().twn_conv2d_bwd_weight_folded_workspace_bytes(C.byref(desc)))


def conv2d_bwd_weight_folded(desc: ConvDesc, Xf, dZ, dW, workspace, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_bwd_weight_folded(desc, Xf, dZ, dW, workspace, dev_status, stream), "twn_conv2d_bwd_weight_folded")


def maxpool2d_fwd(X, B, H, W, Cc, k, stride, pad, Y, argmax=None, stream=None) -> None:
    _check(_C.maxpool2d_fwd(X, B, H, W, Cc, k, stride, pad, Y, argmax, stream), "twn_maxpool2d_fwd")


def maxpool2d_bwd(dY, argmax, B, H, W, Cc, k, stride, pad, dX, stream=None) -> None:
    _check(_C.maxpool2d_bwd(dY, argmax, B, H, W, Cc, k, stride, pad, dX, stream), "twn_maxpool2d_bwd")


def maxpool2d_bwd_act(dY, argmax, pooled, scale, B, H, W, Cc, k, stride, pad, dZ, stream=None) -> None:
    _check(_C.maxpool2d_bwd_act(dY, argmax, pooled, scale, B, H, W, Cc, k, stride, pad, dZ, stream),
           "twn_maxpool2d_bwd_act")


def avgpool_fwd(X, B, HW, Cc, Y, stream=None) -> None:
    _check(_C.avgpool_fwd(X, B, HW, Cc, Y, stream), "twn_avgpool_fwd")


def avgpool_bwd(dY, B, HW, Cc, dX, stream=None) -> None:
    _check(_C.avgpool_bwd(dY, B, HW, Cc, dX, stream), "twn_avgpool_bwd")


def act_bwd(dY, Y, scale, n, Cc, dZ, dPre=None, stream=None) -> None:
    _check(_C.act_bwd(dY, Y, scale, n, Cc, dZ, dPre, stream), "twn_act_bwd")


def conv2d_bwd_weight_workspace_bytes(desc: ConvDesc) -> int:
    return int(lib().twn_conv2d_bwd_weight_workspace_bytes(C.byref(desc)))


def conv2d_bwd_weight(desc: ConvDesc, X, dZ, dW, workspace, dev_status=None, stream=None) -> None:
    _check(_C.conv2d_bwd_weight(desc, X, dZ, dW, workspace, dev_status, stream), "twn_conv2d_bwd_weight")
