"""Which kernel a strided backward pass takes: the general one where its model is 5 % below the split kernel's and 10 % (35 % where a
class has no taps) below launches apart, although the first launches apart alone already pass the split kernel's time."""
import ctypes

import pytest
import torch

from paper_1605_04711_b200 import twn
from test_gpu_code_loads import packed_codes

pytestmark = pytest.mark.gpu


class _KernelNode(ctypes.Structure):
    """CUDA_KERNEL_NODE_PARAMS_v2"""
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def kernel_names(call):
    """Mangled names of the kernels that one call launches, from a graph that captures it."""
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        call()
    cu, count = ctypes.CDLL("libcuda.so.1"), ctypes.c_size_t()
    handle = ctypes.c_void_p(graph.raw_cuda_graph())
    assert cu.cuGraphGetNodes(handle, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert cu.cuGraphGetNodes(handle, nodes, ctypes.byref(count)) == 0
    names = []
    for node in nodes:
        kind, p, name = ctypes.c_int(), _KernelNode(), ctypes.c_char_p()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value != 0:                      # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
        get, fn = (cu.cuFuncGetName, p.func) if p.func else (cu.cuKernelGetName, p.kern)
        assert get(ctypes.byref(name), ctypes.c_void_p(fn)) == 0
        names.append(name.value.decode())
    return names


@pytest.mark.parametrize("B,H,Cin,Cout,k,kernel", [
    (22, 32, 544, 544, 1, "tconv_kernel"), (33, 18, 448, 768, 1, "tconv_kernel"), (75, 19, 160, 256, 1, "tconv_kernel"),
    (2, 14, 256, 512, 1, "tconv_split_kernel"), (8, 31, 512, 192, 5, "tconv_split_kernel")])
def test_one_launch(B, H, Cin, Cout, k, kernel):
    d = twn.conv_desc(B, H, H, Cin, Cout, k, 2, k // 2)
    T, packed, ld = packed_codes(Cin, k * k * Cout, 2, 0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(B)
    dZ = torch.randn((B, d.Ho, d.Wo, Cout), generator=g, device="cuda").bfloat16()
    dX = torch.full((B, H, H, Cin), 7.0, dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    names = kernel_names(lambda: twn.conv2d_bwd_data(d, dZ, packed, ld, None, twn.epilogue(out_dtype=twn.BF16), dX, status))
    assert len(names) == 1 and kernel in names[0]
    w, z = T.reshape(Cin, k, k, Cout).permute(3, 0, 1, 2), dZ.double().permute(0, 3, 1, 2)
    back = lambda a, b: torch.nn.grad.conv2d_input((B, Cin, H, H), b, a, stride=2, padding=k // 2).permute(0, 2, 3, 1)     # noqa: E731
    want, size = back(z, w), back(z.abs(), w.abs())
    assert twn.read_status(status) == 0
    # half a unit of bf16, and the roundings of 32 bits of a sum of k * k * Cout products in any order
    assert ((dX.double() - want).abs() <= want.abs() * 2.0 ** -8 + size * (k * k * Cout + 3) * 2.0 ** -23).all()
