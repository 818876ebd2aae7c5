"""The epilogue of a network's first layer belongs to its caller as well: with a residual or the order of the sums written into it, the
layer is the product over the patch matrix to the bit; with the network's own it is one launch from the image."""
import pytest
import torch

from paper_1605_04711_b200 import nets, twn
from _gpu_util import kernel_launches

pytestmark = pytest.mark.gpu


def network(which, batch):
    net = getattr(nets, which)(batch=batch)
    g = torch.Generator(device="cuda")
    g.manual_seed(batch)
    net.act["input"].copy_(torch.randn(net.act["input"].shape, generator=g, device="cuda"))
    net.ternarize_all()
    return net, g


# launches that the product takes beside its own: the patch matrix, and the pooling of LeNet-5
@pytest.mark.parametrize("which,batch,more", [("lenet5", 7, 2), ("vgg7", 32, 1)])
@pytest.mark.parametrize("change", ["bf16 residual", "f32 residual", "gate", "order"])
def test_fields_of_the_epilogue(which, batch, more, change):
    net, g = network(which, batch)
    L, y = net.layers["conv1"], net.act["conv1"]
    e, epi = L.extra, L.extra["epi"]
    image = kernel_launches(net.forward)
    assert which != "lenet5" or image == 4               # a launch for each layer
    own = net.forward().clone()
    R = torch.randn(y.shape, generator=g, device="cuda").to(torch.float32 if change == "f32 residual" else torch.bfloat16)
    if change == "order":
        epi.residual_op = twn.SUM_IN_ORDER
    else:
        epi.residual, epi.residual_dtype = R.data_ptr(), twn.F32 if change == "f32 residual" else twn.BF16
        epi.residual_op = twn.RESIDUAL_GATE if change == "gate" else twn.RESIDUAL_ADD
    y.fill_(7.0)
    assert kernel_launches(net.forward) == image + more
    net.forward()
    columns = torch.zeros((y.numel() // L.Cout, L.ldk), dtype=torch.bfloat16, device="cuda")
    want = torch.full_like(y, 7.0)
    twn.im2col(L.desc, net.act["input"], columns, L.ldk)
    twn.gemm(columns, L.ldk, e["packed"], e["ld"], e["stats"], columns.shape[0], L.Cout, L.K, epi, want, L.Cout)
    assert torch.equal(y.view(torch.int16), want.view(torch.int16))
    epi.residual, epi.residual_op = None, twn.RESIDUAL_ADD
    assert kernel_launches(net.forward) == image
    assert torch.equal(net.forward(), own)


def test_refused_by_every_contraction():
    net, _ = network("lenet5", 2)
    epi = net.layers["conv1"].extra["epi"]
    net.forward()
    epi.residual_op = 9
    with pytest.raises(twn.TwnError):
        net.forward()


def test_no_epilogue():
    """None stands for fp32 outputs, which a caller may put in place of a layer's own epilogue with a buffer for them."""
    op = ("layer", nets.Layer("conv", 3, 16, 3, 1, 1, 8, 8, src="input"))
    net = nets.TernaryNet("one", 2, (8, 8, 3), [op])
    net.act["input"].normal_()
    net.ternarize_all()
    net.layers["conv"].extra["epi"] = None
    net.act["conv"] = torch.full((2, 8, 8, 16), 7.0, device="cuda")
    L, y = net.layers["conv"], net.forward()
    columns, want = torch.zeros((128, L.ldk), dtype=torch.bfloat16, device="cuda"), torch.zeros_like(y)
    twn.im2col(L.desc, net.act["input"], columns, L.ldk)
    twn.gemm(columns, L.ldk, L.extra["packed"], L.extra["ld"], L.extra["stats"], 128, 16, 27, None, want, 16)
    assert torch.equal(y, want) and torch.equal(net.forward(), want)
