"""Buffers and parameters of a network may be replaced between passes: the next pass uses the new ones, also those whose
addresses a prepared call holds."""
import copy
import gc
import weakref

import pytest
import torch

from paper_1605_04711_b200 import nets

pytestmark = pytest.mark.gpu


def results(net):
    out = {"logits": net.act[net.ops[-1][1].name].clone()}
    if net.train:
        out.update({n: L.extra["dW"].clone() for n, L in net.layers.items()})
    return out


def replace_and_poison(holder, key, value):
    """A copy takes the tensor's place; the old one is filled with what would show in any result."""
    old = value
    new = old.clone()
    if isinstance(holder, dict):
        holder[key] = new
    else:
        setattr(holder, key, new)
    old.view(torch.uint8).fill_(0xFF)
    return old


def vgg7_of_16_classes():
    ops = nets.vgg7_ops()
    ops[-1][1].Cout = 16                 # gradients of 10 logits have no 16-byte rows
    return nets.TernaryNet("vgg7", 5, (32, 32, 3), ops, train=True)


MAKE = {"resnet18_train": lambda: nets.resnet18(batch=3, train=True, image=64, classes=40), "vgg7_train": vgg7_of_16_classes,
        "lenet5": lambda: nets.lenet5(batch=7)}


@pytest.mark.parametrize("which", list(MAKE))
def test_every_tensor_may_be_replaced(which):
    net, train = MAKE[which](), which.endswith("train")
    g = torch.Generator(device="cuda").manual_seed(3)
    net.act["input"].normal_(generator=g)
    last = net.ops[-1][1]
    dl = torch.randn(last.B, last.Cout, device="cuda", generator=g).mul_(0.01).bfloat16()

    def step():
        if train:
            net.train_step(dl)
        else:
            net.ternarize_all()
            net.forward()
        torch.cuda.synchronize()
        return results(net)

    want = step()
    assert all(torch.equal(v, want[k]) for k, v in step().items())
    flat = [op[1] for op in net.ops if op[0] == "flatten"]          # views of another activation, made by the network
    old = []
    for holder in [net.act, net.aux, net.grad] + [L.extra for L in net.layers.values()]:
        for k, v in list(holder.items()):
            if isinstance(v, torch.Tensor) and not (holder is net.act and k in flat):
                old.append(replace_and_poison(holder, k, v))
    for k in ("status", "ws_tern") + (("ws_dw",) if train else ()):
        old.append(replace_and_poison(net, k, getattr(net, k)))
    got = step()
    for k, v in want.items():
        assert torch.equal(got[k], v), k
    for t in old:
        assert bool((t.view(torch.uint8) == 0xFF).all())           # nothing was written there


def test_other_changes_count_as_well():
    net = nets.lenet5(batch=2)
    net.act["input"].normal_()
    net.ternarize_all()
    net.forward()
    calls = net._fwd[1]
    net.forward()
    assert net._fwd[1] is calls
    conv1 = net.layers["conv1"]
    for change in (lambda: net.act.update(pool1=net.act["pool1"].clone()), lambda: setattr(net, "act", dict(net.act)),
                   lambda: setattr(conv1, "extra", dict(conv1.extra)), lambda: net.act.__setitem__("pool1", net.act.pop("pool1"))):
        before = net._fwd[1]
        change()
        net.forward()
        assert net._fwd[1] is not before
    assert type(copy.deepcopy(conv1.extra["packed"])) is torch.Tensor and type(copy.copy(net.act)) is dict
    torch.cuda.synchronize()
    gone = weakref.ref(net)
    gc.disable()
    try:
        del net, conv1, change, before, calls
        assert gone() is None            # no cycle keeps its memory
    finally:
        gc.enable()
