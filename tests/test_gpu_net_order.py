"""The passes of a training step called one by one, with the codes' side stream joined first or not, directly and as a captured
graph: the bits of train_step."""
import pytest
import torch

from paper_1605_04711_b200 import nets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("join", [False, True])
def test_passes_one_by_one(join, captured):
    net = nets.resnet18(batch=2, train=True, image=64, classes=24)
    g = torch.Generator(device="cuda").manual_seed(1)
    net.act["input"].normal_(generator=g)
    dl = torch.randn(2, 24, device="cuda", generator=g).mul_(0.01).bfloat16()
    net.train_step(dl)
    torch.cuda.synchronize()
    want = {n: L.extra["dW"].clone() for n, L in net.layers.items()}

    def step():
        net.ternarize_all(join=join)
        net.forward()
        net.backward(dl)
        net.join_side_streams()

    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
    for L in net.layers.values():
        L.extra["dW"].fill_(float("nan"))
    graph.replay() if captured else step()
    torch.cuda.synchronize()
    for n, w in want.items():
        assert torch.equal(net.layers[n].extra["dW"], w), n
