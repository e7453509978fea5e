"""The chained model as one graph behind its first operator: the same logits, whatever the input's buffer, its stream and the call
around it, and the operators themselves where the graph cannot stand for them."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2008_08272_b200 import binding  # noqa: E402
from paper_2008_08272_b200.resnet50_chain import Resnet50Chain  # noqa: E402


@pytest.fixture(scope="module")
def net():
    n = Resnet50Chain(2, torch.device("cuda:0"), seed=5)
    yield n
    n.close()


def _one_by_one(net, x):
    net.buf["input"] = net.store["input"] = x
    net._run(net.ops)
    return net.buf["logits"].clone()


def _x(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(2, 3, 224, 224, generator=g, device="cuda")


def test_other_inputs_and_streams(net):
    assert net._graph is not None and net.launches > 50
    side = torch.cuda.Stream()
    for seed in range(3):
        x = _x(seed)
        want = _one_by_one(net, x)
        before = binding.launch_count()
        assert torch.equal(net.forward(x), want) and binding.launch_count() - before <= 1
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            net.buf["logits"].zero_()
            got = net.forward(x)
        torch.cuda.current_stream().wait_stream(side)
        assert torch.equal(got, want)
    assert binding.last_device_status() == 0


def test_back_to_back_passes(net):
    xs = [_x(s) for s in range(4)]
    want = [_one_by_one(net, x) for x in xs]
    got = [net.forward(x).clone() for x in xs]
    assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_inside_a_capture(net):
    x, want = _x(7), _one_by_one(net, _x(7))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.forward(x)
    net.buf["logits"].zero_()
    graph.replay()
    assert torch.equal(net.buf["logits"], want)


def test_a_tensor_in_another_s_place(net):
    x = _x(9)
    W, B = net.params["fc"]
    want = net.forward(x).clone()
    net.params["fc"] = (W, B + 1.0)
    try:
        assert torch.allclose(net.forward(x), want + 1.0, rtol=1e-5, atol=1e-5)
    finally:
        net.params["fc"] = (W, B)
    assert torch.equal(net.forward(x), want)
