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


def test_another_tensor_for_the_logits(net):
    x = _x(11)
    want, own = net.forward(x).clone(), net.buf["logits"]
    mine = torch.full_like(own, 7.0)
    net.buf["logits"] = mine
    try:
        for _ in range(2):
            mine.fill_(7.0)
            assert net.forward(x) is mine and torch.equal(mine, want)
    finally:
        net.buf["logits"] = own
    own.fill_(7.0)
    for _ in range(2):
        assert net.forward(x) is own and torch.equal(own, want)


def test_a_parameter_with_other_memory():
    x, net = _x(13), Resnet50Chain(2, torch.device("cuda:0"), seed=5)
    W, B = net.params["fc"]
    want = net.forward(x) - B
    for value, rebind in ((1.0, lambda t: setattr(B, "data", t)), (2.0, lambda t: B.set_(t)), (3.0, lambda t: B.resize_(1 << 20).resize_(1000).copy_(t))):
        rebind(torch.full((1 << 16,), value, device="cuda")[:1000])
        assert torch.allclose(net.forward(x), want + value, rtol=1e-5, atol=1e-5)
    net.close()


def test_pins_set_after_the_chain_was_built(net, monkeypatch):
    x = _x(15)
    want = net.forward(x).clone()
    binding.set_kernel_override("simt_direct")             # (the head's Gemm in fp32)
    try:
        got, one_by_one = net.forward(x).clone(), _one_by_one(net, x)
    finally:
        binding.set_kernel_override(None)
    assert torch.equal(got, one_by_one) and not torch.equal(got, want)
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", "0")
    launches = binding.launch_count()
    net.forward(x)
    assert binding.launch_count() - launches > 50
    monkeypatch.delenv("ONNXB_GEMM_SPLITK")
    launches = binding.launch_count()
    assert torch.equal(net.forward(x), want) and binding.launch_count() - launches == 1


def test_on_another_current_device(net, monkeypatch):
    x = _x(17)
    want, launches = net.forward(x).clone(), binding.launch_count()
    monkeypatch.setattr(net, "_device", net._device + 1)
    assert torch.equal(net.forward(x), want) and binding.launch_count() - launches == net.launches


@pytest.mark.parametrize("prepack", [True, False])
def test_another_tensor_inside_the_graph(prepack):
    """The tensors that the operators write are the graph's as ONNX has it: whole ones also where the chain moved a stride up."""
    x, given = _x(19), ("r50_08_s2b2_b", "r50_08_s2b2_out", "stem", "pooled")
    other, net = (Resnet50Chain(2, torch.device("cuda:0"), seed=5, prepack=p) for p in (False, prepack))
    want = other.forward(x)
    assert set(given) <= set(other.buf)
    near = net.forward(x).clone()
    for name in given:
        net.buf[name] = torch.full_like(other.buf[name], 7.0)
    mine = {name: net.buf[name] for name in given}
    if prepack:
        with pytest.raises(RuntimeError, match="outside a capture"):
            with torch.cuda.graph(torch.cuda.CUDAGraph()):
                mine["stem"].zero_()                       # (a graph of nothing draws a warning)
                net.forward(x)
    for _ in range(2):
        assert torch.equal(net.forward(x), want)
    for op in other.ops:
        assert torch.equal(net.buf[op.dst], other.buf[op.dst]), op.name
    assert all(net.buf[name] is mine[name] for name in given) and torch.allclose(near, want, rtol=0, atol=2e-2 * float(want.std()))
    net.close()
    other.close()


def test_prepack_switched_off():
    x = _x(21)
    other, net = (Resnet50Chain(2, torch.device("cuda:0"), seed=5, prepack=p) for p in (False, True))
    net.forward(x)
    net.prepack = False
    for n in (other, net):
        for W, _ in n.params.values():
            W.mul_(0.9)
    assert torch.equal(net.forward(x), other.forward(x))
    net.close()
    other.close()


def test_the_state_compared(monkeypatch):
    a, b = torch.empty(6, 4, device="cuda"), torch.empty(6, 4, device="cuda")
    plain = binding.call_state({"x": a, "input": b}, (a, b), b)
    assert plain == binding.call_state({"x": a, "input": a}, (a, b), b) == binding.call_state({"x": a}, (a, b), b)
    others = [binding.call_state({"x": t}, (a, u), b) for t, u in ((b, b), (a, a), (a.view(4, 6), b), (a[:, :2], b), (a.t(), b), (a.view(torch.int32), b))]
    assert len({plain, *others, binding.call_state({"x": a}, (a, b)), binding.call_state({"x": a, "y": b}, (a, b), b)}) == 9
    monkeypatch.setenv("ONNXB_GEMM_BN", "64")
    assert plain != binding.call_state({"x": a}, (a, b), b)
    assert binding.call_state([a]) is None and binding.call_state({"x": None}) is None


def test_laid_out_anew_on_another_stream():
    """While a pass on the first stream may still run, whose buffers go back to that stream's allocations."""
    x, net = _x(23), Resnet50Chain(2, torch.device("cuda:0"), seed=5)
    want, side = net.forward(x).clone(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for _ in range(20):
        net.forward(x)
    net.buf["stem"] = torch.empty(2, 64, 112, 112, device="cuda")
    with torch.cuda.stream(side):
        got = net.forward(x)
    torch.cuda.current_stream().wait_stream(side)
    assert torch.allclose(got, want, rtol=0, atol=2e-2 * float(want.std())) and binding.last_device_status() == 0
    net.close()
