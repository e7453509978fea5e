"""Calls on a stream of the caller's that is not the current one: what the binding allocates for them is made on that stream, so
that memory given back by the current stream's work is not handed to them early, nor theirs to it."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(params=["native", "ctypes"])
def binding(request, monkeypatch):
    from paper_2008_08272_b200 import binding as b
    b.load(build_if_missing=False)
    if request.param == "ctypes":
        monkeypatch.setattr(b, "_fast_mod", b._Declined())
    return b


def _conv(binding, g, xs, ws, family, prepacked=False, **kw):
    d = binding.Conv2dDesc(xs, ws, **kw)
    assert d.kernel_family == family and d.workspace_bytes > 0
    X, W = torch.rand(xs, generator=g, device="cuda"), torch.randn(ws, generator=g, device="cuda")
    if prepacked:
        return d.workspace_bytes, lambda **on: d.run_prepacked(X, W, d.prepack(W, stream=on.get("stream")), **on)
    return d.workspace_bytes, lambda **on: d.run(X, W, **on)


def _calls(binding):
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    for M, N, K in ((1001, 1530, 777), (512, 768, 640)):                 # fp32 by split operands, TF32
        A, B = torch.randn(M, K, generator=g, device="cuda"), torch.randn(K, N, generator=g, device="cuda")
        yield binding.gemm_workspace_bytes(False, False, M, N, K), lambda **on: binding.onnx_gemm(A, B, **on)
        yield binding.gemm_workspace_bytes(False, False, M, N, K), lambda **on: binding.onnx_matmul_add(A, B, **on)
    yield _conv(binding, g, (4, 96, 75, 61), (192, 48, 3, 3), "simt_direct", pads=(1,) * 4, group=2)
    yield _conv(binding, g, (4, 96, 75, 61), (192, 48, 3, 3), "simt_direct", True, pads=(1,) * 4, group=2)
    yield _conv(binding, g, (4, 64, 28, 28), (96, 64, 3, 3), "mma_implicit", pads=(1,) * 4)
    yield _conv(binding, g, (4, 64, 28, 28), (96, 64, 1, 1), "mma_gather_gemm", True, strides=(2, 2))


def test_memory_is_the_call_s_stream_s(binding):
    side = torch.cuda.Stream()
    for need, call in _calls(binding):
        assert need > 0
        want = call()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        before = {s["address"] for s in torch.cuda.memory_snapshot()}
        got = call(stream=side)
        made = [s for s in torch.cuda.memory_snapshot() if s["address"] not in before]
        assert made and all(s["stream"] == side.cuda_stream for s in made)
        side.synchronize()
        assert torch.equal(got, want)
        del got
    assert binding.last_device_status() == 0


def test_neither_stream_writes_into_the_other_s(binding):
    """Memory that the current stream is still writing when it is given back, and memory of the call's size that it takes and
    writes while the call runs."""
    side = torch.cuda.Stream()
    for need, call in _calls(binding):
        want = call()
        torch.cuda.synchronize()
        y = torch.empty_like(want)
        for _ in range(3):
            given_back = torch.empty(need, dtype=torch.uint8, device="cuda")
            for _ in range(60):
                given_back.fill_(17)
            del given_back
            call(stream=side, Y=y)
            taken = torch.empty(need, dtype=torch.uint8, device="cuda")
            for _ in range(60):
                taken.fill_(17)
            torch.cuda.synchronize()
            assert torch.equal(y, want)
    assert binding.last_device_status() == 0


def test_a_result_is_not_reused_while_the_current_stream_reads_it(binding):
    """A result given back while the current stream still has it to read, and the next one of that size on the call's stream."""
    side = torch.cuda.Stream()
    X = torch.randn(8, 16, 256, 256, device="cuda")
    zero = torch.zeros_like(X)
    pools = lambda x: binding.onnx_maxpool2d(x, (1, 1), stream=side)
    assert torch.equal(pools(X), X)
    torch.cuda.synchronize()
    y = pools(X)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda._sleep(20_000_000)
    kept = y.clone()
    del y
    for _ in range(4):
        pools(zero)
    torch.cuda.synchronize()
    assert torch.equal(kept, X)
