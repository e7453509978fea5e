"""Where there is no memory for a workspace: the fp32 kernels have a form that needs none, and the call is made with it; the
others raise the allocator's error.  (The limit is the allocator's own, checked on the host.)"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2008_08272_b200 import binding  # noqa: E402


ENOUGH = 20 << 20           # bytes that a call here needs and does not get


@pytest.fixture
def launches_without_memory():
    """launches(call): those of a call for which the allocator has no block of ENOUGH bytes: neither new ones nor, in what it holds,
    parts that earlier tensors have left."""
    def launches(call):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        total, before = torch.cuda.get_device_properties(0).total_memory, binding.launch_count()
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (8 << 20)) / total)
        taken = []
        try:
            with pytest.raises(torch.OutOfMemoryError):
                while True:
                    taken.append(torch.empty(ENOUGH, dtype=torch.uint8, device="cuda"))
            call()
        finally:
            del taken
            torch.cuda.set_per_process_memory_fraction(1.0)
        return binding.launch_count() - before
    return launches


def _same(got, want):
    return float((got - want).norm() / want.norm()) < 1e-5


def test_fp32_gemm(launches_without_memory):
    A, B, Y, want = (torch.randn(s, device="cuda") for s in ((3001, 1001), (1001, 2999), (3001, 2999), (3001, 2999)))
    assert binding.gemm_workspace_bytes(False, False, 3001, 2999, 1001) > ENOUGH
    binding.onnx_gemm(A, B, Y=want)
    for call in (binding.onnx_gemm, binding.onnx_matmul_add):
        assert launches_without_memory(lambda: call(A, B, Y=Y.zero_())) == 1 and _same(Y, want)


@pytest.mark.parametrize("xs,ws,kw", [((16, 2011, 23, 23), (256, 2011, 1, 1), {}), ((1, 768, 33, 33), (768, 768, 3, 3), dict(pads=(1,) * 4))],
                         ids=["packed pixels", "staged"])
def test_fp32_conv(launches_without_memory, xs, ws, kw):
    d = binding.Conv2dDesc(xs, ws, **kw)
    assert d.kernel_family == "simt_direct" and d.workspace_bytes > ENOUGH
    X, W, R, Y, want, added = (torch.randn(s, device="cuda") for s in (xs, ws) + (d.y_shape,) * 4)
    d.run(X, W, Y=want)
    d.run_add(X, W, None, R, Y=added)
    assert launches_without_memory(lambda: d.run(X, W, Y=Y)) == 1 and _same(Y, want)
    assert launches_without_memory(lambda: d.run_add(X, W, None, R, Y=Y)) == 1 and _same(Y, added)
    packed = []
    assert launches_without_memory(lambda: packed.append(d.prepack(W))) == 0 and packed[0].numel() == 16
    assert launches_without_memory(lambda: d.run_prepacked(X, W, packed[0], Y=Y)) == 1 and _same(Y, want)


def test_others_raise(launches_without_memory):
    A, Z = torch.randn(2048, 2048, device="cuda"), torch.empty(2048, 2048, device="cuda")
    d = binding.Conv2dDesc((1, 1024, 32, 32), (1024, 1024, 3, 3))
    X, W, Y = torch.randn(1, 1024, 32, 32, device="cuda"), torch.randn(1024, 1024, 3, 3, device="cuda"), torch.empty(d.y_shape, device="cuda")
    assert d.kernel_family == "mma_implicit"
    for call in (lambda: binding.onnx_gemm(A, A, Y=Z), lambda: d.run(X, W, Y=Y), lambda: d.prepack(W)):
        with pytest.raises(torch.OutOfMemoryError):
            launches_without_memory(call)
