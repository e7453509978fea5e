"""Convolutions whose residual addend is read at every so-many-th row and column of larger images, and the ResNet-50 graph whose
strides were moved up to such layers: the same function as the graph that they were moved in."""
import numpy as np
import pytest

import oracle
from parity import worst_ratio
from paper_2008_08272_b200 import binding

# (batch, C, M, R's H x W, strides): the persistent kernel by TMA rows (28x28, 14x14) and the split one, merged 7x7 and odd images
# behind a gather (their rows stored one by one), odd and even R, unequal strides, a single row, tiles that cross images
SHAPES = [(4, 64, 256, (56, 56), (2, 2)), (3, 128, 512, (27, 28), (2, 2)), (2, 256, 1024, (13, 14), (2, 2)), (1, 96, 80, (9, 33), (3, 1)),
          (16, 32, 272, (39, 40), (3, 5)), (2, 64, 128, (5, 12), (7, 3)), (64, 40, 48, (6, 5), (1, 2))]


def _graph_outputs(ops, x, params):
    """Every tensor of the graph, in float64 by numpy's and torch's own operators."""
    import torch
    import torch.nn.functional as F
    t = {"input": x}
    for op in ops:
        if op.sampled:
            t[op.res] = t[op.sampled][:, :, ::op.sample[0], ::op.sample[1]]
        s = t[op.src]
        if op.case is not None:
            assert tuple(s.shape) == tuple(op.case.x_shape)
            W, B = params[op.name]
            y = F.conv2d(s, W, B, stride=op.case.strides, padding=op.case.pads[0])
            if op.kind == "conv_add":
                y = y + t[op.res]
            y = y.relu() if op.relu else y
        elif op.kind == "maxpool":
            y = F.max_pool2d(s, 3, 2, 1)
        elif op.kind == "gap":
            y = s.mean((2, 3), keepdim=True)
        else:
            y = s.reshape(s.shape[0], -1)
        t[op.dst] = y
    return t


def test_moved_strides_leave_the_function_as_it_is():
    """On the CPU in float64, channels cut to eighths; every tensor of the moved graph is the other's, or its places read."""
    import torch
    from dataclasses import replace
    from paper_2008_08272_b200.resnet50_chain import build_graph, push_strides_up
    graph = build_graph(1)
    for op in graph:
        if op.case is not None:
            (n, c, h, w), (m, cg, kh, kw) = op.case.x_shape, op.case.w_shape
            cut = lambda v: v if v == 3 else v // 8
            op.case = replace(op.case, x_shape=(n, cut(c), h, w), w_shape=(cut(m), cut(cg), kh, kw))
    g = torch.Generator().manual_seed(5)
    params = {op.name: (torch.randn(op.case.w_shape, generator=g, dtype=torch.float64) / np.sqrt(np.prod(op.case.w_shape[1:])),
                        torch.randn(op.case.w_shape[0], generator=g, dtype=torch.float64)) for op in graph if op.case is not None}
    x = torch.rand(1, 3, 224, 224, generator=g, dtype=torch.float64)
    moved = push_strides_up(graph)
    assert [o.name for o in moved] == [o.name for o in graph] and sum(o.sampled is not None for o in moved) == 3
    assert not any(o.case is not None and o.case.w_shape[2:] == (1, 1) and o.case.strides != (1, 1) for o in moved)
    want, got = _graph_outputs(graph, x, params), _graph_outputs(moved, x, params)
    for op in graph:
        w, v = want[op.dst], got[op.dst]
        if w.shape != v.shape:
            w = w[:, :, ::2, ::2]
        assert torch.allclose(v, w, rtol=1e-12, atol=1e-12), op.name


def test_what_the_moved_graph_computes_is_counted():
    """A rate is that of the operations made: three 3x3 layers and the three 1x1 layers behind them make a quarter of the model's."""
    from paper_2008_08272_b200.resnet50_chain import build_graph, pass_flops, push_strides_up
    graph = build_graph(2)
    moved = push_strides_up(graph)
    fewer = [g.case.flops for g, m in zip(graph, moved) if g.case is not None and g.case.y_shape != m.case.y_shape]
    assert len(fewer) == 6 and pass_flops(graph) - pass_flops(moved) == sum(f * 3 // 4 for f in fewer)
    convs = sum(2 * int(np.prod(o.case.y_shape)) * int(np.prod(o.case.w_shape[1:])) for o in moved if o.case is not None)
    assert pass_flops(moved) == convs + 2 * 2 * 2048 * 1000


@pytest.mark.gpu
@pytest.mark.parametrize("rounded", [False, True])
@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("batch,C,M,hw,strides", SHAPES)
def test_sampled_addend(batch, C, M, hw, strides, native, rounded, monkeypatch):
    import torch
    if not native:
        monkeypatch.setattr(binding, "_fast_mod", binding._Declined())
    p, q = (-(-s // t) for s, t in zip(hw, strides))
    rng = np.random.default_rng(C * M + p)
    X, W, B, R = rng.random((batch, C, p, q), dtype=np.float32), rng.standard_normal((M, C, 1, 1), dtype=np.float32), \
        rng.standard_normal(M, dtype=np.float32), rng.standard_normal((batch, M) + hw, dtype=np.float32)
    d = binding.Conv2dDesc(X.shape, W.shape, has_bias=True, fuse_relu=True)
    assert d.kernel_family in ("mma_gemm", "mma_gather_gemm")
    x, w, b, r = (torch.from_numpy(v).cuda() for v in (X, W, B, R))
    packed = d.prepack(w)
    yr = torch.full(d.y_shape, 7.0, device="cuda") if rounded else None
    got = d.run_prepacked_sampled(x, w, packed, b, r, strides, Y_rounded=yr)
    some = np.ascontiguousarray(R[:, :, ::strides[0], ::strides[1]])
    plain = d.run_prepacked(x, w, packed, b, torch.from_numpy(some).cuda())       # the same sums, the addend read as it lies
    assert binding.last_device_status() == 0
    got, plain = got.cpu().numpy(), plain.cpu().numpy()
    assert np.array_equal(got, plain)
    if rounded:
        plain = ((plain.view(np.uint32) + np.uint32(0x1000)) & np.uint32(0xFFFFE000)).view(np.float32)      # (no NaNs here)
        assert np.array_equal(yr.cpu().numpy(), plain)
    conv, S = oracle.conv2d(X, W, B, relu=False)
    assert worst_ratio(got, np.maximum(conv + some.astype(np.float64), 0.0), S) <= 1.0


def test_refused():
    import ctypes
    fake, before = ctypes.c_void_p(0x1000), binding.launch_count()
    two = lambda *v: (ctypes.c_int64 * 2)(*v)
    lib = binding.load()
    call = lambda d, dims, strides, R=fake: lib.onnx_conv2d_run_packed_sampled(d._h, fake, fake, fake, 1 << 30, None, R, dims, strides, fake,
                                                                              None, fake, 1 << 30, None)
    d = binding.Conv2dDesc((2, 64, 28, 28), (128, 64, 1, 1))
    assert call(d, two(56, 56), two(2, 2), None) == 1 and call(d, None, two(2, 2)) == 1 and call(d, two(56, 56), None) == 1
    for dims, strides in (((57, 56), (2, 2)), ((56, 56), (1, 2)), ((28, 28), (0, 1)), ((0, 56), (2, 2))):
        assert call(d, two(*dims), two(*strides)) == 3
    assert call(d, two(1 << 20, 1 << 20), two((1 << 20) // 28 + 1, (1 << 20) // 28 + 1)) == 4
    assert call(binding.Conv2dDesc((2, 64, 28, 28), (128, 64, 3, 3), pads=(1,) * 4), two(56, 56), two(2, 2)) == 4
    assert binding.launch_count() == before


def test_one_tensor_for_both_outputs_is_refused():
    import ctypes
    at, before = (lambda n: ctypes.c_void_p(n << 12)), binding.launch_count()
    two = lambda *v: (ctypes.c_int64 * 2)(*v)
    for x, w in (((2, 64, 28, 28), (128, 64, 1, 1)), ((2, 64, 7, 7), (128, 64, 1, 1))):
        d = binding.Conv2dDesc(x, w)
        assert binding.load().onnx_conv2d_run_packed_sampled(d._h, at(1), at(2), at(3), 1 << 30, None, at(4), two(2 * x[2], 2 * x[3]), two(2, 2),
                                                             at(5), at(5), at(6), 1 << 30, None) == 4
    assert binding.launch_count() == before


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["Size", "list"])
def test_any_sequence_of_sizes_goes_the_native_way(kind, monkeypatch):
    import torch
    kind = torch.Size if kind == "Size" else list
    R = torch.rand(2, 128, 56, 56, device="cuda")
    X, W, d = torch.rand(2, 64, 28, 28, device="cuda"), torch.rand(128, 64, 1, 1, device="cuda"), binding.Conv2dDesc((2, 64, 28, 28), (128, 64, 1, 1))
    packed = d.prepack(W)
    want = d.run_prepacked_sampled(X, W, packed, None, R, (2, 2))
    monkeypatch.setattr(binding, "_i64", None)             # (what the calls through ctypes convert sizes with)
    got = d.run_prepacked_sampled(X, W, packed, None, R, kind((2, 2)), r_dims=kind((56, 56)))
    assert torch.equal(got, want)
