"""fp32 on the tensor cores by split operands: pixel tiles that hold parts of several images and tiles of one image, the last
elements of X that are no whole 16-byte piece, padding on every side, strides and dilations of their own, odd chunks of
channels, several channel tiles and blocks, reductions shared by clusters of every size; from packed filters as from plain ones, and where
no workspace is given; every split and tile width of Gemm."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

REL = 2e-6          # of sum |x*w|: fp32 rounding of the partial sums of up to a few hundred terms

CONVS = [dict(x=(3, 11, 9, 7), w=(20, 11, 3, 3), pads=(1, 1, 1, 1)), dict(x=(7, 5, 5, 5), w=(33, 5, 3, 3), pads=(1, 0, 2, 1)),
         dict(x=(1, 9, 31, 27), w=(130, 9, 5, 5), pads=(2, 2, 2, 2)), dict(x=(2, 24, 25, 33), w=(40, 12, 3, 3), pads=(2, 3, 2, 3), dilations=(2, 3), group=2),
         dict(x=(2, 7, 29, 35), w=(17, 7, 7, 7), pads=(3, 3, 3, 3), strides=(2, 2)), dict(x=(1, 3, 41, 23), w=(24, 3, 5, 3), strides=(3, 1), pads=(0, 1, 4, 0)),
         dict(x=(3, 70, 11, 13), w=(31, 70, 1, 1)), dict(x=(5, 33, 14, 9), w=(130, 33, 1, 1), strides=(2, 3)),
         dict(x=(2, 18, 9, 9), w=(10, 9, 1, 1), group=2), dict(x=(1, 6, 1, 300), w=(9, 6, 1, 9), pads=(0, 4, 0, 4)),
         # blocks and terms enough for every number of CTAs that share a reduction
         dict(x=(2, 58, 11, 13), w=(21, 58, 3, 3), pads=(1, 1, 1, 1)), dict(x=(1, 64, 9, 11), w=(68, 32, 3, 3), pads=(1, 1, 1, 1), strides=(2, 1), group=2),
         dict(x=(2, 1130, 7, 9), w=(33, 1130, 1, 1))]
TILES = ["1,16,1", "2,48,1", "3,128,1", "2,32,2", "1,16,4", "1,32,8"]


@pytest.fixture(scope="module")
def binding():
    from paper_2008_08272_b200 import binding as b
    b.load(build_if_missing=False)
    b.set_kernel_override("simt_direct")
    yield b
    b.set_kernel_override(None)


def _pin(monkeypatch, tile):
    """A tile of the staged convolutions, and its width and split for those that go as a Gemm of packed pixels."""
    monkeypatch.setenv("ONNXB_FP32", "tc")
    if tile:
        monkeypatch.setenv("ONNXB_FP32_TILE", tile)
        monkeypatch.setenv("ONNXB_FP32_GEMM", tile.split(",", 1)[1])


def _desc(binding, c, **more):
    return binding.Conv2dDesc(c["x"], c["w"], **{k: v for k, v in c.items() if k not in "xw"}, **more)


def _launches(binding, call):
    before = binding.launch_count()
    return call(), binding.launch_count() - before


@pytest.mark.parametrize("tile", TILES)
def test_every_tile_has_layers(binding, tile, monkeypatch):
    _pin(monkeypatch, tile)
    assert sum(_desc(binding, c).workspace_bytes > 0 for c in CONVS) >= 2


@pytest.mark.parametrize("tile", [None] + TILES)
@pytest.mark.parametrize("c", CONVS, ids=lambda c: "x".join(map(str, c["x"] + c["w"])))
def test_conv(binding, c, tile, monkeypatch):
    _pin(monkeypatch, tile)
    rng = np.random.default_rng(c["x"][1])
    X, W, B = (rng.standard_normal(s).astype(np.float32) for s in (c["x"], c["w"], c["w"][:1]))
    kw = dict(pads=c.get("pads", (0,) * 4), strides=c.get("strides", (1, 1)), dilations=c.get("dilations", (1, 1)), group=c.get("group", 1))
    d = _desc(binding, c, has_bias=True, fuse_relu=True)
    if d.workspace_bytes == 0:
        pytest.skip("a tile that this layer has no plan for")
    R = rng.standard_normal(d.y_shape).astype(np.float32)
    x, w, b, r = (torch.from_numpy(t).cuda() for t in (X, W, B, R))
    want, S = oracle.conv2d(X, W, B, **kw)
    ok = lambda got, ref, s: (np.abs(got.cpu().numpy() - np.maximum(ref, 0)) <= REL * s + 1e-5).all()
    (got, launches), added = _launches(binding, lambda: d.run(x, w, b)), d.run_add(x, w, b, r)
    assert launches == 2                                  # operands split by the one in front: the kernel under test
    assert ok(got, want, S) and ok(added, want + R, S + np.abs(R))
    packed = d.prepack(w)
    assert torch.equal(d.run_prepacked(x, w, packed, b), got) and torch.equal(d.run_prepacked(x, w, packed, b, r), added)
    short = packed[:16]                                   # not this descriptor's copy: W is read instead
    assert torch.equal(d.run_prepacked(x, w, short, b), got) and torch.equal(d.run_prepacked(x, w, short, b, r), added)
    assert packed.numel() == max(16, d.packed_bytes)
    y, stream = torch.empty_like(got), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    # the entry that is not told the copy's size: no byte of a pointer that may be no copy is read
    wsp = torch.empty(d.workspace_bytes, dtype=torch.uint8, device="cuda")
    assert binding.load().onnx_conv2d_run_prepacked(d._h, ptr(x), ptr(w), ptr(torch.zeros(16, dtype=torch.uint8, device="cuda")), ptr(b), None, ptr(y),
                                                    ptr(wsp), wsp.numel(), stream) == 0 and torch.equal(y, got)
    # without a workspace: the kernel on the FMA units
    assert binding.load().onnx_conv2d_run(d._h, ptr(x), ptr(w), ptr(b), ptr(y.zero_()), None, 0, stream) == 0 and ok(y, want, S)
    assert binding.load().onnx_conv2d_prepack(d._h, ptr(w), None, 0, stream) == 0
    assert binding.last_device_status() == 0


def test_gemm_of_the_fp32_family_whose_rows_tma_could_address(binding, monkeypatch):
    """The kernel override of this module's descriptors holds for Gemm, too."""
    A, B = (torch.randn(1024, 1024, generator=torch.Generator().manual_seed(s)) for s in (1, 2))
    a, b = A.cuda(), B.cuda()
    got, launches = _launches(binding, lambda: binding.onnx_gemm(a, b, transB=True))
    want, S = oracle.gemm(A.numpy(), B.numpy(), None, transB=True)
    assert launches == 2 and (np.abs(got.cpu().numpy() - want) <= REL * S + 1e-5).all()


@pytest.mark.parametrize("tile", ["16,1", "48,1", "128,1", "64,2", "32,4", "16,8"])
def test_gemm(binding, tile, monkeypatch):
    monkeypatch.setenv("ONNXB_FP32", "tc")
    monkeypatch.setenv("ONNXB_FP32_GEMM", tile)
    rng = np.random.default_rng(5)
    pinned = 0
    for M, N, K, tA, tB in ((129, 130, 259, False, False), (131, 257, 290, True, True), (3, 1400, 513, False, True), (150, 33, 1027, True, False),
                            (150, 133, 1130, False, True), (137, 201, 2050, True, False)):
        has_plan = binding.gemm_workspace_bytes(tA, tB, M, N, K) > 0
        pinned += has_plan
        A = rng.standard_normal((K, M) if tA else (M, K)).astype(np.float32)
        B = rng.standard_normal((N, K) if tB else (K, N)).astype(np.float32)
        C = rng.standard_normal((M, N)).astype(np.float32)
        a, b, c = (torch.from_numpy(t).cuda() for t in (A, B, C))
        for addend, beta in ((None, 0.0), (C, -1.5)):
            got, launches = _launches(binding, lambda: binding.onnx_gemm(a, b, None if addend is None else c, alpha=0.5, beta=beta, transA=tA, transB=tB).cpu().numpy())
            assert launches == (2 if has_plan else 1)
            want, S = oracle.gemm(A, B, addend, alpha=0.5, beta=beta, transA=tA, transB=tB)
            assert (np.abs(got - want) <= REL * S + 1e-5).all(), (M, N, K, beta)
    assert pinned >= 2
    assert binding.last_device_status() == 0
