"""The fp32 contractions (operands TMA cannot describe, thin reductions): every tile shape and reduction split of
the FMA kernel, the split-TF32 tensor-core kernel and the dot-product kernel against the oracle, at an fp32
tolerance, on sizes that leave ragged tails in every direction."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from parity import run_conv_gpu, run_gemm_gpu  # noqa: E402

PINS = ["tc"] + [f"{shape},{split}" for shape in range(5) for split in (1, 3, 8)]
GEMMS = [(1, 130, 65, False, False), (129, 257, 31, True, False), (65, 127, 97, False, True), (131, 70, 333, True, True)]
CONVS = [dict(x=(2, 5, 13, 11), w=(17, 5, 3, 3), pads=(1, 1, 1, 1), dilations=(2, 1)),
         dict(x=(1, 6, 19, 23), w=(130, 3, 7, 7), pads=(3, 3, 3, 3), strides=(2, 2), group=2),
         dict(x=(3, 40, 9, 7), w=(33, 40, 1, 1), strides=(2, 2))]
REL = 2e-6          # of sum |x*w|: fp32 rounding of up to a few hundred terms


@pytest.fixture(scope="module")
def binding():
    from paper_2008_08272_b200 import binding as b
    b.load(build_if_missing=False)
    return b


@pytest.mark.parametrize("pin", PINS)
def test_fp32_gemm_and_conv_tiles(binding, pin, monkeypatch):
    monkeypatch.setenv("ONNXB_FP32", pin)           # read at every launch
    rng = np.random.default_rng(len(pin) * 31 + ord(pin[0]))
    binding.set_kernel_override("simt_direct")
    try:
        for M, N, K, tA, tB in GEMMS:
            A = rng.standard_normal((K, M) if tA else (M, K)).astype(np.float32)
            B = rng.standard_normal((N, K) if tB else (K, N)).astype(np.float32)
            C = rng.standard_normal((M, 1)).astype(np.float32)
            kw = dict(alpha=0.5, beta=-1.5, transA=tA, transB=tB)
            # (the first is the dot-product kernel's under every pin)
            assert (binding.gemm_workspace_bytes(tA, tB, M, N, K) > 0) == (pin == "tc" and M > 1)
            got = run_gemm_gpu(binding, torch, A, B, C, fuse_relu=True, **kw)
            want, S = oracle.gemm(A, B, C, relu=True, **kw)
            assert (np.abs(got - want) <= REL * S + 1e-5).all(), (M, N, K)
        for c in CONVS:
            X = rng.standard_normal(c["x"]).astype(np.float32)
            W = rng.standard_normal(c["w"]).astype(np.float32)
            B = rng.standard_normal((c["w"][0],)).astype(np.float32)
            kw = dict(pads=c.get("pads", (0, 0, 0, 0)), strides=c.get("strides", (1, 1)),
                      dilations=c.get("dilations", (1, 1)), group=c.get("group", 1))
            assert (binding.Conv2dDesc(X.shape, W.shape, **kw).workspace_bytes > 0) == (pin == "tc")
            got, fam = run_conv_gpu(binding, torch, X, W, B, relu=True, **kw)
            assert fam == "simt_direct"
            want, S = oracle.conv2d(X, W, B, relu=True, **kw)
            assert (np.abs(got - want) <= REL * S + 1e-5).all(), c
    finally:
        binding.set_kernel_override(None)


SMALL_CONVS = [dict(x=(1, 1, 28, 28), w=(8, 1, 5, 5), pads=(2, 2, 2, 2)), dict(x=(90, 3, 13, 11), w=(7, 3, 3, 3), pads=(1, 0, 2, 1)),
               dict(x=(100, 4, 9, 9), w=(18, 2, 2, 4), strides=(2, 1), dilations=(1, 2), group=2),
               dict(x=(70, 2, 17, 19), w=(16, 2, 5, 5), pads=(2, 2, 2, 2), strides=(2, 2))]


@pytest.mark.parametrize("c", SMALL_CONVS, ids=lambda c: "x".join(map(str, c["x"] + c["w"])))
def test_small_image_conv(binding, c, monkeypatch):
    """The whole-image-in-shared-memory kernel, ragged channels and pixels (every channel count per block: test_small_conv.py)."""
    monkeypatch.setenv("ONNXB_FP32", "small")
    rng = np.random.default_rng(17)
    X = rng.standard_normal(c["x"]).astype(np.float32)
    W = rng.standard_normal(c["w"]).astype(np.float32)
    B = rng.standard_normal((c["w"][0],)).astype(np.float32)
    kw = dict(pads=c.get("pads", (0, 0, 0, 0)), strides=c.get("strides", (1, 1)), dilations=c.get("dilations", (1, 1)),
              group=c.get("group", 1))
    for images in (1, c["x"][0]):
        got, fam = run_conv_gpu(binding, torch, X[:images], W, B, relu=True, **kw)
        assert fam == "simt_direct"
        want, S = oracle.conv2d(X[:images], W, B, relu=True, **kw)
        assert (np.abs(got - want) <= REL * S + 1e-5).all()


@pytest.mark.parametrize("shape,k,st,pads", [((1, 8, 28, 28), 2, 2, 0), ((1, 16, 14, 14), 3, 3, 0), ((2, 5, 9, 11), 3, 2, 1)])
def test_small_max_pool(binding, shape, k, st, pads):
    X = torch.randn(shape, device="cuda")
    got = binding.onnx_maxpool2d(X, (k, k), pads=(pads,) * 4, strides=(st, st))
    assert torch.equal(got.cpu(), torch.nn.functional.max_pool2d(X.cpu(), k, st, padding=pads))


@pytest.mark.parametrize("tA", [False, True])
@pytest.mark.parametrize("shape", [(1, 10, 256), (64, 10, 256), (33, 31, 7), (3, 5, 291)])
def test_tiny_gemm(binding, shape, tA):
    M, N, K = shape
    rng = np.random.default_rng(K)
    for tB in (False, True):
        A = rng.standard_normal((K, M) if tA else (M, K)).astype(np.float32)
        B = rng.standard_normal((N, K) if tB else (K, N)).astype(np.float32)
        C = rng.standard_normal((N,)).astype(np.float32)
        got = run_gemm_gpu(binding, torch, A, B, C, transA=tA, transB=tB)
        want, S = oracle.gemm(A, B, C, transA=tA, transB=tB)
        assert (np.abs(got - want) <= REL * S + 1e-6).all()


def _as_an_fp32_sum(got, want):
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.isnan(want).any() and np.isinf(want).any() and np.allclose(got[ok], want[ok], rtol=1e-5, atol=1e-4)


@pytest.mark.parametrize("tile", [None, "16,1", "32,2"])        # (a reduction shared by two CTAs)
def test_split_operands_that_overflow(binding, tile, monkeypatch):
    """Infinite, NaN and near-overflow operands have no hi/lo split: the outputs they reach are summed in
    plain fp32 and come out as an fp32 sum gives them."""
    monkeypatch.setenv("ONNXB_FP32", "tc")
    if tile:
        monkeypatch.setenv("ONNXB_FP32_GEMM", tile)
    assert binding.gemm_workspace_bytes(False, False, 70, 131, 75) > 0
    rng = np.random.default_rng(8)
    A = rng.standard_normal((70, 75)).astype(np.float32)
    B = rng.standard_normal((75, 131)).astype(np.float32)
    A[3, 5], A[60, 7], A[20, 1] = np.inf, np.nan, 3.40282e38
    B[1, :] = 1e-3
    got = run_gemm_gpu(binding, torch, A, B, None)
    with np.errstate(all="ignore"):
        want = A.astype(np.float64) @ B.astype(np.float64)
    _as_an_fp32_sum(got, want)


@pytest.mark.parametrize("split", [1, 8])                       # CTAs that share a reduction
@pytest.mark.parametrize("xs,ws,pads", [((2, 58, 11, 13), (21, 58, 3, 3), (1, 1, 1, 1)), ((2, 1130, 7, 9), (33, 1130, 1, 1), (0, 0, 0, 0))],
                         ids=["staged", "packed pixels"])
def test_split_conv_operands_that_overflow(binding, xs, ws, pads, split, monkeypatch):
    monkeypatch.setenv("ONNXB_FP32", "tc")
    monkeypatch.setenv("ONNXB_FP32_TILE", f"1,16,{split}")
    monkeypatch.setenv("ONNXB_FP32_GEMM", f"16,{split}")
    rng = np.random.default_rng(9)
    X = rng.standard_normal(xs).astype(np.float32)
    W = (rng.standard_normal(ws) * 0.05).astype(np.float32)
    X[0, 5, 1, 2], X[1, 7, 6, 3], X[1, 31, 2, 6] = np.inf, np.nan, 3.40282e38
    W[:, 31] = 1e-3
    assert binding.Conv2dDesc(xs, ws, pads=pads).workspace_bytes > 0
    got, fam = run_conv_gpu(binding, torch, X, W, None, pads=pads)
    assert fam == "simt_direct"
    _as_an_fp32_sum(got, oracle.conv2d(X, W, None, pads=pads)[0])


@pytest.mark.parametrize("pin", ["tc", "0,1", "2,3", "3,1", "4,8"])
def test_conv_offsets_beyond_32_bits(binding, pin, monkeypatch):
    """A dilation and a pad of 2^19 rows of 4096 and more columns: filter taps inside the image whose offset from the
    window's start is 2^31 elements and more, and (700 rows fewer) just below that."""
    monkeypatch.setenv("ONNXB_FP32", pin)
    rng = np.random.default_rng(11)
    far, near = 1 << 19, (1 << 19) - 700
    for xs, ws, kw in (((2, 6, 4, 4096), (6, 3, 2, 1), dict(pads=(far, 0, 0, 0), dilations=(far, 1), group=2)),
                       ((2, 6, 4, 4096), (6, 3, 2, 1), dict(pads=(near, 0, 0, 0), dilations=(near, 1), group=2)),
                       ((1, 3, 3, 5000), (40, 3, 2, 3), dict(pads=(far, 1, 0, 1), dilations=(far, 1)))):
        X, W, B = (rng.standard_normal(s).astype(np.float32) for s in (xs, ws, ws[:1]))
        got, fam = run_conv_gpu(binding, torch, X, W, B, **kw)
        assert fam == "simt_direct"
        want, S = oracle.conv2d(X, W, B, **kw)
        assert (np.abs(got - want) <= REL * S + 1e-5).all()
