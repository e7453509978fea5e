"""The tile and stage variants that the tensor-core kernels choose between, and the depthwise kernel's streamed form, at
the sizes where each can go wrong: partial channel blocks, reductions that end inside a stage, tiles of few rows, units of
fewer planes."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from parity import check_conv, run_gemm_gpu, worst_ratio  # noqa: E402


@pytest.fixture(scope="module")
def binding():
    from paper_2008_08272_b200 import binding as b
    b.load(build_if_missing=False)
    return b


def _operands(xs, ws):
    rng = np.random.default_rng(xs[1] + ws[0])
    X = rng.standard_normal(xs).astype(np.float32)
    W = (rng.standard_normal(ws) * np.sqrt(2.0 / (ws[1] * ws[2] * ws[3]))).astype(np.float32)
    return X, W, rng.standard_normal((ws[0],)).astype(np.float32)


@pytest.mark.parametrize("tile", ["1,1,96,64", "2,1,64,32", "1,2,64,32", "2,2,96,16"])
def test_conv_channel_blocks_and_tile_widths(binding, tile, monkeypatch):
    monkeypatch.setenv("ONNXB_CONV_TILE", tile)           # read when the descriptor is created
    for xs, ws, kw in (((9, 100, 6, 8), (104, 100, 3, 3), dict(pads=(1, 1, 1, 1))),
                       ((5, 168, 6, 8), (200, 84, 3, 3), dict(pads=(1, 0, 0, 1), group=2))):
        ratio, family = check_conv(binding, torch, *_operands(xs, ws), relu=True, **kw)
        assert family == "mma_implicit" and ratio <= 1.0, (xs, ws)


@pytest.mark.parametrize("tile", ["1,1,48,16", "2,2,48,16"])
def test_thin_conv_keeps_its_weights_over_several_tiles(binding, tile, monkeypatch):
    monkeypatch.setenv("ONNXB_CONV_TILE", tile)
    ratio, family = check_conv(binding, torch, *_operands((9, 3, 128, 112), (40, 3, 7, 7)), relu=True, pads=(3, 3, 3, 3), strides=(2, 2))
    assert family == "mma_implicit" and ratio <= 1.0


@pytest.mark.parametrize("pair", ["0", "1"])
@pytest.mark.parametrize("ks", ["1", "2"])
def test_gemm_k_blocks_per_stage(binding, ks, pair, monkeypatch):
    monkeypatch.setenv("ONNXB_GEMM_KS", ks)
    monkeypatch.setenv("ONNXB_GEMM_PAIR", pair)
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", "0")
    rng = np.random.default_rng(3)
    for tA in (False, True):
        for tB in (False, True):
            for M, N, K in ((260, 132, 160), (256, 100, 132)):
                A = rng.standard_normal((K, M) if tA else (M, K)).astype(np.float32)
                B = rng.standard_normal((N, K) if tB else (K, N)).astype(np.float32)
                got = run_gemm_gpu(binding, torch, A, B, None, transA=tA, transB=tB)
                want, S = oracle.gemm(A, B, None, transA=tA, transB=tB)
                assert worst_ratio(got, want, S) <= 1.0, (M, N, K, tA, tB)


@pytest.mark.parametrize("rows", [1, 7, 9, 65])
def test_gemm_split_of_few_rows(binding, rows, monkeypatch):
    rng = np.random.default_rng(rows)
    binding.set_kernel_override("mma_gemm")                     # else the dot-product kernel takes the tiny ones
    try:
        for shape in ("32,1", "32,8", "128,4"):
            monkeypatch.setenv("ONNXB_GEMM_SPLITK", shape)
            for N, K in ((1000, 768), (132, 356)):
                A = rng.standard_normal((rows, K)).astype(np.float32)
                B = rng.standard_normal((N, K)).astype(np.float32)
                C = rng.standard_normal((N,)).astype(np.float32)
                before = binding.launch_count()
                got = run_gemm_gpu(binding, torch, A, B, C, transB=True)
                assert binding.launch_count() == before + 1     # the other tensor-core form has a rounding launch in front
                want, S = oracle.gemm(A, B, C, transB=True)
                assert worst_ratio(got, want, S) <= 1.0, (shape, N, K)
    finally:
        binding.set_kernel_override(None)


@pytest.mark.parametrize("xs,pads", [((47, 126, 28, 28), (1, 1, 1, 1)), ((75, 128, 32, 32), (0, 1, 0, 1)), ((151, 128, 15, 16), (2, 1, 1, 1))])
def test_depthwise_streamed_planes(binding, xs, pads):
    X, W, B = _operands(xs, (xs[1], 1, 3, 3))
    images = [0, xs[0] // 2, xs[0] - 1]
    ratio, family = check_conv(binding, torch, X, W, B, relu=True, pads=pads, group=xs[1], images=images)
    assert family == "simt_depthwise" and ratio <= 1.0


@pytest.mark.parametrize("cs", [(), (1,), ("N",), (1, "N"), ("M", 1), ("M", "N")], ids=str)
def test_gemm_addend_forms(binding, cs, monkeypatch):
    """C of every broadcast form in the persistent kernel's epilogue, where Y goes out by TMA and where it does not (rows that
    are no multiples of 16 bytes), on tiles that end inside a block of rows and of columns."""
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", "0")
    rng = np.random.default_rng(2)
    for M, N, K in ((300, 332, 96), (300, 330, 96), (20, 37, 64)):
        A, B = rng.standard_normal((M, K)).astype(np.float32), rng.standard_normal((N, K)).astype(np.float32)
        C = rng.standard_normal([{"M": M, "N": N}.get(d, d) for d in cs]).astype(np.float32)
        before = binding.launch_count()
        binding.set_kernel_override("mma_gemm")                 # else the dot-product kernel takes the last one
        try:
            got = run_gemm_gpu(binding, torch, A, B, C, transB=True, alpha=0.5, beta=-1.5, fuse_relu=True)
        finally:
            binding.set_kernel_override(None)
        assert binding.launch_count() == before + 2             # operands rounded by a launch in front: not the split form
        want, S = oracle.gemm(A, B, C, transB=True, alpha=0.5, beta=-1.5, relu=True)
        assert worst_ratio(got, want, S) <= 1.0, (M, N)


@pytest.mark.parametrize("tA,tB", [(False, True), (True, False)])
@pytest.mark.parametrize("M,N,K", [(640, 640, 1280), (704, 304, 2640), (144, 176, 4784)])
def test_gemm_rounded_ahead_of_the_split(binding, M, N, K, tA, tB, monkeypatch):
    """Problems whose operands are rounded by a launch of their own and then go to the split kernel: the first one's tiles to a CTA
    each, the others' to clusters."""
    rng = np.random.default_rng(M)
    A = rng.standard_normal((K, M) if tA else (M, K)).astype(np.float32)
    B = rng.standard_normal((N, K) if tB else (K, N)).astype(np.float32)
    C = rng.standard_normal((N,)).astype(np.float32)
    before = binding.launch_count()
    got = run_gemm_gpu(binding, torch, A, B, C, transA=tA, transB=tB, alpha=0.5, beta=-1.5)
    assert binding.launch_count() == before + 2
    want, S = oracle.gemm(A, B, C, transA=tA, transB=tB, alpha=0.5, beta=-1.5)
    assert worst_ratio(got, want, S) <= 1.0
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", "0")                # the persistent kernel, also with a launch in front: a sum in one piece
    whole = run_gemm_gpu(binding, torch, A, B, C, transA=tA, transB=tB, alpha=0.5, beta=-1.5)
    assert np.array_equal(whole, got) == (K == 1280)
