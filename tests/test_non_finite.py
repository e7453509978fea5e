"""NaN operands: without Relu, an output is NaN exactly where its sum has a NaN term, on every path an operand can take to the
tensor core, whatever the NaN's bit pattern; every other output is what it is without them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from parity import ABS, REL, run_conv_gpu, run_gemm_gpu  # noqa: E402


@pytest.fixture(scope="module")
def binding():
    from paper_2008_08272_b200 import binding as b
    b.load(build_if_missing=False)
    return b


def _same_nans(got, reached, want, S):
    assert np.array_equal(np.isnan(got), reached), "NaN outputs are not the ones a NaN reaches"
    ok = ~reached
    assert ok.any() and (np.abs(got - want)[ok] <= (REL * S + ABS)[ok]).all()


def _conv(binding, xs, ws, pattern, family, **kw):
    rng = np.random.default_rng(xs[1] * 5 + ws[0])
    X = rng.standard_normal(xs).astype(np.float32)
    W = (rng.standard_normal(ws) * np.sqrt(2.0 / np.prod(ws[1:]))).astype(np.float32)
    B = rng.standard_normal((ws[0],)).astype(np.float32)
    want, S = oracle.conv2d(X, W, B, **kw)
    spot = tuple(np.asarray(xs) // 2)
    nan = np.array([pattern], dtype=np.uint32).view(np.float32)[0]
    for bad, at in ((X.copy(), "X"), (W.copy(), "W")):
        mx, mw = np.zeros_like(X), np.zeros_like(W)
        if at == "X":
            bad[spot] = nan
            mx[spot], mw[:] = 1, 1
        else:
            tap = (ws[0] // 2, ws[1] // 2, ws[2] // 2, ws[3] // 2)        # the middle one: never on padding
            bad[tap] = nan
            mw[tap], mx[:] = 1, 1
        reached = oracle.conv2d(mx, mw, None, **kw)[0] > 0
        got, fam = run_conv_gpu(binding, torch, bad if at == "X" else X, bad if at == "W" else W, B, **kw)
        assert fam == family
        _same_nans(got, reached, want, S)


IMPLICIT = [("whole tiles", dict(ONNXB_CONV_SPLIT="0"), (4, 64, 20, 20), (48, 64, 3, 3), dict(pads=(1, 1, 1, 1))),
            ("tile pairs", dict(ONNXB_CONV_TILE="2,2,64"), (4, 64, 20, 20), (96, 64, 3, 3), dict(pads=(1, 1, 1, 1))),
            ("split", dict(ONNXB_CONV_SPLIT="64,16,4"), (2, 128, 12, 12), (48, 128, 3, 3), dict(pads=(1, 1, 1, 1))),
            ("thin", {}, (6, 3, 64, 64), (64, 3, 7, 7), dict(pads=(3, 3, 3, 3), strides=(2, 2)))]


# as numpy writes it, as GPU arithmetic makes it, and that negated
PATTERNS = [0x7FC00000, 0x7FFFFFFF, 0xFFFFFFFF]


@pytest.mark.parametrize("pattern", PATTERNS, ids=hex)
@pytest.mark.parametrize("case", IMPLICIT, ids=lambda c: c[0])
def test_implicit_conv_without_relu_keeps_nan(binding, case, pattern, monkeypatch):
    _, env, xs, ws, kw = case
    for k, v in env.items():
        monkeypatch.setenv(k, v)                        # read when the descriptor is created
    binding.set_kernel_override("mma_implicit")
    try:
        _conv(binding, xs, ws, pattern, "mma_implicit", **kw)
    finally:
        binding.set_kernel_override(None)


@pytest.mark.parametrize("pattern", PATTERNS, ids=hex)
@pytest.mark.parametrize("split", ["0", "64,2"])
def test_1x1_conv_without_relu_keeps_nan(binding, split, pattern, monkeypatch):
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", split)
    _conv(binding, (2, 64, 16, 16), (136, 64, 1, 1), pattern, "mma_gemm")
    _conv(binding, (2, 64, 32, 32), (136, 64, 1, 1), pattern, "mma_gather_gemm", strides=(2, 2))      # 16-byte loads
    _conv(binding, (3, 64, 7, 7), (136, 64, 1, 1), pattern, "mma_gather_gemm")                        # scalar loads, merged images


def _gemm(binding, M, N, K, pattern):
    rng = np.random.default_rng(M + N)
    A = rng.standard_normal((M, K)).astype(np.float32)
    B = rng.standard_normal((K, N)).astype(np.float32)
    want, S = oracle.gemm(A, B, None)
    nan = np.array([pattern], dtype=np.uint32).view(np.float32)[0]
    a, b = A.copy(), B.copy()
    a[M // 2, K - 1] = b[3, N - 2] = nan
    reached = np.zeros((M, N), bool)
    reached[M // 2] = True
    _same_nans(run_gemm_gpu(binding, torch, a, B, None), reached, want, S)
    reached = np.zeros((M, N), bool)
    reached[:, N - 2] = True
    _same_nans(run_gemm_gpu(binding, torch, A, b, None), reached, want, S)


@pytest.mark.parametrize("pattern", PATTERNS, ids=hex)
@pytest.mark.parametrize("split", ["0", "64,2"])           # operands rounded by a launch in front, or in shared memory
def test_gemm_keeps_nan(binding, split, pattern, monkeypatch):
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", split)
    _gemm(binding, 140, 132, 128, pattern)


@pytest.mark.parametrize("pattern", PATTERNS, ids=hex)
@pytest.mark.parametrize("split", [1, 2])                  # CTAs that share a reduction
def test_split_fp32_keeps_nan(binding, split, pattern, monkeypatch):
    """fp32 on the tensor cores, by two TF32 parts of every operand: Gemm, and Conv with staged pixels and with packed ones."""
    monkeypatch.setenv("ONNXB_FP32", "tc")
    monkeypatch.setenv("ONNXB_FP32_GEMM", f"16,{split}")
    if split > 1:
        monkeypatch.setenv("ONNXB_FP32_TILE", f"1,16,{split}")
    binding.set_kernel_override("simt_direct")
    try:
        assert binding.gemm_workspace_bytes(False, False, 70, 131, 75) > 0
        _gemm(binding, 70, 131, 75, pattern)
        for xs, ws, kw in (((2, 6, 19, 23), (130, 3, 3, 3), dict(pads=(1, 1, 1, 1), group=2)) if split == 1 else
                           ((2, 58, 11, 13), (21, 58, 3, 3), dict(pads=(1, 1, 1, 1))), ((2, 70, 11, 13), (31, 70, 1, 1), {})):
            assert binding.Conv2dDesc(xs, ws, **kw).workspace_bytes > 0
            _conv(binding, xs, ws, pattern, "simt_direct", **kw)
    finally:
        binding.set_kernel_override(None)
