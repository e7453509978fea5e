"""The cluster-split forms of the tensor-core kernels (few output tiles): every tile width, channel block and cluster
size of the convolution, every shape of the GEMM form with the convolution epilogues, on ragged problems."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from parity import run_gemm_gpu, worst_ratio  # noqa: E402


@pytest.fixture(scope="module")
def binding():
    from paper_2008_08272_b200 import binding as b
    b.load(build_if_missing=False)
    return b


def _conv_add(binding, xs, ws, **kw):
    rng = np.random.default_rng(xs[1] * 7 + ws[0])
    X = rng.standard_normal(xs).astype(np.float32)
    W = (rng.standard_normal(ws) * np.sqrt(2.0 / (ws[1] * ws[2] * ws[3]))).astype(np.float32)
    B = rng.standard_normal((ws[0],)).astype(np.float32)
    conv, S = oracle.conv2d(X, W, B, relu=False, **kw)
    R = rng.standard_normal(conv.shape).astype(np.float32)
    dev = torch.device("cuda:0")
    d = binding.Conv2dDesc(xs, ws, has_bias=True, fuse_relu=True, **kw)
    buf = torch.full((conv.size + 128,), 4321.0, device=dev)
    Y = buf[64:64 + conv.size].view(conv.shape)
    Xd, Wd, Bd, Rd = (torch.from_numpy(a).to(dev) for a in (X, W, B, R))
    for r in (None, R):
        if r is None:
            d.run(Xd, Wd, Bd, Y=Y)
        else:
            d.run_add(Xd, Wd, Bd, Rd, Y=Y)
        torch.cuda.synchronize()
        assert binding.last_device_status() == 0
        want = np.maximum(conv if r is None else conv + r, 0.0)
        assert worst_ratio(Y.cpu().numpy(), want, S) <= 1.0, (xs, ws, r is None)
    assert bool((buf[:64] == 4321.0).all()) and bool((buf[64 + conv.size:] == 4321.0).all()), "store outside Y"
    d.close()


@pytest.mark.parametrize("split", [2, 4, 8])
@pytest.mark.parametrize("bn", [16, 64, 256])
def test_conv_split_channel_blocks(binding, bn, split, monkeypatch):
    for kb in (16, 32):
        monkeypatch.setenv("ONNXB_CONV_SPLIT", f"{bn},{kb},{split}")      # read when the descriptor is created
        _conv_add(binding, (2, 256, 14, 14), (72, 256, 3, 3), pads=(1, 1, 1, 1))
        _conv_add(binding, (3, 272, 7, 7), (40, 272, 3, 3), pads=(1, 1, 1, 1))
        _conv_add(binding, (1, 512, 20, 20), (34, 256, 3, 3), pads=(1, 1, 1, 1), group=2, strides=(2, 2))


@pytest.mark.parametrize("shape", ["32,1", "32,8", "64,2", "128,1", "128,4"])
def test_gemm_split_conv_epilogues_and_transposes(binding, shape, monkeypatch):
    monkeypatch.setenv("ONNXB_GEMM_SPLITK", shape)
    _conv_add(binding, (2, 256, 14, 14), (136, 256, 1, 1))                       # one GEMM per image
    _conv_add(binding, (3, 288, 7, 7), (72, 288, 1, 1))                          # gathered, merged columns
    _conv_add(binding, (2, 256, 28, 28), (130, 256, 1, 1), strides=(2, 2))       # gathered, per image
    rng = np.random.default_rng(5)
    for tA in (False, True):
        for tB in (False, True):
            M, N, K = 132, 68, 260
            A = rng.standard_normal((K, M) if tA else (M, K)).astype(np.float32)
            B = rng.standard_normal((N, K) if tB else (K, N)).astype(np.float32)
            C = rng.standard_normal((M, N)).astype(np.float32)
            got = run_gemm_gpu(binding, torch, A, B, C, alpha=0.5, beta=2.0, transA=tA, transB=tB)
            want, S = oracle.gemm(A, B, C, alpha=0.5, beta=2.0, transA=tA, transB=tB)
            assert worst_ratio(got, want, S) <= 1.0
