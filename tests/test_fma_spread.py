"""The fp32 FMA kernels at launches on either side of the sizes from which an SM's share of the blocks is kept by the shared memory
asked for: 100 blocks, one to four per SM and more, clusters, every tile shape; Gemm and convolution, one launch behind the other."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2008_08272_b200 import binding  # noqa: E402

TILES = [(128, 128), (64, 128), (64, 64), (16, 128), (32, 32)]


@pytest.mark.parametrize("shape", range(len(TILES)))
@pytest.mark.parametrize("split", [1, 2, 8])
@pytest.mark.parametrize("blocks", [96, 104, 148, 152, 592, 600])
def test_gemm(shape, split, blocks, monkeypatch):
    monkeypatch.setenv("ONNXB_FP32", "%d,%d" % (shape, split))
    bm, bn = TILES[shape]
    tiles = -(-blocks // split)
    rows = 2 if tiles % 2 == 0 else 1
    M, N, K = bm * rows - 3, bn * (tiles // rows) - 1, 37 + 32 * split
    rng = np.random.default_rng(blocks)
    A, B = rng.standard_normal((M, K), dtype=np.float32), rng.standard_normal((K, N), dtype=np.float32)
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    first = binding.onnx_gemm(a, b)
    for _ in range(3):                                     # (placed beside the launch before)
        again = binding.onnx_gemm(a, b)
    assert binding.last_device_status() == 0 and torch.equal(first, again)
    want, S = A.astype(np.float64) @ B.astype(np.float64), np.abs(A).astype(np.float64) @ np.abs(B)
    assert np.all(np.abs(first.cpu().numpy() - want) <= (K + 8) * 2.0 ** -24 * 1.01 * S)      # K fused additions, and a cluster's


@pytest.mark.parametrize("split", [1, 4])
@pytest.mark.parametrize("batch", [3, 9, 40])
def test_convolution(batch, split, monkeypatch):
    monkeypatch.setenv("ONNXB_FP32", "4,%d" % split)
    rng = np.random.default_rng(batch)
    X, W = rng.standard_normal((batch, 12, 33, 31), dtype=np.float32), rng.standard_normal((40, 12, 3, 3), dtype=np.float32)
    binding.set_kernel_override("simt_direct")
    try:
        d = binding.Conv2dDesc(X.shape, W.shape, pads=(1,) * 4)
    finally:
        binding.set_kernel_override(None)
    got = d.run(torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda())
    want, S = oracle.conv2d(X, W, None, relu=False, pads=(1,) * 4)
    assert binding.last_device_status() == 0 and np.all(np.abs(got.cpu().numpy() - want) <= (108 + 8) * 2.0 ** -24 * 1.01 * S)
