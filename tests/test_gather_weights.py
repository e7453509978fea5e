"""1x1 convolutions behind a gather with weights of the call, which the gather rounds: more weights than pixels and fewer, one
turn of the blocks and several."""
import numpy as np
import pytest

import oracle
from parity import worst_ratio

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2008_08272_b200 import binding  # noqa: E402


def _desc(x, m, s):
    d = binding.Conv2dDesc(x, (m, x[1], 1, 1), strides=(s, s), has_bias=True)
    assert d.kernel_family == "mma_gather_gemm"
    return d


# images merged or not, rows by pieces of 16 bytes or not; weights: one turn's share of a block, of many blocks, more than all blocks at once
@pytest.mark.parametrize("x,m,s", [((1, 32, 5, 5), 16, 2), ((1, 64, 9, 9), 2048, 1), ((1, 1024, 14, 14), 1024, 2), ((1, 2048, 7, 7), 1024, 2),
                                   ((2, 1280, 3, 3), 1284, 1), ((1, 640, 28, 28), 2048, 2), ((3, 96, 56, 48), 80, 2)])
def test_values(x, m, s):
    rng = np.random.default_rng(m + x[1])
    X, W, B = rng.random(x, dtype=np.float32), rng.standard_normal((m, x[1], 1, 1), dtype=np.float32), rng.standard_normal(m, dtype=np.float32)
    d = _desc(x, m, s)
    xt, wt, bt = (torch.from_numpy(v).cuda() for v in (X, W, B))
    got = d.run(xt, wt, bt)
    assert torch.equal(got, d.run_prepacked(xt, wt, d.prepack(wt), bt)) and binding.last_device_status() == 0
    want, S = oracle.conv2d(X, W, B, strides=(s, s))
    assert worst_ratio(got.cpu().numpy(), want, S) <= 1.0


@pytest.mark.parametrize("x,m,s", [((1, 512, 7, 7), 2048, 1), ((1, 1024, 14, 14), 2048, 2), ((1, 2048, 7, 7), 2048, 2)])
def test_no_longer_than_with_a_launch_for_the_weights(x, m, s):
    """By the pixels' blocks alone the weights took 15 to 35 us where a launch of their own in front takes some 3."""
    d = _desc(x, m, s)
    X, W, B, Y = torch.rand(x, device="cuda"), torch.randn(m, x[1], 1, 1, device="cuda"), torch.randn(m, device="cuda"), torch.empty(d.y_shape, device="cuda")
    ws, packed = torch.empty(d.workspace_bytes, dtype=torch.uint8, device="cuda"), d.prepack(W)

    def two():
        binding._check(d._lib.onnx_conv2d_prepack(d._h, W.data_ptr(), packed.data_ptr(), packed.numel(), torch.cuda.current_stream().cuda_stream), "prepack")
        d.run_prepacked(X, W, packed, B, Y=Y, workspace=ws)

    def us(f):
        best = float("inf")
        for _ in range(6):                                 # (the first warms up)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(50):
                f()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 20)
        return best
    assert us(lambda: d.run(X, W, B, Y=Y, workspace=ws)) <= 1.25 * us(two)
