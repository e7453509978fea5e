"""The small-image convolution at widths around a warp's share of lanes, images brought in by positions and (many blocks, rows of all
but whole warps) by rows, and for every number of channels per block, pinned and as the rule picks them; fp32 throughout."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2008_08272_b200 import binding  # noqa: E402

# (x, w, attributes): padded rows of 7 to 9, 15 to 17, 31 to 33 and 64 columns; one to many blocks; remainders of channels; groups, strides
CASES = [((n, c, h, wd), (m, c // kw.get("group", 1), k, k), kw) for n, c, h, wd, m, k, kw in (
    (1, 3, 5, 5, 5, 3, dict(pads=(1,) * 4)), (2, 2, 9, 8, 7, 3, {}), (3, 4, 6, 7, 16, 3, dict(pads=(1,) * 4)),
    (18, 8, 14, 14, 16, 5, dict(pads=(2,) * 4)), (39, 8, 14, 14, 16, 5, dict(pads=(2,) * 4)), (5, 8, 13, 11, 13, 5, dict(pads=(2,) * 4)),
    (40, 1, 28, 28, 8, 5, dict(pads=(2,) * 4)), (200, 1, 28, 28, 8, 5, dict(pads=(2,) * 4)), (4, 6, 30, 29, 9, 3, dict(pads=(1,) * 4, group=3)),
    (7, 2, 20, 64, 6, 4, dict(strides=(2, 1))), (300, 2, 9, 31, 3, 3, dict(pads=(1,) * 4, dilations=(2, 1))))]


@pytest.mark.parametrize("x,w,kw", CASES)
@pytest.mark.parametrize("addend", [False, True])
def test_small_conv(x, w, kw, addend, monkeypatch, pin="small"):
    monkeypatch.setenv("ONNXB_FP32", pin)
    rng = np.random.default_rng(x[0] + w[0])
    X, W, B = rng.standard_normal(x, dtype=np.float32), rng.standard_normal(w, dtype=np.float32), rng.standard_normal(w[0], dtype=np.float32)
    binding.set_kernel_override("simt_direct")
    try:
        d = binding.Conv2dDesc(x, w, has_bias=True, **kw)
    finally:
        binding.set_kernel_override(None)
    R = rng.standard_normal(d.y_shape, dtype=np.float32) if addend else None
    xt, wt, bt = (torch.from_numpy(v).cuda() for v in (X, W, B))
    got = d.run_add(xt, wt, bt, torch.from_numpy(R).cuda()) if addend else d.run(xt, wt, bt)
    want, S = oracle.conv2d(X, W, B, relu=False, **kw)
    if addend:
        want, S = want + R.astype(np.float64), S + np.abs(R)
    # one chain of fp32 additions of the window's terms, the bias and the addend
    bound = (W[0].size + 3) * 2.0 ** -24 * (S + np.abs(B).reshape(1, -1, 1, 1)) * 1.01
    assert binding.last_device_status() == 0 and np.all(np.abs(got.cpu().numpy() - want) <= bound)


# a quotient and a remainder of channels at every number per block; 3x3, 5x5 and other filters; one block, and several per SM
SIZES = [((n, c, h, wd), (m, c // kw.get("group", 1)) + k, kw) for n, c, h, wd, m, k, kw in (
    (2, 3, 9, 17, 21, (3, 3), dict(pads=(1,) * 4)), (70, 2, 12, 15, 37, (3, 3), dict(pads=(1,) * 4)), (3, 5, 14, 14, 19, (5, 5), dict(pads=(2,) * 4)),
    (80, 4, 10, 33, 34, (5, 5), dict(pads=(2,) * 4, group=2)), (2, 3, 11, 8, 18, (2, 4), {}), (90, 2, 13, 16, 23, (4, 3), dict(strides=(2, 1))),
    # by rows of 29, 32, 30 and 64, and by positions at 28 and 33 beside them
    (120, 2, 10, 27, 21, (3, 3), dict(pads=(1,) * 4)), (130, 1, 9, 28, 19, (5, 5), dict(pads=(2,) * 4)), (120, 3, 9, 30, 18, (2, 4), {}),
    (230, 1, 4, 64, 17, (3, 3), {}), (120, 2, 10, 26, 21, (3, 3), dict(pads=(1,) * 4)), (130, 1, 9, 29, 19, (5, 5), dict(pads=(2,) * 4)))]


@pytest.mark.parametrize("x,w,kw", SIZES)
@pytest.mark.parametrize("channels", [1, 4, 8, 16])
def test_every_number_of_channels_per_block(x, w, kw, channels, monkeypatch):
    test_small_conv(x, w, kw, False, monkeypatch, "small,%d" % channels)
