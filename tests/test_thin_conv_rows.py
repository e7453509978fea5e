"""Convolutions of few channels per group whose rows are staged one copy per channel: tiles inside one image and across two,
channels that end a block early, rows of any length, far pads, dilations; and an addend too large for L2, asked for ahead."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from parity import check_conv, worst_ratio  # noqa: E402

CASES = [((3, 3, 60, 62), (40, 3, 7, 7), dict(pads=(3, 3, 3, 3), strides=(2, 2))),
         ((2, 10, 52, 83), (70, 5, 3, 3), dict(pads=(1, 1, 1, 1), group=2)),
         ((3, 13, 36, 41), (24, 13, 3, 3), dict(pads=(9, 0, 2, 11))),
         ((1, 6, 68, 31), (33, 6, 3, 5), dict(pads=(2, 4, 2, 4), dilations=(2, 3))),
         ((2, 4, 101, 36), (40, 4, 5, 5), dict(pads=(2, 2, 2, 2), strides=(3, 1))),
         ((2, 9, 64, 64), (300, 9, 2, 3), dict(strides=(1, 2)))]


def _operands(xs, ws):
    rng = np.random.default_rng(xs[1] + ws[0])
    W = (rng.standard_normal(ws) * np.sqrt(2.0 / (ws[1] * ws[2] * ws[3]))).astype(np.float32)
    return rng.standard_normal(xs).astype(np.float32), W, rng.standard_normal((ws[0],)).astype(np.float32)


@pytest.mark.parametrize("tile", [None, "1,1,32", "2,2,48"])
@pytest.mark.parametrize("xs,ws,kw", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else "")
def test_thin_rows(xs, ws, kw, tile, monkeypatch):
    from paper_2008_08272_b200 import binding
    if tile:
        monkeypatch.setenv("ONNXB_CONV_TILE", tile)
    binding.set_kernel_override("mma_implicit")             # whatever their size
    try:
        ratio, family = check_conv(binding, torch, *_operands(xs, ws), relu=True, **kw)
    finally:
        binding.set_kernel_override(None)
    assert family == "mma_implicit" and ratio <= 1.0


@pytest.mark.parametrize("tile", [None, "1,1,32", "2,2,32"])
@pytest.mark.parametrize("xs,ws,pads", [((1, 1, 1, 20000), (64, 1, 1, 33), (0, 16, 0, 50000)), ((2, 8, 2, 2000), (16, 8, 1, 25), (0, 0, 0, 64000)),
                                        ((1, 4, 1, 2000), (16, 4, 1, 9), (0, 4, 0, 63536))], ids=str)
def test_slot_rows_of_65536_and_more(xs, ws, pads, tile, monkeypatch):
    """Padding at the end of the rows that makes a slot row longer than 16 bits count."""
    from paper_2008_08272_b200 import binding
    if tile:
        monkeypatch.setenv("ONNXB_CONV_TILE", tile)
    binding.set_kernel_override("mma_implicit")
    try:
        ratio, family = check_conv(binding, torch, *_operands(xs, ws), pads=pads)
    finally:
        binding.set_kernel_override(None)
    assert family == "mma_implicit" and ratio <= 1.0


@pytest.mark.parametrize("xs,ws", [((3, 8, 472, 500), (24, 8, 3, 3)), ((6, 16, 240, 180), (65, 16, 3, 3))])
def test_far_addend(xs, ws):
    from paper_2008_08272_b200 import binding
    X, W, B = _operands(xs, ws)
    d = binding.Conv2dDesc(xs, ws, pads=(1, 1, 1, 1), has_bias=True, fuse_relu=True)
    assert d.kernel_family == "mma_implicit" and np.prod(d.y_shape) * 4 >= 64 << 20
    R = torch.randn(d.y_shape, generator=torch.Generator().manual_seed(1))
    got = d.run_add(*(torch.from_numpy(t).cuda() for t in (X, W, B)), R.cuda()).cpu().numpy()
    assert binding.last_device_status() == 0
    want, S = oracle.conv2d(X, W, B, pads=(1, 1, 1, 1))
    R = R.numpy()
    assert worst_ratio(got, np.maximum(want + R, 0), S + np.abs(R)) <= 1.0
