"""The depthwise kernel of one column per thread: row and column strides and dilations of their own, planes of fewer rows
than a thread owns, dilations beyond the image, ragged columns, a residual addend; and the planes of odd rows that it shares
with the kernel of column strips, on both sides of the rule between them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

REL = 2e-6          # of sum |x*w|: 25 products, their sum, a bias and an addend, 2^-24 each

CASES = [dict(x=(2, 7, 17, 19), k=3, strides=(2, 2), pads=(1, 1, 1, 1)), dict(x=(1, 5, 30, 33), k=5, strides=(2, 1), pads=(2, 0, 1, 2)),
         dict(x=(3, 4, 29, 21), k=3, strides=(1, 2), dilations=(3, 2), pads=(3, 2, 3, 2)),
         dict(x=(1, 3, 26, 40), k=5, dilations=(2, 4), pads=(4, 8, 4, 8)), dict(x=(2, 2, 5, 3), k=3, dilations=(7, 1), pads=(7, 1, 9, 1)),
         dict(x=(1, 6, 1, 5), k=3, pads=(1, 1, 1, 1)), dict(x=(80, 40, 37, 41), k=3, strides=(2, 2), pads=(1, 1, 1, 1)),
         dict(x=(64, 33, 45, 47), k=3, pads=(1, 1, 1, 1)), dict(x=(33, 16, 45, 47), k=3, pads=(1, 1, 1, 1)),
         dict(x=(2, 2, 4, 9), k=3, dilations=(90, 1), pads=(90, 1, 90, 1)), dict(x=(20, 8, 50, 61), k=5, pads=(2, 2, 2, 2))]


@pytest.mark.parametrize("c", CASES, ids=lambda c: "x".join(map(str, c["x"])) + "k%d" % c["k"])
def test_columns(c):
    from paper_2008_08272_b200 import binding
    rng = np.random.default_rng(c["x"][1])
    C, kw = c["x"][1], dict(pads=c["pads"], strides=c.get("strides", (1, 1)), dilations=c.get("dilations", (1, 1)), group=c["x"][1])
    X, W, B = (rng.standard_normal(s).astype(np.float32) for s in (c["x"], (C, 1, c["k"], c["k"]), (C,)))
    d = binding.Conv2dDesc(X.shape, W.shape, has_bias=True, fuse_relu=True, **kw)
    assert d.kernel_family == "simt_depthwise"
    R = rng.standard_normal(d.y_shape).astype(np.float32)
    dev = [torch.from_numpy(t).cuda() for t in (X, W, B, R)]
    want, S = oracle.conv2d(X, W, B, **kw)
    for add in (0, R):
        got = (d.run(*dev[:3]) if isinstance(add, int) else d.run_add(*dev)).cpu().numpy()
        assert (np.abs(got - np.maximum(want + add, 0)) <= REL * (S + np.abs(add)) + 1e-6).all()
