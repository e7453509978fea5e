"""Channel-major tensors ([channel][image][row][column], channels padded to whole lines) between layers: the same convolutions."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from parity import worst_ratio
from paper_2008_08272_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Every slot of every tile finds its pixel in the range of pixels that the tile stages, which begins on a 16-byte boundary, and no
# tile's range is longer than that of the starts by which a plan sizes its stages.
RANGES = r"""
#include <algorithm>
#include <cstdio>
#include "tc_conv_plan.h"
using namespace onnxb;
static int check(int N, int H, int W, int k, int pad, int s, int tile, int boxp) {
    TcConvPlan g{};
    const int P = (H + 2 * pad - k) / s + 1, Q = (W + 2 * pad - k) / s + 1;
    ConvAxis ah, aw;
    if (!conv_plan_axis(H, P, pad, s, 1, k, ah) || !conv_plan_axis(W, Q, pad, s, 1, k, aw)) return 0;
    g.N = N; g.H = H; g.W = W; g.P = P; g.Q = Q; g.pt = g.pl = pad; g.sh = g.sw = s;
    g.Hs = ah.E; g.Ws = aw.E; g.L = g.Hs * g.Ws; g.total_slots = (long long)N * g.L;
    g.a_min = ah.par[0]; g.a_max = ah.par[ah.npar - 1];
    g.SLOTS = tile + ah.Amax * g.Ws + aw.Amax; g.x_cm = 1; g.BOXP = boxp; g.KBR = 16;
    if ((g.SLOTS + g.L - 2) / g.L + 1 > kConvMaxSeg) return 0;
    int sized = 0;
    for (int n = 0; n < std::min(N, 4); ++n)
        for (int r = 0; r < g.Hs; ++r) {
            TcConvSegs t;
            tc_conv_segments(g, std::min<long long>(n * (long long)g.L + r * g.Ws + g.Ws - 1, g.total_slots - 1), t);
            sized = std::max(sized, t.total_floats);
        }
    for (long long G0 = 0; G0 < g.total_slots; ++G0) {
        TcConvSegs t;
        tc_conv_segments(g, G0, t);
        if (t.total_floats > sized) return std::printf("tile at %lld stages %d floats, sized for %d\n", G0, t.total_floats, sized), 1;
        int boxes = 0;
        for (int i = 0; i < t.nseg; ++i) boxes += t.nbox[i];
        if (t.nseg && boxes != t.nbox[0]) return std::printf("copies outside the first segment\n"), 1;
        const long long start = (long long)t.n_first * H * W + t.f0[0];
        if (boxes && (start % 4 != 0 || start < 0)) return std::printf("range from %lld\n", start), 1;
        for (int pl = 0; pl < ah.npar * aw.npar; ++pl)
            for (int j = 0; j < g.SLOTS && G0 + j < g.total_slots; ++j) {
                const long long G = G0 + j;
                const int n = (int)(G / g.L), u = (int)(G % g.L), kk = n - t.n_first;
                const int h = u / g.Ws * s + ah.par[pl / aw.npar] - pad, w = u % g.Ws * s + aw.par[pl % aw.npar] - pad;
                if (h < 0 || h >= H || w < 0 || w >= W) continue;
                const int f = h * W + w - t.f0[kk];
                if (kk >= t.nseg || t.base[kk] != 0 || f < 0 || f >= t.nbox[0] * boxp || start + f != ((long long)n * H + h) * W + w)
                    return std::printf("slot %lld of the tile at %lld\n", G, G0), 1;
            }
    }
    return 0;
}
int main() {
    for (int N : {1, 2, 3, 5, 9})
        for (int hw = 0; hw < 6; ++hw) {
            const int H[] = {7, 14, 5, 9, 28, 6}, W[] = {7, 14, 11, 6, 28, 33};
            for (int s : {1, 2})
                for (int pad : {0, 1, 3})
                    for (int tile : {128, 256})
                        for (int boxp : {4, 100, 256})
                            if (check(N, H[hw], W[hw], pad == 3 ? 5 : 3, pad, s, tile, boxp)) return std::printf("%d images %dx%d stride %d pad %d tile %d\n", N, H[hw], W[hw], s, pad, tile), 1;
        }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_ranges_hold_every_pixel(tmp_path):
    (tmp_path / "t.cpp").write_text(RANGES)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_2008_08272_b200", "csrc"), str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True)
    run = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout + run.stderr


def test_descriptors():
    for (x, w, kw), fine in (
            (((2, 64, 7, 7), (96, 64, 1, 1), {}), True), (((2, 64, 7, 7), (96, 64, 3, 3), dict(pads=(1,) * 4)), True),
            (((2, 64, 8, 8), (96, 64, 1, 1), dict(strides=(2, 2))), False), (((2, 64, 7, 7), (64, 1, 3, 3), dict(group=64)), False),
            (((2, 3, 64, 64), (64, 3, 7, 7), {}), False), (((2, 24, 7, 7), (96, 24, 1, 1), {}), True)):
        if fine:
            d = binding.Conv2dDesc(x, w, x_channel_major=True, y_channel_major=True, **kw)
            assert d.kernel_family in ("mma_gemm", "mma_implicit") and d.y_storage == (96, binding.channel_pitch(d.y_shape), 1, 1)
        else:
            with pytest.raises(binding.OnnxB200Error) as e:
                binding.Conv2dDesc(x, w, x_channel_major=True, y_channel_major=True, **kw)
            assert e.value.status == 4
    assert binding.channel_pitch((1, 5, 7, 7)) == 64 and binding.channel_pitch((64, 5, 14, 14)) == 64 * 196


# x, w, attributes: tiles of several odd images, pairs and single CTAs, split reductions, strides, groups, channels that fill no block;
# 1x1 layers as wide GEMMs of few and of many columns
CONVS = [((1, 64, 7, 7), (96, 64, 3, 3), dict(pads=(1,) * 4)), ((5, 72, 7, 7), (80, 72, 3, 3), dict(pads=(1,) * 4)),
         ((64, 128, 7, 7), (128, 128, 3, 3), dict(pads=(1,) * 4)), ((3, 64, 14, 14), (64, 64, 3, 3), dict(pads=(1,) * 4, strides=(2, 2))),
         ((9, 64, 13, 11), (48, 32, 5, 3), dict(pads=(2, 1, 2, 1), group=2)), ((32, 64, 56, 56), (64, 64, 3, 3), dict(pads=(1,) * 4)),
         ((1, 256, 14, 14), (256, 256, 3, 3), dict(pads=(1,) * 4)), ((2, 40, 9, 10), (24, 40, 3, 3), dict(dilations=(2, 2))),
         ((1, 512, 7, 7), (256, 512, 1, 1), {}), ((3, 96, 7, 7), (80, 96, 1, 1), {}), ((64, 512, 7, 7), (512, 512, 1, 1), {}),
         ((16, 128, 14, 14), (256, 128, 1, 1), {}), ((2, 64, 56, 56), (256, 64, 1, 1), {})]


def _channel_major(t):
    """A channel-major copy; what lies between the channels is NaN."""
    import torch
    n, c, h, w = t.shape
    s = torch.full((c, binding.channel_pitch(t.shape)), float("nan"), device=t.device)
    s[:, :n * h * w] = t.transpose(0, 1).reshape(c, -1)
    return s


def _nchw(s, shape):
    n, c, h, w = shape
    return s.view(c, -1)[:, :n * h * w].reshape(c, n, h, w).transpose(0, 1)


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [(True, True), (True, False), (False, True)], ids=["both", "x", "y"])
@pytest.mark.parametrize("x,w,kw", CONVS)
def test_convolutions(x, w, kw, layout):
    import torch
    rng = np.random.default_rng(x[1] + w[0])
    try:
        d = binding.Conv2dDesc(x, w, has_bias=True, fuse_relu=True, x_channel_major=layout[0], y_channel_major=layout[1], **kw)
    except binding.OnnxB200Error:
        assert not layout[0] and x[2] * x[3] % 4 != 0           # (planes that TMA cannot address)
        return
    X, W, B = rng.random(x, dtype=np.float32), rng.standard_normal(w, dtype=np.float32), rng.standard_normal(w[0], dtype=np.float32)
    R = rng.standard_normal(d.y_shape, dtype=np.float32)
    xt, wt, bt, rt = (torch.from_numpy(v).cuda() for v in (X, W, B, R))
    packed = d.prepack(wt)
    lay = lambda t, cm: _channel_major(t) if cm else t
    conv, S = oracle.conv2d(X, W, B, relu=False, **kw)
    for addend in (None, R):
        got = d.run_prepacked(lay(xt, layout[0]), wt, packed, bt, None if addend is None else lay(rt, layout[1]))
        got = _nchw(got, d.y_shape) if layout[1] else got
        want = np.maximum(conv if addend is None else conv + R.astype(np.float64), 0.0)
        assert worst_ratio(got.cpu().numpy(), want, S) <= 1.0
    assert binding.last_device_status() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("x,w,kw", [c for c in CONVS if c[0][1] >= 16])
def test_rounded_outputs(x, w, kw):
    """The second output of a 1x1 layer with an addend, and the other layers' output itself."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    d = binding.Conv2dDesc(x, w, has_bias=True, x_channel_major=True, y_channel_major=True, **kw)
    X, W, B, R = (torch.randn(s, generator=g, device="cuda") for s in (x, w, (w[0],), d.y_shape))
    packed, X = d.prepack(W), _channel_major(X)
    R = _channel_major(R) if d.kernel_family == "mma_gemm" else None
    want = d.run_prepacked(X, W, packed, B, R)
    y = torch.empty_like(want)
    yr = torch.empty_like(want) if R is not None else y
    d.run_prepacked_rounded(X, W, packed, B, R, y, yr)
    assert binding.last_device_status() == 0
    want, y, yr = (_nchw(t, d.y_shape) for t in (want, y, yr))
    if R is not None:
        assert torch.equal(y, want)
    assert torch.equal(yr, ((want.contiguous().view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("given", [True, False])
@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("x,w,strides", [((3, 64, 28, 28), (96, 64, 1, 1), (2, 2)), ((5, 96, 7, 7), (80, 96, 1, 1), (1, 1))])
def test_rounded_outputs_behind_a_gather(x, w, strides, native, given, monkeypatch):
    """The copy of the pixels needs a workspace beside the packed weights, the caller's or one made for the call."""
    import torch
    if not native:
        monkeypatch.setattr(binding, "_fast_mod", binding._Declined())
    g = torch.Generator(device="cuda").manual_seed(3)
    d = binding.Conv2dDesc(x, w, has_bias=True, strides=strides)
    assert d.kernel_family == "mma_gather_gemm"
    X, W, B, R = (torch.randn(s, generator=g, device="cuda") for s in (x, w, (w[0],), d.y_shape))
    packed = d.prepack(W)
    want = d.run_prepacked(X, W, packed, B, R)
    y, yr = torch.empty_like(want), torch.empty_like(want)
    d.run_prepacked_rounded(X, W, packed, B, R, y, yr, workspace=torch.empty(d.workspace_bytes, dtype=torch.uint8, device="cuda") if given else None)
    assert binding.last_device_status() == 0 and torch.equal(y, want)
    assert torch.equal(yr, ((want.view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("batch,C,M,hw,strides", [(4, 64, 256, (56, 56), (2, 2)), (3, 128, 512, (27, 28), (2, 2)), (1, 256, 1024, (14, 14), (2, 2)),
                                                  (64, 64, 272, (13, 14), (2, 2))])
def test_sampled_addend(batch, C, M, hw, strides, native, monkeypatch):
    import torch
    if not native:
        monkeypatch.setattr(binding, "_fast_mod", binding._Declined())
    g = torch.Generator(device="cuda").manual_seed(2)
    p, q = (-(-s // t) for s, t in zip(hw, strides))
    X, W, B, R = (torch.randn(s, generator=g, device="cuda") for s in ((batch, C, p, q), (M, C, 1, 1), (M,), (batch, M) + hw))
    d = binding.Conv2dDesc(X.shape, W.shape, has_bias=True, fuse_relu=True, x_channel_major=True, y_channel_major=True)
    packed, X = d.prepack(W), _channel_major(X)
    want = d.run_prepacked(X, W, packed, B, _channel_major(R[:, :, ::strides[0], ::strides[1]]))
    yr = torch.empty_like(want)
    got = d.run_prepacked_sampled(X, W, packed, B, _channel_major(R), strides, Y_rounded=yr, r_dims=hw)
    assert binding.last_device_status() == 0
    want, got, yr = (_nchw(t, d.y_shape) for t in (want, got, yr))
    # the reduction may be split another way: two sums of C products in fp32, each addition off by 2^-23 of the sum of magnitudes
    S = torch.nn.functional.conv2d(_nchw(X, (batch, C, p, q)).abs(), W.abs()) + B.abs().view(1, -1, 1, 1) + R[:, :, ::strides[0], ::strides[1]].abs()
    assert bool(((got - want).abs() <= 2 * (C + 2) * 2.0 ** -23 * S).all())
    assert torch.equal(yr, ((got.contiguous().view(torch.int32) + 0x1000) & ~0x1FFF).view(torch.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1, 96, 7, 7), (5, 33, 14, 14), (64, 48, 3, 5)])
def test_global_average_pool(shape):
    import torch
    X = torch.rand(shape, device="cuda")
    Y = torch.empty(shape[:2] + (1, 1), device="cuda")
    binding.global_average_pool_channel_major(_channel_major(X), shape, Y)
    assert torch.equal(Y, binding.onnx_global_average_pool(X))
