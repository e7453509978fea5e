"""ResNet-50 v1 as one chained run of the library's operators (Sec. 4.2 times this model end to end).

The graph is the ONNX Model Zoo ResNet50 with batch normalisation folded into the convolutions (as
an inference compiler's constant propagation leaves it, Sec. 3.4.4): stem Conv 7x7/2 + Relu,
MaxPool 3x3/2, sixteen bottleneck blocks (1x1 -> 3x3 -> 1x1, stride on the first 1x1 of a
down-sampling block and on its 1x1 projection), each closed by Add + Relu fused into the last 1x1
convolution, GlobalAveragePool, Gemm 2048 -> 1000.  Weights are synthetic (He-normal, seeded): the
model file is not available offline.  Only marshalling and buffer bookkeeping happen here; every
operator runs in the library's kernels.
"""
from __future__ import annotations

from dataclasses import dataclass, replace
from typing import Dict, List, Optional

import numpy as np

from . import binding
from . import workloads as wl


@dataclass
class Op:
    kind: str                 # "conv" | "conv_add" | "maxpool" | "gap" | "gemm"
    name: str
    src: str                  # name of the input tensor
    dst: str                  # name of the output tensor
    res: Optional[str] = None  # residual addend (conv_add)
    case: Optional[wl.ConvCase] = None
    relu: bool = False
    sampled: Optional[str] = None  # conv_add: `res` is every so-many-th row and column of this tensor
    sample: tuple = (1, 1)


def build_graph(batch: int) -> List[Op]:
    """The operator list in execution order, wired by tensor names."""
    convs = wl.resnet50_v1_convs(batch)
    ops: List[Op] = [Op("conv", convs[0].name, "input", "stem", case=convs[0], relu=True),
                     Op("maxpool", "pool1", "stem", "pool1")]
    cur, i = "pool1", 1
    while i < len(convs):
        a, b3, c1 = convs[i], convs[i + 1], convs[i + 2]
        has_proj = i + 3 < len(convs) and convs[i + 3].name.endswith("_proj")
        blk = a.name[:-5]                                  # e.g. r50_01_s2b0
        ops.append(Op("conv", a.name, cur, blk + "_a", case=a, relu=True))
        ops.append(Op("conv", b3.name, blk + "_a", blk + "_b", case=b3, relu=True))
        shortcut = cur
        if has_proj:
            pj = convs[i + 3]
            ops.append(Op("conv", pj.name, cur, blk + "_sc", case=pj, relu=False))
            shortcut = blk + "_sc"
        ops.append(Op("conv_add", c1.name, blk + "_b", blk + "_out", res=shortcut, case=c1, relu=True))
        cur = blk + "_out"
        i += 4 if has_proj else 3
    ops.append(Op("gap", "gap", cur, "pooled"))
    ops.append(Op("gemm", "fc", "pooled", "logits"))
    return ops


def push_strides_up(ops: List[Op]) -> List[Op]:
    """The same model with the stride of 1x1 convolutions moved to what produces their input.

    A tensor that only unpadded, strided 1x1 convolutions read is needed at the places these read and nowhere else: the last
    block of a stage, whose output the next stage's two strided layers read.  So its producer computes those places alone, and
    the readers, of unit stride now, get the same values (rounded to TF32, as a strided one's gather does it); a producer that
    is a 1x1 convolution itself is in turn a strided one, and so on up.  The residual addend of such a producer is read at
    those places (its other reader, the block's first convolution, needs all of it).  Per stage boundary a 3x3 layer and the
    widest 1x1 layer of the stage, with its addend, on a fourth of the pixels, and no gathering of every other pixel for the
    two readers: 64 images 2036 -> 1883 us; one image 402 either way, its layers being bound by their launches' latency.  The
    logits' error against float64 (2-norm, relative, mean of six networks at one image) is 2.2e-3, 2.3e-3 before."""
    ops = [replace(op) for op in ops]
    for op in reversed(ops):
        if op.kind not in ("conv", "conv_add"):
            continue
        readers = [o for o in ops if op.dst in (o.src, o.res, o.sampled)]
        strides = {o.case.strides if o.case is not None and op.dst not in (o.res, o.sampled) and tuple(o.case.w_shape[2:]) == (1, 1) and
                   o.case.pads == (0, 0, 0, 0) and o.case.group == 1 else (1, 1) for o in readers}
        if len(strides) != 1 or strides == {(1, 1)}:
            continue
        s = strides.pop()
        op.case = replace(op.case, strides=(op.case.strides[0] * s[0], op.case.strides[1] * s[1]))
        if op.kind == "conv_add":
            op.sampled, op.sample, op.res = op.res, s, "%s::%d,%d" % (op.res, *s)
        for o in readers:
            o.case = replace(o.case, x_shape=op.case.y_shape, strides=(1, 1))
    return ops


def pass_flops(ops: List[Op]) -> int:
    """Operations of the convolutions and the classifier of a graph, as its operators compute them."""
    return sum(op.case.flops for op in ops if op.case is not None) + 2 * ops[0].case.x_shape[0] * 2048 * 1000


class Resnet50Chain:
    """The model with its buffers.  Between the layers tensors are channel-major: a channel's pixels of all images in one row, rows
    of whole 128-byte lines.  A 1x1 layer is then one wide GEMM whatever the images' size (7x7 planes are no whole 16-byte pieces,
    14x14 ones no whole lines), and no layer's input is gathered: 64 images 1883 -> 1743 us, one image 402 -> 388.

    ``buf`` shows them as the ONNX tensors that they are, those that only strided 1x1 layers read at the places read
    (``push_strides_up``).  A tensor put in another's place there is what the operator writes from then on.  Where it is not one of
    the last two, ``pooled`` and ``logits``, the chain is laid out anew for it, as ONNX lays out the graph and every tensor (so from
    the beginning with ``prepack`` off), and the other entries are new tensors, too; inside a capture that raises an error."""

    def __init__(self, batch: int, device, seed: int = wl.SEED_BASE + 9000, prepack: bool = True):
        import torch
        self.torch = torch
        self.batch, self.dev = batch, device
        graph = build_graph(batch)
        rng = np.random.default_rng(seed)
        self.prepack = prepack                  # weights are constants of the graph: pack them once (Sec. 3.4.4)
        self.params: Dict[str, tuple] = {}
        for op in graph:
            if op.case is not None:
                c = op.case
                fan = c.w_shape[1] * c.w_shape[2] * c.w_shape[3]
                W = (rng.standard_normal(c.w_shape, dtype=np.float32) * np.float32(np.sqrt(2.0 / fan)))
                if op.kind == "conv_add":
                    W *= np.float32(0.5)                   # keeps the activations of 16 stacked blocks in range
                B = rng.standard_normal((c.w_shape[0],), dtype=np.float32) * np.float32(0.01)
                self.params[op.name] = (torch.from_numpy(W).to(device), torch.from_numpy(B).to(device))
        Wf = rng.standard_normal((2048, 1000), dtype=np.float32) * np.float32(np.sqrt(1.0 / 2048))
        Bf = rng.standard_normal((1000,), dtype=np.float32) * np.float32(0.01)
        self.params["fc"] = (torch.from_numpy(Wf).to(device), torch.from_numpy(Bf).to(device))
        self.fc_workspace = torch.empty(max(binding.gemm_workspace_bytes(False, False, batch, 1000, 2048), 16),
                                        dtype=torch.uint8, device=device)
        self.buf: Dict[str, "torch.Tensor"] = {}
        self._lay_out(prepack, {})
        self.flops = pass_flops(graph)          # the model's; of a pass as it is run: pass_flops(self.ops)
        self._capture()

    def _lay_out(self, channel_major: bool, given: Dict[str, "torch.Tensor"]):
        """The operators, their descriptors, packed weights and buffers, on channel-major tensors where every layer knows them;
        ``given``: tensors of ``buf`` to use as they are."""
        torch = self.torch
        graph = build_graph(self.batch)
        self.ops, self.descs, self.channel_major = graph, None, False
        if channel_major:
            moved = push_strides_up(graph)
            self.descs = self._descriptors(moved, True)
            if self.descs is not None:
                self.ops, self.channel_major = moved, True
        if self.descs is None:                  # (a kernel family pinned by the override knows one layout)
            self.descs = self._descriptors(graph, False)
        # What a gather would round to TF32 for the tensor cores reaches them rounded, not truncated.
        self._reads_rounded = {op.src for ops in (graph, self.ops) for op in ops if self._gathers(op)} if self.channel_major else set()
        self.packed: Dict[str, object] = {}
        if self.prepack:
            self.packed = {name: d.prepack(self.params[name][0]) for name, d in self.descs.items()}
        ws_bytes = max([16] + [d.workspace_bytes for d in self.descs.values()])
        self.workspace = torch.empty(ws_bytes, dtype=torch.uint8, device=self.dev)
        # one buffer per tensor of the graph, as it lies in memory and as the ONNX tensor it is; and the rounded second outputs
        self.store: Dict[str, "torch.Tensor"] = {}
        self.buf.clear()
        self.rounded: Dict[str, "torch.Tensor"] = {}
        shapes: Dict[str, tuple] = {}
        for op in self.ops:
            if op.case is not None:
                shape = self.descs[op.name].y_shape
                if op.sampled:
                    self.buf[op.res] = self.buf[op.sampled][:, :, ::op.sample[0], ::op.sample[1]]
            elif op.kind == "maxpool":
                shape = binding.maxpool2d_shape(shapes[op.src], (3, 3), (1, 1, 1, 1), (2, 2))
            elif op.kind == "gap":
                shape = shapes[op.src][:2] + (1, 1)
            else:
                shape = (self.batch, 1000)
            shapes[op.dst] = shape
            if self.channel_major and op.kind in ("conv", "conv_add", "maxpool"):
                n, c, h, w = shape
                self.store[op.dst] = torch.empty((c, binding.channel_pitch(shape)), dtype=torch.float32, device=self.dev)
                self.buf[op.dst] = self.store[op.dst].as_strided(shape, (h * w, self.store[op.dst].shape[1], w, 1))
                if op.kind == "conv_add" and op.dst in self._reads_rounded:
                    self.rounded[op.dst] = torch.empty_like(self.store[op.dst])
            else:
                t = given[op.dst] if op.dst in given else torch.empty(shape, dtype=torch.float32, device=self.dev)
                self.store[op.dst] = self.buf[op.dst] = t
        # where the views lie: an entry of buf that lies elsewhere is another tensor, put in a view's place
        self._views = {name: self._place(t) for name, t in self.buf.items() if name in self.store and self.store[name] is not t}

    def _descriptors(self, ops: List[Op], channel_major: bool):
        """The convolutions' descriptors; None where one of them knows no channel-major tensors."""
        descs: Dict[str, binding.Conv2dDesc] = {}
        for op in ops:
            if op.case is not None:
                c = op.case
                try:
                    descs[op.name] = binding.Conv2dDesc(c.x_shape, c.w_shape, pads=c.pads, strides=c.strides, has_bias=True,
                                                        fuse_relu=op.relu, x_channel_major=channel_major and op.src != "input",
                                                        y_channel_major=channel_major)
                except binding.OnnxB200Error as e:
                    if not channel_major or e.status != 4:
                        raise
                    for d in descs.values():
                        d.close()
                    return None
        return descs

    @staticmethod
    def _gathers(op: Op) -> bool:
        """Whether a layer of the graph as ONNX has it, on tensors as ONNX lays them out, gathers (and rounds) its input."""
        if op.case is None or tuple(op.case.w_shape[2:]) != (1, 1):
            return False
        d = binding.Conv2dDesc(op.case.x_shape, op.case.w_shape, pads=op.case.pads, strides=op.case.strides)
        family = d.kernel_family
        d.close()
        return family == "mma_gather_gemm"

    @staticmethod
    def _place(t):
        return t.data_ptr(), t.dtype, t.shape, t.stride()

    def _state(self):
        """Where all tensors but the input lie and how, and what the library chooses its kernels by (None without the native call
        path): what the graph was captured with, and what a replay of it stands for."""
        state = binding.call_state(self.store, self.buf, self.rounded, self.packed, self.params, self.workspace, self.fc_workspace)
        return None if state is None else (self.prepack, state)

    def _follow_buf(self):
        """Goes over to the tensors that ``buf`` holds now, and to ``prepack`` as it is now."""
        if self.channel_major and (not self.prepack or any(self._place(self.buf[k]) != place for k, place in self._views.items())):
            if self.torch.cuda.is_current_stream_capturing():
                raise RuntimeError("Resnet50Chain: an entry of buf was replaced; its buffers are made anew by a pass outside a capture")
            self.torch.cuda.synchronize(self.dev)      # (a pass on another stream may still use what is let go here)
            x, descs = self.buf["input"], self.descs
            self._graph = self._captured = None
            self._lay_out(False, {k: t for k, t in self.buf.items() if k not in self._views or self._place(t) != self._views[k]})
            self.buf["input"] = self.store["input"] = x
            for d in descs.values():
                d.close()
        for op in self.ops:
            if op.dst not in self._views:
                self.store[op.dst] = self.buf[op.dst]

    def _capture(self):
        """The operators behind the first one, which alone reads the caller's tensor, as one CUDA graph."""
        torch = self.torch
        with torch.cuda.device(self.dev):
            self._device = torch.cuda.current_device()
            stream, before = torch.cuda.Stream(), binding.launch_count()
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                self.store["input"] = torch.zeros((self.batch, 3, 224, 224), device=self.dev)
                self._run(self.ops)                 # (what a first launch sets up is set up before the capture)
                del self.store["input"]
                self.launches = binding.launch_count() - before
                # (begun and ended by hand: the context manager also collects garbage and empties the allocator's cache)
                graph = torch.cuda.CUDAGraph()
                graph.capture_begin(capture_error_mode="thread_local")
                try:
                    self._run(self.ops[1:])
                finally:
                    graph.capture_end()
            torch.cuda.current_stream().wait_stream(stream)
        self._graph, self._captured = graph, self._state()

    def forward(self, x):
        """Enqueue the whole model on the current stream; returns the logits buffer.  (``binding.launch_count`` counts the one kernel
        launched beside the graph; ``launches`` is how many a pass has.)"""
        self.buf["input"] = self.store["input"] = x
        # All but the first operator in one launch in place of some fifty.  Made one by one where the call is itself being captured or
        # on another device, or where anything differs from what the graph was captured with.
        cuda = self.torch.cuda
        state = None if self._graph is None or cuda.is_current_stream_capturing() or cuda.current_device() != self._device else self._state()
        if state is None or state != self._captured:
            self._follow_buf()
            self._run(self.ops)
        else:
            self._run(self.ops[:1])
            self._graph.replay()
        return self.buf["logits"]

    def _run(self, ops: List[Op]):
        for op in ops:
            src, dst = self.store[op.src], self.store[op.dst]
            if op.kind in ("conv", "conv_add") and self.channel_major:
                d, (W, B), packed = self.descs[op.name], self.params[op.name], self.packed[op.name]
                src = self.rounded.get(op.src, src)
                if op.sampled:
                    d.run_prepacked_sampled(src, W, packed, B, self.store[op.sampled], op.sample, Y=dst, Y_rounded=self.rounded.get(op.dst),
                                            r_dims=self.buf[op.sampled].shape[2:])
                elif op.dst in self._reads_rounded:
                    d.run_prepacked_rounded(src, W, packed, B, self.store[op.res] if op.res else None, dst, self.rounded.get(op.dst, dst))
                else:
                    d.run_prepacked(src, W, packed, B, self.store[op.res] if op.res else None, Y=dst, workspace=self.workspace)
            elif op.kind in ("conv", "conv_add") and self.prepack:
                W, B = self.params[op.name]
                R = self.buf[op.res] if op.kind == "conv_add" else None
                self.descs[op.name].run_prepacked(src, W, self.packed[op.name], B, R, Y=dst, workspace=self.workspace)
            elif op.kind == "conv":
                W, B = self.params[op.name]
                self.descs[op.name].run(src, W, B, Y=dst, workspace=self.workspace)
            elif op.kind == "conv_add":
                W, B = self.params[op.name]
                self.descs[op.name].run_add(src, W, B, self.buf[op.res], Y=dst, workspace=self.workspace)
            elif op.kind == "maxpool":
                if self.channel_major:          # planes in another order, without padding between them
                    planes = lambda t, v: t.view(t.shape[0], self.batch, *v.shape[2:])
                    src, dst = planes(src, self.buf[op.src]), planes(dst, self.buf[op.dst])
                binding.onnx_maxpool2d(src, (3, 3), pads=(1, 1, 1, 1), strides=(2, 2), Y=dst)
            elif op.kind == "gap":
                if self.channel_major:
                    binding.global_average_pool_channel_major(src, self.buf[op.src].shape, dst)
                else:
                    binding.onnx_global_average_pool(src, Y=dst)
            else:
                W, B = self.params["fc"]
                binding.onnx_matmul_add(src.view(self.batch, 2048), W, B, Y=dst, workspace=self.fc_workspace)

    def close(self):
        self._graph = self._captured = None
        for d in self.descs.values():
            d.close()
        self.descs.clear()
