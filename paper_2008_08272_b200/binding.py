"""Thin ctypes binding over the C ABI declared in ``include/onnx_b200.h``.

Argument marshalling only: every step of Conv and Gemm runs in the library's
CUDA kernels.  Tensors are torch CUDA tensors used as device memory; the current
torch stream is passed through.  There is no CPU fallback: if the compiled
library is missing, or a tensor is not on a CUDA device, the call raises.

The operator calls go through ``ext/fast_binding.cpp``, which does the marshalling below natively; a call it
declines (returning None, nothing launched) is repeated here, where every check raises its own error.  Where it cannot be
built or loaded (no compiler, another torch), a warning says so and every call is made here.
"""
from __future__ import annotations

import ctypes
import os
from typing import Optional, Sequence

from . import build as _build

OK = 0
STATUS_NAMES = ["OK", "ERR_NULL", "ERR_ATTR", "ERR_SHAPE", "ERR_UNSUPPORTED", "ERR_WORKSPACE",
                "ERR_CUDA", "ERR_DEVICE_TIMEOUT"]
AUTO_PAD = {"NOTSET": 0, "SAME_UPPER": 1, "SAME_LOWER": 2, "VALID": 3}
KERNEL_FAMILIES = ["simt_direct", "simt_depthwise", "mma_gemm", "mma_implicit", "mma_gather_gemm"]
WEIGHT_COPY_FAMILIES = ("mma_implicit", "mma_gemm", "mma_gather_gemm")   # prepack always makes their derived copy of W once

EXPORTS = [
    "onnx_conv2d_desc", "onnx_conv2d_desc_query", "onnx_conv2d_desc_query_kernel", "onnx_conv2d_run",
    "onnx_conv2d_desc_destroy", "onnx_conv2d_run_static", "onnx_conv2d_static_scratch_bytes",
    "onnx_gemm_workspace_bytes", "onnx_gemm_run", "onnxb_status_string",
    "onnxb_last_device_status", "onnxb_set_kernel_override", "onnxb_launch_count",
    "onnxb_probe_tf32_mma_rate", "onnx_matmul_add_run",
    "onnx_maxpool2d_shape", "onnx_maxpool2d_run", "onnx_global_average_pool_run", "onnx_conv2d_add_run",
    "onnx_conv2d_prepack", "onnx_conv2d_run_prepacked", "onnx_conv2d_packed_bytes", "onnx_conv2d_run_packed",
    "onnx_conv2d_run_packed_sampled", "onnx_conv2d_run_packed_rounded", "onnx_conv2d_desc_layout", "onnxb_channel_pitch",
    "onnx_global_average_pool_channel_major_run", "onnxb_dispatch_state",
    "onnxb_probe_wait_timeout",
]


class OnnxB200Error(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = int(status)
        name = STATUS_NAMES[status] if 0 <= status < len(STATUS_NAMES) else str(status)
        super().__init__(f"{where}: {name}")


class ConvAttrs(ctypes.Structure):
    _fields_ = [
        ("x_dims", ctypes.c_int64 * 4), ("w_dims", ctypes.c_int64 * 4),
        ("kernel_shape", ctypes.c_int64 * 2), ("pads", ctypes.c_int64 * 4),
        ("strides", ctypes.c_int64 * 2), ("dilations", ctypes.c_int64 * 2),
        ("group", ctypes.c_int64), ("auto_pad", ctypes.c_int32), ("has_bias", ctypes.c_int32),
        ("fuse_relu", ctypes.c_int32), ("reserved", ctypes.c_int32),
    ]


_lib = None
_fast_mod = None


class _Declined:
    """Stands in for the native call path where there is none: every call is declined."""

    def __getattr__(self, name):
        return lambda *args: None


def _fast():
    """The native call path, loaded with the first operator call (it needs torch's C++ libraries)."""
    global _fast_mod
    if _fast_mod is None:
        import importlib.util
        import torch  # noqa: F401  (its libraries must be loaded first)
        load()
        try:
            path = _build.ext_path()
            if not os.path.exists(path):
                _build.build_ext()
            spec = importlib.util.spec_from_file_location("_onnxb_fast", path)
            mod = importlib.util.module_from_spec(spec)
            spec.loader.exec_module(mod)
            mod.bind(_build.LIB_PATH)
        except Exception as e:
            import warnings
            warnings.warn(f"no native call path ({e}): operator calls go through ctypes, some 10 us of host time each")
            mod = _Declined()
        _fast_mod = mod
    return _fast_mod


def library_path() -> str:
    return _build.LIB_PATH


def load(build_if_missing: bool = True):
    """Load libonnx_b200.so (building it first when absent and nvcc is available)."""
    global _lib
    if _lib is not None:
        return _lib
    path = _build.LIB_PATH
    if not os.path.exists(path):
        if not build_if_missing:
            raise OnnxB200Error(6, f"{path} is missing; run python -m paper_2008_08272_b200.build")
        _build.build()
    lib = ctypes.CDLL(path)
    vp, i64, sz = ctypes.c_void_p, ctypes.c_int64, ctypes.c_size_t
    lib.onnx_conv2d_desc.restype = ctypes.c_int
    lib.onnx_conv2d_desc.argtypes = [ctypes.POINTER(ConvAttrs), ctypes.POINTER(vp)]
    lib.onnx_conv2d_desc_query.restype = ctypes.c_int
    lib.onnx_conv2d_desc_query.argtypes = [vp, ctypes.POINTER(i64), ctypes.POINTER(i64), ctypes.POINTER(sz)]
    lib.onnx_conv2d_desc_query_kernel.restype = ctypes.c_int
    lib.onnx_conv2d_desc_query_kernel.argtypes = [vp]
    lib.onnx_conv2d_run.restype = ctypes.c_int
    lib.onnx_conv2d_run.argtypes = [vp, vp, vp, vp, vp, vp, sz, vp]
    lib.onnx_conv2d_add_run.restype = ctypes.c_int
    lib.onnx_conv2d_add_run.argtypes = [vp, vp, vp, vp, vp, vp, vp, sz, vp]
    lib.onnx_conv2d_prepack.restype = ctypes.c_int
    lib.onnx_conv2d_prepack.argtypes = [vp, vp, vp, sz, vp]
    lib.onnx_conv2d_packed_bytes.restype = sz
    lib.onnx_conv2d_packed_bytes.argtypes = [vp]
    lib.onnx_conv2d_run_packed.restype = ctypes.c_int
    lib.onnx_conv2d_run_packed.argtypes = [vp, vp, vp, vp, sz, vp, vp, vp, vp, sz, vp]
    lib.onnx_conv2d_run_packed_sampled.restype = ctypes.c_int
    lib.onnx_conv2d_run_packed_sampled.argtypes = [vp, vp, vp, vp, sz, vp, vp, ctypes.POINTER(i64), ctypes.POINTER(i64),
                                                   vp, vp, vp, sz, vp]
    lib.onnx_conv2d_run_packed_rounded.restype = ctypes.c_int
    lib.onnx_conv2d_run_packed_rounded.argtypes = [vp, vp, vp, vp, sz, vp, vp, vp, vp, vp, sz, vp]
    lib.onnx_conv2d_desc_layout.restype = ctypes.c_int
    lib.onnx_conv2d_desc_layout.argtypes = [vp, ctypes.c_int, ctypes.c_int, ctypes.POINTER(vp)]
    lib.onnxb_channel_pitch.restype = sz
    lib.onnxb_channel_pitch.argtypes = [i64, i64, i64]
    lib.onnx_global_average_pool_channel_major_run.restype = ctypes.c_int
    lib.onnx_global_average_pool_channel_major_run.argtypes = [ctypes.POINTER(i64), vp, vp, vp]
    lib.onnx_conv2d_run_prepacked.restype = ctypes.c_int
    lib.onnx_conv2d_run_prepacked.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, sz, vp]
    lib.onnx_conv2d_run_static.restype = ctypes.c_int
    lib.onnx_conv2d_run_static.argtypes = [vp, vp, vp, vp, vp, vp]
    lib.onnx_conv2d_static_scratch_bytes.restype = sz
    lib.onnx_conv2d_static_scratch_bytes.argtypes = []
    lib.onnx_conv2d_desc_destroy.restype = None
    lib.onnx_conv2d_desc_destroy.argtypes = [vp]
    lib.onnx_gemm_workspace_bytes.restype = sz
    lib.onnx_gemm_workspace_bytes.argtypes = [ctypes.c_int, ctypes.c_int, i64, i64, i64]
    lib.onnx_gemm_run.restype = ctypes.c_int
    lib.onnx_gemm_run.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_float, ctypes.c_float, i64, i64, i64,
                                  vp, vp, vp, ctypes.c_int, ctypes.POINTER(i64), ctypes.c_int, vp, vp, sz, vp]
    lib.onnx_matmul_add_run.restype = ctypes.c_int
    lib.onnx_matmul_add_run.argtypes = [i64, i64, i64, vp, vp, vp, ctypes.c_int, ctypes.POINTER(i64), ctypes.c_int, vp,
                                        vp, sz, vp]
    p64 = ctypes.POINTER(i64)
    lib.onnx_maxpool2d_shape.restype = ctypes.c_int
    lib.onnx_maxpool2d_shape.argtypes = [p64, p64, p64, p64, p64]
    lib.onnx_maxpool2d_run.restype = ctypes.c_int
    lib.onnx_maxpool2d_run.argtypes = [p64, p64, p64, p64, vp, vp, vp]
    lib.onnx_global_average_pool_run.restype = ctypes.c_int
    lib.onnx_global_average_pool_run.argtypes = [p64, vp, vp, vp]
    lib.onnxb_status_string.restype = ctypes.c_char_p
    lib.onnxb_status_string.argtypes = [ctypes.c_int]
    lib.onnxb_last_device_status.restype = ctypes.c_int
    lib.onnxb_last_device_status.argtypes = [vp]
    lib.onnxb_set_kernel_override.restype = None
    lib.onnxb_set_kernel_override.argtypes = [ctypes.c_int]
    lib.onnxb_dispatch_state.restype = ctypes.c_uint64
    lib.onnxb_dispatch_state.argtypes = []
    lib.onnxb_launch_count.restype = ctypes.c_uint64
    lib.onnxb_launch_count.argtypes = []
    lib.onnxb_probe_tf32_mma_rate.restype = ctypes.c_int
    lib.onnxb_probe_tf32_mma_rate.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_double), vp]
    lib.onnxb_probe_wait_timeout.restype = ctypes.c_int
    lib.onnxb_probe_wait_timeout.argtypes = [ctypes.c_longlong, vp]
    _lib = lib
    return lib


def _check(status: int, where: str, no_memory=None):
    """``no_memory``: what stood in the way of a workspace (``_scratch``)."""
    if no_memory is not None and STATUS_NAMES[status] == "ERR_WORKSPACE":
        raise no_memory
    if status != OK:
        raise OnnxB200Error(status, where)


def _dev_ptr(t, name: str, allow_none: bool = False):
    if t is None:
        if allow_none:
            return None
        raise OnnxB200Error(1, f"{name} is None")
    import torch
    if not isinstance(t, torch.Tensor) or not t.is_cuda:
        raise TypeError(f"{name} must be a torch CUDA tensor (there is no CPU path)")
    if t.dtype != torch.float32 or not t.is_contiguous():
        raise TypeError(f"{name} must be contiguous float32")
    return ctypes.c_void_p(t.data_ptr())


def _stream_ptr(stream=None):
    import torch
    s = stream if stream is not None else torch.cuda.current_stream()
    return ctypes.c_void_p(s.cuda_stream)


def _new(size, device, stream, dtype="float32", kept=True):
    """Memory for a call on ``stream`` (None: the current one).  The allocator hands a block out and takes it back in the order of
    the stream it was made on: made on another than the call's, the block's last user may not have finished when the call's kernels
    begin, nor they when its next one does.  What the caller keeps goes on to be used from the current stream, too."""
    import torch
    dtype = getattr(torch, dtype)
    if stream is None or not str(device).startswith("cuda"):
        return torch.empty(size, dtype=dtype, device=device)
    current = torch.cuda.current_stream(device)
    if stream.cuda_stream == current.cuda_stream:
        return torch.empty(size, dtype=dtype, device=device)
    if not isinstance(stream, torch.cuda.Stream):        # anything with a handle
        stream = torch.cuda.ExternalStream(stream.cuda_stream, device) if stream.cuda_stream else torch.cuda.default_stream(device)
    with torch.cuda.stream(stream):
        t = torch.empty(size, dtype=dtype, device=device)
    if kept:
        t.record_stream(current)
    return t


def _scratch(size, device, stream):
    """A workspace of ``size`` bytes as (tensor, pointer, bytes, None), or where there is no memory for it (None, None, 0, the error):
    the fp32 kernels do without, and for the others ``_check`` raises the error."""
    import torch
    try:
        t = _new(size, device, stream, "uint8", kept=False)
    except torch.OutOfMemoryError as e:
        return None, None, 0, e.with_traceback(None)     # (whose frames would hold the caller's tensors)
    return t, ctypes.c_void_p(t.data_ptr()), size, None


def _given(workspace):
    if workspace is None:
        return None, None, 0, None
    return workspace, ctypes.c_void_p(workspace.data_ptr()), workspace.numel() * workspace.element_size(), None


def make_attrs(x_shape, w_shape, *, kernel_shape=None, pads=None, strides=None, dilations=None, group=0,
               auto_pad="NOTSET", has_bias=False, fuse_relu=False) -> ConvAttrs:
    a = ConvAttrs()
    a.x_dims[:] = list(x_shape)
    a.w_dims[:] = list(w_shape)
    if kernel_shape is not None:
        a.kernel_shape[:] = list(kernel_shape)
    if pads is not None:
        a.pads[:] = list(pads)
    if strides is not None:
        a.strides[:] = list(strides)
    if dilations is not None:
        a.dilations[:] = list(dilations)
    a.group = int(group)
    a.auto_pad = AUTO_PAD[auto_pad] if isinstance(auto_pad, str) else int(auto_pad)
    a.has_bias = int(bool(has_bias))
    a.fuse_relu = int(bool(fuse_relu))
    return a


def channel_pitch(shape) -> int:
    """Floats from one channel to the next of a channel-major tensor of the logical shape (images, channels, rows, columns)."""
    return int(load().onnxb_channel_pitch(shape[0], shape[2], shape[3]))


class Conv2dDesc:
    """Owns an ``onnxb_conv2d_desc_t`` (``onnx_conv2d_desc`` .. ``onnx_conv2d_desc_destroy``)."""

    def __init__(self, x_shape, w_shape, *, x_channel_major=False, y_channel_major=False, **attrs):
        self._lib = load()
        self._h = ctypes.c_void_p()
        self.attrs = make_attrs(x_shape, w_shape, **attrs)
        _check(self._lib.onnx_conv2d_desc_layout(ctypes.byref(self.attrs), int(x_channel_major), int(y_channel_major),
                                                 ctypes.byref(self._h)), "onnx_conv2d_desc")
        y = (ctypes.c_int64 * 4)()
        p = (ctypes.c_int64 * 4)()
        ws = ctypes.c_size_t()
        _check(self._lib.onnx_conv2d_desc_query(self._h, y, p, ctypes.byref(ws)), "onnx_conv2d_desc_query")
        self.y_shape = tuple(int(v) for v in y)
        # as it lies in memory: itself, or (channel, floats from one channel to the next)
        self.y_storage = (self.y_shape[1], channel_pitch(self.y_shape), 1, 1) if y_channel_major else self.y_shape
        self.pads = tuple(int(v) for v in p)
        self.workspace_bytes = int(ws.value)
        self.kernel_family = KERNEL_FAMILIES[self._lib.onnx_conv2d_desc_query_kernel(self._h)]
        self.packed_bytes = int(self._lib.onnx_conv2d_packed_bytes(self._h))
        self._packed_needs_ws = self.workspace_bytes > self.packed_bytes
        self._plan = None

    def _native(self, X, W, packed, B, R, Y, workspace, stream):
        """The call through the native path; None when it declined."""
        if self._plan is None:
            if not self._h:
                return None
            self._plan = _fast().plan(self._h.value, self.y_storage, self.workspace_bytes, self.packed_bytes, self._packed_needs_ws)
        return _fast_mod.conv(self._plan, X, W, packed, B, R, Y, workspace, stream)

    def _native_rounded(self, X, W, packed, B, R, Y, workspace, stream, r_dims, strides, Y_rounded):
        """The same with an addend that is sampled (r_dims not None), or Y rounded as well.  (A function of its own: arguments passed on
        as a tuple would cost every call 0.1 us.)"""
        if self._plan is None:
            if not self._h:
                return None
            self._plan = _fast().plan(self._h.value, self.y_storage, self.workspace_bytes, self.packed_bytes, self._packed_needs_ws)
        return _fast_mod.conv(self._plan, X, W, packed, B, R, Y, workspace, stream, r_dims, strides, Y_rounded)

    def run(self, X, W, B=None, Y=None, workspace=None, stream=None):
        """``onnx_conv2d_run``; allocates Y (and a workspace) with torch when not supplied."""
        y = self._native(X, W, None, B, None, Y, workspace, stream)
        if y is not None:
            return y
        if Y is None:
            Y = _new(self.y_storage, X.device, stream)
        needs = workspace is None and self.workspace_bytes
        workspace, ws_ptr, ws_len, no_memory = _scratch(self.workspace_bytes, X.device, stream) if needs else _given(workspace)
        _check(self._lib.onnx_conv2d_run(self._h, _dev_ptr(X, "X"), _dev_ptr(W, "W"),
                                         _dev_ptr(B, "B", allow_none=True), _dev_ptr(Y, "Y"),
                                         ws_ptr, ws_len, _stream_ptr(stream)), "onnx_conv2d_run", no_memory)
        return Y

    def run_add(self, X, W, B, R, Y=None, workspace=None, stream=None):
        """``onnx_conv2d_add_run``: Y = relu?(Conv(X, W) + B + R), R shaped like Y (a residual connection)."""
        if R is not None:
            y = self._native(X, W, None, B, R, Y, workspace, stream)
            if y is not None:
                return y
        if Y is None:
            Y = _new(self.y_storage, X.device, stream)
        needs = workspace is None and self.workspace_bytes
        workspace, ws_ptr, ws_len, no_memory = _scratch(self.workspace_bytes, X.device, stream) if needs else _given(workspace)
        _check(self._lib.onnx_conv2d_add_run(self._h, _dev_ptr(X, "X"), _dev_ptr(W, "W"),
                                             _dev_ptr(B, "B", allow_none=True), _dev_ptr(R, "R"), _dev_ptr(Y, "Y"),
                                             ws_ptr, ws_len, _stream_ptr(stream)), "onnx_conv2d_add_run", no_memory)
        return Y

    def prepack(self, W, stream=None):
        """``onnx_conv2d_prepack``: the packed copy of constant weights (a uint8 device tensor; untouched when
        this descriptor's kernel reads W directly)."""
        import torch
        try:
            packed = _new(max(self.packed_bytes, 16), W.device, stream, "uint8")
        except torch.OutOfMemoryError:
            if self.kernel_family != "simt_direct":      # (the fp32 kernels take W itself)
                raise
            packed = _new(16, W.device, stream, "uint8")
        _check(self._lib.onnx_conv2d_prepack(self._h, _dev_ptr(W, "W"), ctypes.c_void_p(packed.data_ptr()),
                                             packed.numel(), _stream_ptr(stream)), "onnx_conv2d_prepack")
        return packed

    def run_prepacked(self, X, W, packed, B=None, R=None, Y=None, workspace=None, stream=None):
        """``onnx_conv2d_run_packed``: run (R None) or run_add (R given) from a packed copy of W."""
        if packed is not None:
            y = self._native(X, W, packed, B, R, Y, workspace, stream)
            if y is not None:
                return y
        if Y is None:
            Y = _new(self.y_storage, X.device, stream)
        packed_len = packed.numel() * packed.element_size()
        needs = workspace is None and self.workspace_bytes and (self._packed_needs_ws or packed_len < self.packed_bytes)
        workspace, ws_ptr, ws_len, no_memory = _scratch(self.workspace_bytes, X.device, stream) if needs else _given(workspace)
        _check(self._lib.onnx_conv2d_run_packed(self._h, _dev_ptr(X, "X"), _dev_ptr(W, "W"),
                                                ctypes.c_void_p(packed.data_ptr()), packed_len,
                                                _dev_ptr(B, "B", allow_none=True), _dev_ptr(R, "R", allow_none=True),
                                                _dev_ptr(Y, "Y"), ws_ptr, ws_len, _stream_ptr(stream)),
               "onnx_conv2d_run_packed", no_memory)
        return Y

    def run_prepacked_sampled(self, X, W, packed, B, R, strides, Y=None, Y_rounded=None, r_dims=None, workspace=None, stream=None):
        """``onnx_conv2d_run_packed_sampled``: run_prepacked with the addend R[:, :, ::strides[0], ::strides[1]]; Y rounded to TF32
        goes to ``Y_rounded`` where it is given.  ``r_dims``: rows and columns of a channel-major R."""
        if r_dims is None:
            if R.dim() != 4 or tuple(R.shape[:2]) != self.y_shape[:2]:
                raise OnnxB200Error(3, "run_prepacked_sampled: the addend's images and channels are not the output's")
            r_dims = R.shape[2:]
        # (tuples: of a torch.Size the native path knows nothing)
        y = self._native_rounded(X, W, packed, B, R, Y, workspace, stream, tuple(r_dims), tuple(strides), Y_rounded)
        if y is not None:
            return y
        if Y is None:
            Y = _new(self.y_storage, X.device, stream)
        needs = workspace is None and self.workspace_bytes and self._packed_needs_ws
        workspace, ws_ptr, ws_len, no_memory = _scratch(self.workspace_bytes, X.device, stream) if needs else _given(workspace)
        _check(self._lib.onnx_conv2d_run_packed_sampled(self._h, _dev_ptr(X, "X"), _dev_ptr(W, "W"),
                                                        ctypes.c_void_p(packed.data_ptr()), packed.numel() * packed.element_size(),
                                                        _dev_ptr(B, "B", allow_none=True), _dev_ptr(R, "R"),
                                                        _i64(r_dims, 2), _i64(strides, 2), _dev_ptr(Y, "Y"),
                                                        _dev_ptr(Y_rounded, "Y_rounded", allow_none=True), ws_ptr, ws_len, _stream_ptr(stream)),
               "onnx_conv2d_run_packed_sampled", no_memory)
        return Y

    def run_prepacked_rounded(self, X, W, packed, B, R, Y, Y_rounded, stream=None, workspace=None):
        """``onnx_conv2d_run_packed_rounded``: run_prepacked, and Y rounded to TF32 into ``Y_rounded`` (Y itself where it is that)."""
        y = self._native_rounded(X, W, packed, B, R, Y, workspace, stream, None, None, Y_rounded)
        if y is not None:
            return y
        needs = workspace is None and self.workspace_bytes and self._packed_needs_ws
        workspace, ws_ptr, ws_len, no_memory = _scratch(self.workspace_bytes, X.device, stream) if needs else _given(workspace)
        _check(self._lib.onnx_conv2d_run_packed_rounded(self._h, _dev_ptr(X, "X"), _dev_ptr(W, "W"), ctypes.c_void_p(packed.data_ptr()),
                                                        packed.numel() * packed.element_size(), _dev_ptr(B, "B", allow_none=True),
                                                        _dev_ptr(R, "R", allow_none=True), _dev_ptr(Y, "Y"),
                                                        _dev_ptr(Y_rounded, "Y_rounded"), ws_ptr, ws_len, _stream_ptr(stream)),
               "onnx_conv2d_run_packed_rounded", no_memory)
        return Y

    def run_static(self, X, W, B=None, Y=None, stream=None):
        """``onnx_conv2d_run_static``: like run(), but the library's built-in scratch array
        stands in for the workspace, so no device memory is allocated for scratch.  (Y is
        still allocated here with torch when the caller does not pass one.)"""
        if Y is None:
            Y = _new(self.y_storage, X.device, stream)
        _check(self._lib.onnx_conv2d_run_static(self._h, _dev_ptr(X, "X"), _dev_ptr(W, "W"),
                                                _dev_ptr(B, "B", allow_none=True), _dev_ptr(Y, "Y"),
                                                _stream_ptr(stream)), "onnx_conv2d_run_static")
        return Y

    def close(self):
        self._plan = None
        if self._h:
            self._lib.onnx_conv2d_desc_destroy(self._h)
            self._h = ctypes.c_void_p()

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def onnx_conv2d(X, W, B=None, *, pads=None, strides=None, dilations=None, group=0, auto_pad="NOTSET",
                kernel_shape=None, fuse_relu=False, Y=None, workspace=None, stream=None):
    """One-shot ONNX Conv: build a descriptor, run, destroy."""
    d = Conv2dDesc(tuple(X.shape), tuple(W.shape), kernel_shape=kernel_shape, pads=pads, strides=strides,
                   dilations=dilations, group=group, auto_pad=auto_pad, has_bias=B is not None,
                   fuse_relu=fuse_relu)
    try:
        return d.run(X, W, B, Y=Y, workspace=workspace, stream=stream)
    finally:
        d.close()


def gemm_workspace_bytes(transA, transB, M, N, K) -> int:
    return int(load().onnx_gemm_workspace_bytes(int(bool(transA)), int(bool(transB)), M, N, K))


def onnx_gemm(A, B, C=None, *, alpha=1.0, beta=1.0, transA=False, transB=False, fuse_relu=False,
              Y=None, workspace=None, stream=None):
    """``onnx_gemm_run``: Y = relu?(alpha * A' @ B' + beta * C)."""
    y = (_fast_mod or _fast()).gemm(A, B, C, alpha, beta, transA, transB, fuse_relu, Y, workspace, stream)
    if y is not None:
        return y
    lib = load()
    M, K = (A.shape[1], A.shape[0]) if transA else (A.shape[0], A.shape[1])
    N = B.shape[0] if transB else B.shape[1]
    kb = B.shape[1] if transB else B.shape[0]
    if kb != K:
        raise OnnxB200Error(3, "onnx_gemm: inner dimensions differ")
    if Y is None:
        Y = _new((M, N), A.device, stream)
    c_rank, c_dims = 0, None
    if C is not None:
        c_rank = C.dim()
        c_dims = (ctypes.c_int64 * max(c_rank, 1))(*[int(v) for v in C.shape])
    need = gemm_workspace_bytes(transA, transB, M, N, K)
    workspace, ws_ptr, ws_len, no_memory = _scratch(need, A.device, stream) if workspace is None and need else _given(workspace)
    _check(lib.onnx_gemm_run(int(bool(transA)), int(bool(transB)), float(alpha), float(beta), M, N, K,
                             _dev_ptr(A, "A"), _dev_ptr(B, "B"), _dev_ptr(C, "C", allow_none=True),
                             c_rank, c_dims, int(bool(fuse_relu)), _dev_ptr(Y, "Y"), ws_ptr, ws_len,
                             _stream_ptr(stream)), "onnx_gemm_run", no_memory)
    return Y


def static_scratch_bytes() -> int:
    return int(load().onnx_conv2d_static_scratch_bytes())


def last_device_status(stream=None) -> int:
    return int(load().onnxb_last_device_status(_stream_ptr(stream)))


def set_kernel_override(family) -> None:
    """``None``/"auto" = automatic; or one of KERNEL_FAMILIES."""
    v = -1 if family in (None, "auto") else KERNEL_FAMILIES.index(family)
    load().onnxb_set_kernel_override(v)


def launch_count() -> int:
    """``onnxb_launch_count``: kernels launched by operator calls (those of a replayed CUDA graph are launched by no call)."""
    return int(load().onnxb_launch_count())


def call_state(*tensors):
    """Where tensors lie and how (address, type, sizes, strides) and ``onnxb_dispatch_state``, as bytes to compare: calls on the same
    tensors at the same state launch the same kernels on the same memory.  ``tensors``: tensors, tuples of them, and dicts of either,
    whose entry "input" is left out.  None without the native call path."""
    return (_fast_mod or _fast()).state(*tensors)


def probe_tf32_mma_rate(n: int, instructions: int = 4096, stream=None) -> float:
    """``onnxb_probe_tf32_mma_rate``: SM cycles per 128 x n x 8 TF32 MMA with operands resident
    in shared memory (the tensor pipe's ceiling for that shape; ideal n / 2)."""
    out = ctypes.c_double()
    _check(load().onnxb_probe_tf32_mma_rate(int(n), int(instructions), ctypes.byref(out), _stream_ptr(stream)),
           "onnxb_probe_tf32_mma_rate")
    return float(out.value)


def probe_wait_timeout(limit_cycles: int = 1000000, stream=None) -> None:
    """``onnxb_probe_wait_timeout``: enqueue a kernel whose only (bounded) wait runs out after
    ``limit_cycles`` SM cycles; the next ``last_device_status`` then reports ERR_DEVICE_TIMEOUT once."""
    _check(load().onnxb_probe_wait_timeout(int(limit_cycles), _stream_ptr(stream)), "onnxb_probe_wait_timeout")


def onnx_matmul_add(A, B, C=None, *, fuse_relu=False, Y=None, workspace=None, stream=None):
    """``onnx_matmul_add_run``: Y = relu?(A @ B + C), the MatMul + Add pair as one fused Gemm."""
    # (exactly onnx_gemm_run with transA = transB = 0 and alpha = beta = 1)
    y = (_fast_mod or _fast()).gemm(A, B, C, 1.0, 1.0, False, False, fuse_relu, Y, workspace, stream)
    if y is not None:
        return y
    lib = load()
    M, K = A.shape
    if B.shape[0] != K:
        raise OnnxB200Error(3, "onnx_matmul_add: inner dimensions differ")
    N = B.shape[1]
    if Y is None:
        Y = _new((M, N), A.device, stream)
    c_rank, c_dims = 0, None
    if C is not None:
        c_rank = C.dim()
        c_dims = (ctypes.c_int64 * max(c_rank, 1))(*[int(v) for v in C.shape])
    need = gemm_workspace_bytes(False, False, M, N, K)
    workspace, ws_ptr, ws_len, no_memory = _scratch(need, A.device, stream) if workspace is None and need else _given(workspace)
    _check(lib.onnx_matmul_add_run(M, N, K, _dev_ptr(A, "A"), _dev_ptr(B, "B"), _dev_ptr(C, "C", allow_none=True),
                                   c_rank, c_dims, int(bool(fuse_relu)), _dev_ptr(Y, "Y"), ws_ptr, ws_len,
                                   _stream_ptr(stream)), "onnx_matmul_add_run", no_memory)
    return Y


def _i64(values, n):
    if values is None:
        return None
    return (ctypes.c_int64 * n)(*[int(v) for v in values])


def maxpool2d_shape(x_shape, kernel_shape, pads=None, strides=None):
    """``onnx_maxpool2d_shape``: output dims of ONNX MaxPool (host only)."""
    y = (ctypes.c_int64 * 4)()
    _check(load().onnx_maxpool2d_shape(_i64(x_shape, 4), _i64(kernel_shape, 2), _i64(pads, 4), _i64(strides, 2), y),
           "onnx_maxpool2d_shape")
    return tuple(int(v) for v in y)


def onnx_maxpool2d(X, kernel_shape, *, pads=None, strides=None, Y=None, stream=None):
    """``onnx_maxpool2d_run``: ONNX MaxPool (2-D, NCHW, dilation 1, ceil_mode 0)."""
    y = (_fast_mod or _fast()).maxpool(X, kernel_shape, pads, strides, Y, stream)
    if y is not None:
        return y
    y_shape = maxpool2d_shape(tuple(X.shape), kernel_shape, pads, strides)
    if Y is None:
        Y = _new(y_shape, X.device, stream)
    _check(load().onnx_maxpool2d_run(_i64(tuple(X.shape), 4), _i64(kernel_shape, 2), _i64(pads, 4), _i64(strides, 2),
                                     _dev_ptr(X, "X"), _dev_ptr(Y, "Y"), _stream_ptr(stream)), "onnx_maxpool2d_run")
    return Y


def global_average_pool_channel_major(X, x_shape, Y, stream=None):
    """``onnx_global_average_pool_channel_major_run``: Y[n,c,0,0] = mean of X[n,c,:,:], X channel-major."""
    _check(load().onnx_global_average_pool_channel_major_run(_i64(x_shape, 4), _dev_ptr(X, "X"), _dev_ptr(Y, "Y"), _stream_ptr(stream)),
           "onnx_global_average_pool_channel_major_run")
    return Y


def onnx_global_average_pool(X, *, Y=None, stream=None):
    """``onnx_global_average_pool_run``: Y[n,c,0,0] = mean of X[n,c,:,:]."""
    y = (_fast_mod or _fast()).gap(X, Y, stream)
    if y is not None:
        return y
    if Y is None:
        Y = _new((X.shape[0], X.shape[1], 1, 1), X.device, stream)
    _check(load().onnx_global_average_pool_run(_i64(tuple(X.shape), 4), _dev_ptr(X, "X"), _dev_ptr(Y, "Y"),
                                               _stream_ptr(stream)), "onnx_global_average_pool_run")
    return Y
