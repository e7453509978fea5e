"""The build and the binding without what the native call path needs: the library is compiled without torch, and operator
calls go through ctypes where that path cannot be built."""
import os
import subprocess
import sys

import pytest

from paper_2008_08272_b200 import binding
from paper_2008_08272_b200 import build as lib_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_is_built_without_torch(tmp_path):
    code = f"""
import os, subprocess, sys
sys.modules["torch"] = None                                  # an import of it raises
from paper_2008_08272_b200 import build
build.LIB_DIR, build.LIB_PATH = {str(tmp_path)!r}, os.path.join({str(tmp_path)!r}, "lib.so")
commands = []
def compiler(cmd, **kw):                                     # stands in for nvcc
    commands.append(cmd)
    open(cmd[cmd.index("-o") + 1], "w").close()
    return subprocess.CompletedProcess(cmd, 0, "")
build.subprocess.run = compiler
assert build.build(force=True) == build.LIB_PATH and os.path.exists(build.LIB_PATH)
assert len(commands) == 1 and "nvcc" in commands[0][0] and any(c.endswith("api.cu") for c in commands[0])
"""
    proc = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert proc.returncode == 0, proc.stderr


def test_native_call_path_is_one_per_torch_version(monkeypatch):
    import importlib.metadata
    here = lib_build.ext_path()
    monkeypatch.setattr(importlib.metadata, "version", lambda name: "0.0.1")
    other = lib_build.ext_path()
    assert here != other and os.path.dirname(here) == os.path.dirname(other)


@pytest.mark.parametrize("fault", ["no compiler", "not loadable"])
def test_calls_go_through_ctypes_without_the_native_path(fault, monkeypatch, tmp_path):
    torch = pytest.importorskip("torch")

    def no_compiler(*a, **kw):
        raise RuntimeError("no compiler")

    path = tmp_path / "ext.so"
    if fault == "not loadable":
        path.write_bytes(b"no library")
    monkeypatch.setattr(lib_build, "ext_path", lambda: str(path))
    monkeypatch.setattr(lib_build, "build_ext", no_compiler)
    monkeypatch.setattr(binding, "_fast_mod", None)
    a = torch.zeros(4, 4)
    with pytest.warns(UserWarning, match="ctypes"), pytest.raises(TypeError, match="CUDA tensor"):
        binding.onnx_gemm(a, a)                              # declined, and refused by the checked path
    d = binding.Conv2dDesc((1, 1, 4, 4), (1, 1, 3, 3))
    with pytest.raises(TypeError, match="CUDA tensor"):
        d.run(torch.zeros(1, 1, 4, 4), torch.zeros(1, 1, 3, 3))
    d.close()


@pytest.mark.gpu
def test_ctypes_path_gives_the_native_path_s_results(monkeypatch):
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev)
    g.manual_seed(1)
    X, W, B, A = (torch.randn(s, generator=g, device=dev) for s in ((2, 64, 12, 12), (32, 64, 3, 3), (32,), (40, 64)))
    d = binding.Conv2dDesc(tuple(X.shape), tuple(W.shape), pads=(1, 1, 1, 1), has_bias=True)
    packed = d.prepack(W)
    calls = [lambda: d.run(X, W, B), lambda: d.run_prepacked(X, W, packed, B), lambda: binding.onnx_gemm(A, A, transB=True),
             lambda: binding.onnx_matmul_add(A, A.t().contiguous(), B[:1]), lambda: binding.onnx_maxpool2d(X, (2, 2), strides=(2, 2)),
             lambda: binding.onnx_global_average_pool(X)]
    native = [call() for call in calls]
    assert not isinstance(binding._fast_mod, binding._Declined)
    monkeypatch.setattr(binding, "_fast_mod", binding._Declined())
    for call, want in zip(calls, native):
        assert torch.equal(call(), want)
    d.close()
