// The binding's call path in native code: argument checks on torch tensors, allocation of outputs the caller
// did not supply, the current stream, and the C-ABI call, in one C function per operator.  An operator of a
// few microseconds costs more on the host than on the GPU, so this path is what small calls are made of:
// written in Python over ctypes the same steps took 8 to 17 us per call, here 1 to 2 us.
//
// A call that is not entirely ordinary (an argument that is no contiguous fp32 CUDA tensor, a status other
// than OK, a shape that does not fit) returns None without having launched anything, and the Python caller
// repeats it through its checked path, which raises the precise error.
#include <Python.h>
#include <dlfcn.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <vector>

#include "onnx_b200.h"

namespace {

struct Abi {
    decltype(&onnx_conv2d_run) conv_run;
    decltype(&onnx_conv2d_add_run) conv_add_run;
    decltype(&onnx_conv2d_run_packed) conv_run_packed;
    decltype(&onnx_conv2d_run_packed_sampled) conv_run_packed_sampled;
    decltype(&onnx_conv2d_run_packed_rounded) conv_run_packed_rounded;
    decltype(&onnx_gemm_workspace_bytes) gemm_workspace_bytes;
    decltype(&onnx_gemm_run) gemm_run;
    decltype(&onnx_maxpool2d_shape) maxpool2d_shape;
    decltype(&onnx_maxpool2d_run) maxpool2d_run;
    decltype(&onnx_global_average_pool_run) global_average_pool_run;
    decltype(&onnxb_dispatch_state) dispatch_state;
} abi;

struct Plan {                    // what a convolution descriptor resolved to
    onnxb_conv2d_desc_t desc;
    int64_t y[4];
    size_t workspace;            // bytes onnx_conv2d_run needs
    size_t packed;               // bytes of the copy of W (0: none)
    bool packed_needs_ws;        // onnx_conv2d_run_packed needs the workspace too
};

// An argument as the library takes it: nullptr for None; `fine` cleared when it is anything but a contiguous
// fp32 CUDA tensor.
inline const float *in_ptr(PyObject *o, bool &fine, const at::Tensor **t = nullptr) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_CheckExact(o)) { fine = false; return nullptr; }
    const at::Tensor &x = THPVariable_Unpack(o);
    if (!x.is_cuda() || x.scalar_type() != at::kFloat || !x.is_contiguous()) { fine = false; return nullptr; }
    if (t) *t = &x;
    return static_cast<const float *>(x.data_ptr());
}

// A workspace tensor of any type, or None.
inline void *ws_ptr(PyObject *o, size_t &bytes, bool &fine) {
    bytes = 0;
    if (o == Py_None) return nullptr;
    if (!THPVariable_CheckExact(o)) { fine = false; return nullptr; }
    const at::Tensor &x = THPVariable_Unpack(o);
    bytes = x.nbytes();
    return x.data_ptr();
}

// (only asked for once the tensors are known to be CUDA tensors: without a device it throws)
inline void *stream_ptr(PyObject *o, bool &fine) {
    if (!fine) return nullptr;
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *a = PyObject_GetAttrString(o, "cuda_stream");
    if (!a) { PyErr_Clear(); fine = false; return nullptr; }
    void *p = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
    if (PyErr_Occurred()) { PyErr_Clear(); fine = false; }
    return p;
}

// Memory for a call on `st`; `given` is the stream argument it came from.  The allocator hands a block out and takes it back in
// the order of the stream it was made on: made on another than the call's, the block's last user may not have finished when the
// call's kernels begin, nor they when its next one does.  A result goes on to be used from the current stream, too.
inline at::Tensor new_tensor(at::IntArrayRef size, at::ScalarType type, const at::Device &dev, PyObject *given, void *st, bool is_result) {
    if (given != Py_None) {
        const c10::cuda::CUDAStream current = c10::cuda::getCurrentCUDAStream(dev.index());
        if (current.stream() != st) {
            const c10::cuda::CUDAStreamGuard on(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(st), dev.index()));
            at::Tensor t(at::detail::empty_cuda(size, type, dev, c10::nullopt));
            if (is_result) c10::cuda::CUDACachingAllocator::recordStream(t.storage().data_ptr(), current);
            return t;
        }
    }
    return at::Tensor(at::detail::empty_cuda(size, type, dev, c10::nullopt));
}

// The result: the caller's own Y object, or the tensor made here.
inline PyObject *result(PyObject *given, at::Tensor &made) {
    if (given == Py_None) return THPVariable_Wrap(std::move(made));
    Py_INCREF(given);
    return given;
}

inline PyObject *slow_path() { Py_RETURN_NONE; }

inline Plan *plan_of(PyObject *o) { return static_cast<Plan *>(PyCapsule_GetPointer(o, "onnxb.plan")); }

void plan_free(PyObject *o) { delete plan_of(o); }

// bind(path): resolve the C ABI in the library the ctypes binding has loaded
PyObject *py_bind(PyObject *, PyObject *arg) {
    const char *path = PyUnicode_AsUTF8(arg);
    if (!path) return nullptr;
    void *h = dlopen(path, RTLD_NOW | RTLD_NOLOAD);
    if (!h) { PyErr_SetString(PyExc_OSError, "the library is not loaded"); return nullptr; }
    bool ok = true;
    auto get = [&](auto &fn, const char *name) {
        fn = reinterpret_cast<std::decay_t<decltype(fn)>>(dlsym(h, name));
        ok = ok && fn;
    };
    get(abi.conv_run, "onnx_conv2d_run");
    get(abi.conv_add_run, "onnx_conv2d_add_run");
    get(abi.conv_run_packed, "onnx_conv2d_run_packed");
    get(abi.conv_run_packed_sampled, "onnx_conv2d_run_packed_sampled");
    get(abi.conv_run_packed_rounded, "onnx_conv2d_run_packed_rounded");
    get(abi.gemm_workspace_bytes, "onnx_gemm_workspace_bytes");
    get(abi.gemm_run, "onnx_gemm_run");
    get(abi.maxpool2d_shape, "onnx_maxpool2d_shape");
    get(abi.maxpool2d_run, "onnx_maxpool2d_run");
    get(abi.global_average_pool_run, "onnx_global_average_pool_run");
    get(abi.dispatch_state, "onnxb_dispatch_state");
    if (!ok) { PyErr_SetString(PyExc_OSError, "a symbol of the C ABI is missing"); return nullptr; }
    Py_RETURN_NONE;
}

// plan(desc address, (n, m, p, q), workspace bytes, packed bytes, whether a run from the copy needs workspace) -> capsule
PyObject *py_plan(PyObject *, PyObject *args) {
    unsigned long long desc, ws, packed;
    long long y[4];
    int needs;
    if (!PyArg_ParseTuple(args, "K(LLLL)KKp", &desc, &y[0], &y[1], &y[2], &y[3], &ws, &packed, &needs)) return nullptr;
    Plan *p = new Plan{reinterpret_cast<onnxb_conv2d_desc_t>(desc), {y[0], y[1], y[2], y[3]}, (size_t)ws, (size_t)packed, needs != 0};
    return PyCapsule_New(p, "onnxb.plan", plan_free);
}

// n integers of a tuple or list; None leaves the defaults
inline bool ints(PyObject *o, int64_t *out, Py_ssize_t n) {
    if (o == Py_None) return true;
    PyObject *const *items;
    if (PyTuple_CheckExact(o) && PyTuple_GET_SIZE(o) == n) items = &PyTuple_GET_ITEM(o, 0);
    else if (PyList_CheckExact(o) && PyList_GET_SIZE(o) == n) items = &PyList_GET_ITEM(o, 0);
    else return false;
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (!PyLong_CheckExact(items[i])) return false;
        out[i] = PyLong_AsLongLong(items[i]);
    }
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    return true;
}

// conv(plan, X, W, packed, B, R, Y, workspace, stream): run (packed and R None), run_add (R given) or
// run_packed (packed given); with three more arguments (dims, strides, Y_rounded)
// packed is given, R, of those rows and columns, is read at every such row and column, and Y_rounded, if any, gets Y rounded;
// dims and strides None: R, if any, is read as it lies
PyObject *py_conv(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (n != 9 && n != 12) return slow_path();
    Plan *p = plan_of(a[0]);
    if (!p) { PyErr_Clear(); return slow_path(); }
    bool fine = true;
    const at::Tensor *xt = nullptr;
    size_t packed_bytes, ws_bytes;
    const float *x = in_ptr(a[1], fine, &xt), *w = in_ptr(a[2], fine);
    const void *packed = ws_ptr(a[3], packed_bytes, fine);
    const float *b = in_ptr(a[4], fine), *r = in_ptr(a[5], fine);
    float *y = const_cast<float *>(in_ptr(a[6], fine));
    void *ws = ws_ptr(a[7], ws_bytes, fine), *st = stream_ptr(a[8], fine);
    if (!fine || !x || !w) return slow_path();
    const bool pre = a[3] != Py_None;
    int64_t dims[2], every[2];
    float *y_rounded = n == 12 ? const_cast<float *>(in_ptr(a[11], fine)) : nullptr;
    const bool sampled = n == 12 && a[9] != Py_None;
    if (!fine || (n == 12 && !pre) || (sampled && (!r || a[10] == Py_None || !ints(a[9], dims, 2) || !ints(a[10], every, 2)))) return slow_path();
    at::Tensor ym, wm;
    if (!y) {
        ym = new_tensor(p->y, at::kFloat, xt->device(), a[8], st, true);
        y = static_cast<float *>(ym.data_ptr());
    }
    if (!ws && p->workspace && (!pre || p->packed_needs_ws || packed_bytes < p->packed)) {
        wm = new_tensor({(int64_t)p->workspace}, at::kByte, xt->device(), a[8], st, false);
        ws = wm.data_ptr();
        ws_bytes = p->workspace;
    }
    const onnxb_status s = sampled   ? abi.conv_run_packed_sampled(p->desc, x, w, packed, packed_bytes, b, r, dims, every, y, y_rounded, ws, ws_bytes, st)
                           : n == 12 ? abi.conv_run_packed_rounded(p->desc, x, w, packed, packed_bytes, b, r, y, y_rounded, ws, ws_bytes, st)
                           : pre ? abi.conv_run_packed(p->desc, x, w, packed, packed_bytes, b, r, y, ws, ws_bytes, st)
                           : r ? abi.conv_add_run(p->desc, x, w, b, r, y, ws, ws_bytes, st)
                               : abi.conv_run(p->desc, x, w, b, y, ws, ws_bytes, st);
    return s == ONNXB_OK ? result(a[6], ym) : slow_path();
}

// gemm(A, B, C, alpha, beta, transA, transB, relu, Y, workspace, stream)
PyObject *py_gemm(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (n != 11) return slow_path();
    bool fine = true;
    const at::Tensor *at_ = nullptr, *bt = nullptr, *ct = nullptr;
    const float *A = in_ptr(a[0], fine, &at_), *B = in_ptr(a[1], fine, &bt), *C = in_ptr(a[2], fine, &ct);
    const double alpha = PyFloat_AsDouble(a[3]), beta = PyFloat_AsDouble(a[4]);
    const int ta = PyObject_IsTrue(a[5]), tb = PyObject_IsTrue(a[6]), relu = PyObject_IsTrue(a[7]);
    if (PyErr_Occurred()) { PyErr_Clear(); return slow_path(); }
    float *y = const_cast<float *>(in_ptr(a[8], fine));
    size_t ws_bytes;
    void *ws = ws_ptr(a[9], ws_bytes, fine), *st = stream_ptr(a[10], fine);
    if (!fine || !A || !B || at_->dim() != 2 || bt->dim() != 2) return slow_path();
    const int64_t M = at_->size(ta ? 1 : 0), K = at_->size(ta ? 0 : 1), N = bt->size(tb ? 0 : 1);
    if (bt->size(tb ? 1 : 0) != K || (ct && ct->dim() > 2)) return slow_path();
    int64_t c_dims[2] = {1, 1};
    const int c_rank = ct ? (int)ct->dim() : 0;
    for (int i = 0; i < c_rank; ++i) c_dims[i] = ct->size(i);
    at::Tensor ym, wm;
    if (!y) {
        ym = new_tensor({M, N}, at::kFloat, at_->device(), a[10], st, true);
        y = static_cast<float *>(ym.data_ptr());
    }
    if (!ws) {
        const size_t need = abi.gemm_workspace_bytes(ta, tb, M, N, K);
        if (need) {
            wm = new_tensor({(int64_t)need}, at::kByte, at_->device(), a[10], st, false);
            ws = wm.data_ptr();
            ws_bytes = need;
        }
    }
    const onnxb_status s = abi.gemm_run(ta, tb, (float)alpha, (float)beta, M, N, K, A, B, C, c_rank, C ? c_dims : nullptr,
                                        relu, y, ws, ws_bytes, st);
    return s == ONNXB_OK ? result(a[8], ym) : slow_path();
}

// maxpool(X, kernel_shape, pads, strides, Y, stream)
PyObject *py_maxpool(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (n != 6) return slow_path();
    bool fine = true;
    const at::Tensor *xt = nullptr;
    const float *x = in_ptr(a[0], fine, &xt);
    int64_t ks[2], pads[4] = {0, 0, 0, 0}, st[2] = {0, 0}, yd[4];
    if (a[1] == Py_None || !ints(a[1], ks, 2) || !ints(a[2], pads, 4) || !ints(a[3], st, 2)) return slow_path();
    float *y = const_cast<float *>(in_ptr(a[4], fine));
    void *stream = stream_ptr(a[5], fine);
    if (!fine || !x || xt->dim() != 4) return slow_path();
    const int64_t *xd = xt->sizes().data();
    if (abi.maxpool2d_shape(xd, ks, pads, st, yd) != ONNXB_OK) return slow_path();
    at::Tensor ym;
    if (!y) {
        ym = new_tensor(yd, at::kFloat, xt->device(), a[5], stream, true);
        y = static_cast<float *>(ym.data_ptr());
    }
    return abi.maxpool2d_run(xd, ks, pads, st, x, y, stream) == ONNXB_OK ? result(a[4], ym) : slow_path();
}

// gap(X, Y, stream)
PyObject *py_gap(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (n != 3) return slow_path();
    bool fine = true;
    const at::Tensor *xt = nullptr;
    const float *x = in_ptr(a[0], fine, &xt);
    float *y = const_cast<float *>(in_ptr(a[1], fine));
    void *stream = stream_ptr(a[2], fine);
    if (!fine || !x || xt->dim() != 4) return slow_path();
    at::Tensor ym;
    if (!y) {
        ym = new_tensor({xt->size(0), xt->size(1), 1, 1}, at::kFloat, xt->device(), a[2], stream, true);
        y = static_cast<float *>(ym.data_ptr());
    }
    return abi.global_average_pool_run(xt->sizes().data(), x, y, stream) == ONNXB_OK ? result(a[1], ym) : slow_path();
}

// Address, type, sizes and strides of a tensor, or of those in a tuple or a dict (whose entry "input" is left out); false for anything else
bool add_state(PyObject *o, std::vector<int64_t> &out) {
    if (THPVariable_CheckExact(o)) {
        const at::Tensor &x = THPVariable_Unpack(o);
        out.push_back((int64_t)reinterpret_cast<uintptr_t>(x.data_ptr()));
        out.push_back((int64_t)x.scalar_type() << 32 | x.dim());
        out.insert(out.end(), x.sizes().begin(), x.sizes().end());
        out.insert(out.end(), x.strides().begin(), x.strides().end());
        return true;
    }
    if (PyTuple_CheckExact(o)) {
        for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(o); ++i)
            if (!add_state(PyTuple_GET_ITEM(o, i), out)) return false;
        return true;
    }
    if (!PyDict_CheckExact(o)) return false;
    PyObject *key, *value;
    for (Py_ssize_t i = 0; PyDict_Next(o, &i, &key, &value);) {
        if (!PyUnicode_Check(key)) return false;
        if (PyUnicode_CompareWithASCIIString(key, "input") != 0 && !add_state(value, out)) return false;
    }
    return true;
}

// state(tensors, tuples, dicts...): that of all of them and the library's dispatch state, as bytes
PyObject *py_state(PyObject *, PyObject *const *a, Py_ssize_t n) {
    std::vector<int64_t> out;
    out.reserve(4096);
    out.push_back((int64_t)abi.dispatch_state());
    for (Py_ssize_t i = 0; i < n; ++i)
        if (!add_state(a[i], out)) return slow_path();
    return PyBytes_FromStringAndSize(reinterpret_cast<const char *>(out.data()), (Py_ssize_t)(out.size() * sizeof(int64_t)));
}

// a C++ exception (out of memory, no device) also leads to the checked path, which raises its own
template <PyObject *(*F)(PyObject *, PyObject *const *, Py_ssize_t)>
PyObject *guarded(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    try {
        return F(self, a, n);
    } catch (...) {
        return slow_path();
    }
}

PyMethodDef methods[] = {
    {"bind", py_bind, METH_O, nullptr},
    {"plan", py_plan, METH_VARARGS, nullptr},
    {"conv", reinterpret_cast<PyCFunction>(&guarded<py_conv>), METH_FASTCALL, nullptr},
    {"gemm", reinterpret_cast<PyCFunction>(&guarded<py_gemm>), METH_FASTCALL, nullptr},
    {"maxpool", reinterpret_cast<PyCFunction>(&guarded<py_maxpool>), METH_FASTCALL, nullptr},
    {"gap", reinterpret_cast<PyCFunction>(&guarded<py_gap>), METH_FASTCALL, nullptr},
    {"state", reinterpret_cast<PyCFunction>(&guarded<py_state>), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_onnxb_fast", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__onnxb_fast(void) { return PyModule_Create(&module); }
