// The per-layer calls of the binding without ctypes: a serving loop calls w4a8_quantize_act and w4a8_linear
// once per layer each, and at a few microseconds of device time the call itself is what it waits for.
// Through ctypes a call cost about 7 us (five to eight pointer objects, a conversion per argument, attribute
// look-ups on the tensors); here the tensors' addresses and strides are read directly, which leaves the
// launch.  Marshalling only: every check and decision is the C-ABI library's.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "../../include/w4a8.h"

namespace {

// Thrown after a Python error has been set.
struct Raised {};

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "expected a tensor, got %s", Py_TYPE(o)->tp_name);
        throw Raised{};
    }
    return THPVariable_Unpack(o);
}
void* address(PyObject* o) { return o == Py_None ? nullptr : tensor(o).data_ptr(); }
int64_t integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
void check(bool ok, const char* what) {
    if (!ok) {
        PyErr_SetString(PyExc_AssertionError, what);
        throw Raised{};
    }
}

template <class F>
PyObject* guarded(Py_ssize_t nargs, Py_ssize_t want, F f) {
    if (nargs != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
        return nullptr;
    }
    try {
        return PyLong_FromLong(f());
    } catch (const Raised&) {
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    } catch (...) {
        PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
    }
    return nullptr;
}

// (x, x8, s_x, scale_mode, static_scale or None) -> status
PyObject* quantize_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 5, [&]() -> int {
        const at::Tensor &x = tensor(a[0]), &x8 = tensor(a[1]);
        check(x.is_cuda() && x.scalar_type() == at::kBFloat16 && x.dim() == 2 && x.stride(1) == 1,
              "x: BF16 [M, K] on the device, contiguous along K");
        const void* xp = x.data_ptr();
        const int64_t M = x.size(0), K = x.size(1), ldx = x.stride(0), ldx8 = x8.stride(0);
        uint8_t* x8p = static_cast<uint8_t*>(x8.data_ptr());
        float* sp = static_cast<float*>(address(a[2]));
        const int mode = static_cast<int>(integer(a[3]));
        const float* ss = static_cast<const float*>(address(a[4]));
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = w4a8_quantize_act(xp, M, K, ldx, x8p, ldx8, sp, mode, ss, stream);
        Py_END_ALLOW_THREADS
        return rc;
    });
}

// (x8, s_x, weights, gscale or None, gzero or None, format, s_w, N, K, group, out, out_dtype, workspace or None) -> status
PyObject* linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 13, [&]() -> int {
        const at::Tensor &x8 = tensor(a[0]), &s_w = tensor(a[6]), &out = tensor(a[10]);
        check(x8.dim() == 2, "x8: [M, K]");
        const int64_t M = x8.size(0), N = integer(a[7]), K = integer(a[8]);
        check(x8.size(1) == K, "x8 and the weights differ in K");
        const uint8_t* xp = static_cast<const uint8_t*>(x8.data_ptr());
        const float* sp = static_cast<const float*>(address(a[1]));
        const uint8_t* wp = static_cast<const uint8_t*>(address(a[2]));
        const void* gs = address(a[3]);
        const uint8_t* gz = static_cast<const uint8_t*>(address(a[4]));
        const float* sw = static_cast<const float*>(s_w.data_ptr());
        const int64_t ldx8 = x8.stride(0), ldy = out.stride(0);
        void* yp = out.data_ptr();
        void* ws = address(a[12]);
        const size_t wsn = ws ? tensor(a[12]).nbytes() : 0;
        const int fmt = static_cast<int>(integer(a[5])), group = static_cast<int>(integer(a[9])),
                  od = static_cast<int>(integer(a[11])), sw_stride = s_w.numel() == 1 ? 0 : 1;
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = w4a8_linear(xp, ldx8, sp, M, wp, gs, gz, fmt, sw, sw_stride, N, K, group, yp, ldy, od, ws, wsn, stream);
        Py_END_ALLOW_THREADS
        return rc;
    });
}

// (M, N, K, format) -> bytes
PyObject* linear_workspace_bytes(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 4, [&]() -> long {
        return static_cast<long>(w4a8_linear_workspace_bytes(integer(a[0]), integer(a[1]), integer(a[2]),
                                                             static_cast<int>(integer(a[3]))));
    });
}

PyMethodDef methods[] = {
    {"quantize_act", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(quantize_act)), METH_FASTCALL, nullptr},
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear)), METH_FASTCALL, nullptr},
    {"linear_workspace_bytes", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear_workspace_bytes)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
// (the versions that it was compiled against: the build looks for them and compiles again for others)
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_w4a8_host", W4A8_HOST_VERSIONS, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__w4a8_host(void) { return PyModule_Create(&module); }
