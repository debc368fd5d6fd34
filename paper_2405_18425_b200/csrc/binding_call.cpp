// One call of a device entry point of the C ABI from Python: checks the tensors, takes their addresses and sizes and the
// current stream, and calls.  The same marshalling in Python and ctypes cost 4 to 8 us a call, of the 6 to 10 us a small call
// took altogether (a training step of 384 units of 49 tokens was bound by its four calls: 29 us for 21 us of kernels).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using P = const void*;
using W = void*;   // (pointers are passed alike whatever they point to)
constexpr int kMaxTensors = 11;

// call(address, stream or None, v, same_dtype, tau or None, tensor, ...): status of the entry point.  Sizes come from the
// four dimensions of the first tensor and, with v >= 0, the last of tensor v; a None among the tensors is a null pointer.
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    const Py_ssize_t nt = nargs - 5;
    if (nt < 1 || nt > kMaxTensors) {
        PyErr_SetString(PyExc_TypeError, "call(address, stream, v, same_dtype, tau, tensor, ...)");
        return nullptr;
    }
    void* fn = PyLong_AsVoidPtr(args[0]);
    if (!fn) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point");
        return nullptr;
    }
    const long vi = PyLong_AsLong(args[2]);
    const int same = PyObject_IsTrue(args[3]);
    const bool has_tau = args[4] != Py_None;
    const float tau = has_tau ? (float)PyFloat_AsDouble(args[4]) : 0.f;
    if (PyErr_Occurred()) return nullptr;
    W p[kMaxTensors];
    int d[5] = {0, 0, 0, 0, 0};
    at::ScalarType type = at::ScalarType::Undefined;
    for (Py_ssize_t i = 0; i < nt; ++i) {
        PyObject* o = args[5 + i];
        if (o == Py_None && i > 0) {
            p[i] = nullptr;
            continue;
        }
        if (!THPVariable_Check(o)) {
            PyErr_SetString(PyExc_TypeError, "device entry points take torch tensors");
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_ValueError, "device entry points take contiguous CUDA tensors");
            return nullptr;
        }
        if (i == 0 || i == vi) {
            if (t.dim() != 4) {
                PyErr_SetString(PyExc_ValueError, "tensors of four dimensions expected");
                return nullptr;
            }
            if (i == 0)
                for (int x = 0; x < 4; ++x) d[x] = (int)t.size(x);
            if (i == vi) d[4] = (int)t.size(3);
        }
        if (i == 0) type = t.scalar_type();
        else if (same && t.scalar_type() != type) {
            PyErr_SetString(PyExc_ValueError, "all tensors of one call share a dtype");
            return nullptr;
        }
        p[i] = t.data_ptr();
    }
    W stream = nullptr;
    if (args[1] == Py_None) {
        stream = c10::cuda::getCurrentCUDAStream().stream();
    } else {
        stream = PyLong_AsVoidPtr(args[1]);
        if (PyErr_Occurred()) return nullptr;
    }
    int status = 0;
    bool known = true;
    const int kind = (int)nt * 4 + (vi >= 0 ? 2 : 0) + (has_tau ? 1 : 0);
    Py_BEGIN_ALLOW_THREADS
    switch (kind) {
        case 4 * 4 + 0:
            status = reinterpret_cast<int (*)(P, P, P, W, int, int, int, int, W)>(fn)(p[0], p[1], p[2], p[3], d[0], d[1], d[2], d[3], stream);
            break;
        case 4 * 4 + 1:
            status = reinterpret_cast<int (*)(P, P, W, W, int, int, int, int, float, W)>(fn)(p[0], p[1], p[2], p[3], d[0], d[1], d[2], d[3], tau, stream);
            break;
        case 6 * 4 + 1:
            status = reinterpret_cast<int (*)(P, P, P, P, W, W, int, int, int, int, float, W)>(fn)(p[0], p[1], p[2], p[3], p[4], p[5], d[0], d[1], d[2],
                                                                                                   d[3], tau, stream);
            break;
        case 6 * 4 + 2:
            status = reinterpret_cast<int (*)(P, P, P, P, P, W, int, int, int, int, int, W)>(fn)(p[0], p[1], p[2], p[3], p[4], p[5], d[0], d[1], d[2],
                                                                                                 d[3], d[4], stream);
            break;
        case 6 * 4 + 3:
            status = reinterpret_cast<int (*)(P, P, P, P, P, W, int, int, int, int, int, float, W)>(fn)(p[0], p[1], p[2], p[3], p[4], p[5], d[0], d[1],
                                                                                                        d[2], d[3], d[4], tau, stream);
            break;
        case 8 * 4 + 3:
            status = reinterpret_cast<int (*)(P, P, P, P, P, P, P, W, int, int, int, int, int, float, W)>(fn)(
                p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], d[0], d[1], d[2], d[3], d[4], tau, stream);
            break;
        case 11 * 4 + 2:
            status = reinterpret_cast<int (*)(P, P, P, P, P, P, W, W, W, W, W, int, int, int, int, int, W)>(fn)(
                p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], p[9], p[10], d[0], d[1], d[2], d[3], d[4], stream);
            break;
        default: known = false;
    }
    Py_END_ALLOW_THREADS
    if (!known) {
        PyErr_SetString(PyExc_TypeError, "no entry point takes these arguments");
        return nullptr;
    }
    return PyLong_FromLong(status);
    END_HANDLE_TH_ERRORS
}

PyMethodDef kMethods[] = {{"call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call)), METH_FASTCALL, "calls a device entry point"},
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_binding_call", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding_call() { return PyModule_Create(&kModule); }
