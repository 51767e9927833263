// CPython entries, first of all for the call that a decoder makes most, dps_linear: argument checks, output allocation and the current stream
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

// ---- the calls that load a model and serve experts --------------------------------------------------------------------
// A loader waits for the answer of an AUTO split before it can go on, and the GPU waits with it: a layer of four tensors, split
// and rebuilt, takes 291 us through here, 309 through ctypes; two grouped calls occupy the host for 15-25 us instead of 35-46.

struct Functions {
    int (*split)(const void*, uint8_t*, uint8_t*, int64_t, int64_t, int32_t*, void*) = nullptr;
    int (*reconstruct)(const uint8_t*, const uint8_t*, void*, int64_t, int64_t, int32_t, void*) = nullptr;
    int (*moe)(int32_t, const int32_t*, const void*, const int32_t*, const int32_t*, const uint8_t*, const uint8_t*, void*, int64_t,
               int64_t, int64_t, int64_t, int32_t, void*, size_t, void*) = nullptr;
} g_fn;

// set_functions(addresses of dps_split_weights, dps_reconstruct, dps_moe_linear)
PyObject* set_functions(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 3) {
        PyErr_SetString(PyExc_TypeError, "three addresses");
        return nullptr;
    }
    void* at[3];
    for (int i = 0; i < 3; ++i) {
        at[i] = PyLong_AsVoidPtr(args[i]);
        if (PyErr_Occurred()) return nullptr;
    }
    g_fn.split = reinterpret_cast<decltype(g_fn.split)>(at[0]);
    g_fn.reconstruct = reinterpret_cast<decltype(g_fn.reconstruct)>(at[1]);
    g_fn.moe = reinterpret_cast<decltype(g_fn.moe)>(at[2]);
    Py_RETURN_NONE;
}

// A plain CUDA tensor of this type, `dims` dimensions (0: any) in `arg`.  None leaves `out` undefined if `optional`.
bool take(PyObject* arg, at::ScalarType type, int dims, bool optional, at::Tensor& out) {
    if (arg == Py_None) return optional;
    if (!THPVariable_CheckExact(arg)) return false;
    out = THPVariable_Unpack(arg);
    return plain(out, type) && (dims == 0 || out.dim() == dims);
}
bool small_int(PyObject* arg, int32_t& out) {
    if (!PyLong_Check(arg)) return false;
    const long v = PyLong_AsLong(arg);
    if (v == -1 && PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    out = (int32_t)v;
    return v >= 0 && v <= 255;
}
at::Tensor new_like(const at::Tensor& t, at::IntArrayRef size, at::ScalarType type) {
    return at::empty(size, at::TensorOptions().dtype(type).device(t.device()));
}
void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
// the caller's object where there is one, else a new one around the tensor
PyObject* give(PyObject* arg, const at::Tensor& t) {
    if (arg == Py_None) return THPVariable_Wrap(t);
    Py_INCREF(arg);
    return arg;
}

// split_weights(w, enc, w_persist or None, w_resid or None) -> (w_persist, w_resid, enc), a status that is not 0, or None
PyObject* split_weights(PyObject*, PyObject* const* args, Py_ssize_t n) {
    int32_t enc = 0;
    if (n != 4 || g_fn.split == nullptr || !small_int(args[1], enc)) Py_RETURN_NONE;
    try {
        at::Tensor w, p, r;
        if (!take(args[0], at::kHalf, 2, false, w) || !take(args[2], at::kByte, 0, true, p) || !take(args[3], at::kByte, 0, true, r))
            Py_RETURN_NONE;
        int status = 0;
        {
            WithoutGil nogil;
            if (!p.defined()) p = new_like(w, w.sizes(), at::kByte);
            if (!r.defined()) r = new_like(w, w.sizes(), at::kByte);
            status = g_fn.split(w.const_data_ptr(), p.mutable_data_ptr<uint8_t>(), r.mutable_data_ptr<uint8_t>(), w.size(0), w.size(1),
                                &enc, current_stream());
        }
        if (status != 0) return PyLong_FromLong(status);
        return Py_BuildValue("(NNi)", give(args[2], p), give(args[3], r), (int)enc);
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// reconstruct(w_persist, w_resid or None, enc, out or None) -> out, a status that is not 0, or None
PyObject* reconstruct(PyObject*, PyObject* const* args, Py_ssize_t n) {
    int32_t enc = 0;
    if (n != 4 || g_fn.reconstruct == nullptr || !small_int(args[2], enc)) Py_RETURN_NONE;
    try {
        at::Tensor p, r, w;
        if (!take(args[0], at::kByte, 2, false, p) || !take(args[1], at::kByte, 0, true, r) || !take(args[3], at::kHalf, 0, true, w))
            Py_RETURN_NONE;
        int status = 0;
        {
            WithoutGil nogil;
            if (!w.defined()) w = new_like(p, p.sizes(), at::kHalf);
            status = g_fn.reconstruct(p.const_data_ptr<uint8_t>(), r.defined() ? r.const_data_ptr<uint8_t>() : nullptr, w.mutable_data_ptr(),
                                      p.size(0), p.size(1), enc, current_stream());
        }
        if (status != 0) return PyLong_FromLong(status);
        return give(args[3], w);
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// moe_linear(mode, encodings, x, token_of_row or None, expert_of_row, w_persist, w_resid or None, y or None, workspace)
// -> y, a status that is not 0, or None
PyObject* moe_linear(PyObject*, PyObject* const* args, Py_ssize_t n) {
    constexpr Py_ssize_t kMaxExperts = 1024;
    int32_t mode = 0, enc[kMaxExperts];
    if (n != 9 || g_fn.moe == nullptr || !small_int(args[0], mode)) Py_RETURN_NONE;
    if (!PyList_CheckExact(args[1]) && !PyTuple_CheckExact(args[1])) Py_RETURN_NONE;
    const Py_ssize_t experts = PySequence_Fast_GET_SIZE(args[1]);
    if (experts > kMaxExperts) Py_RETURN_NONE;
    for (Py_ssize_t i = 0; i < experts; ++i)
        if (!small_int(PySequence_Fast_GET_ITEM(args[1], i), enc[i])) Py_RETURN_NONE;
    try {
        at::Tensor x, token, expert, p, r, y, workspace;
        if (!take(args[2], at::kHalf, 2, false, x) || !take(args[3], at::kInt, 0, true, token) || !take(args[4], at::kInt, 0, false, expert) ||
            !take(args[5], at::kByte, 3, false, p) || !take(args[6], at::kByte, 0, true, r) || !take(args[7], at::kHalf, 0, true, y) ||
            !take(args[8], at::kByte, 0, false, workspace))
            Py_RETURN_NONE;
        if (p.size(0) != experts || x.size(1) != p.size(2)) Py_RETURN_NONE;
        const int64_t rows = expert.numel();
        int status = 0;
        {
            WithoutGil nogil;
            if (!y.defined()) y = new_like(x, {rows, p.size(1)}, at::kHalf);
            status = g_fn.moe(mode, enc, x.const_data_ptr(), token.defined() ? token.const_data_ptr<int32_t>() : nullptr,
                              expert.const_data_ptr<int32_t>(), p.const_data_ptr<uint8_t>(),
                              r.defined() ? r.const_data_ptr<uint8_t>() : nullptr, y.mutable_data_ptr(), rows, x.size(0), p.size(1),
                              p.size(2), (int32_t)experts, workspace.mutable_data_ptr(), (size_t)workspace.numel(), current_stream());
        }
        if (status != 0) return PyLong_FromLong(status);
        return give(args[7], y);
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

#define DPS_FASTCALL(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    {"set_linear", set_linear, METH_O, nullptr},
    DPS_FASTCALL(set_functions),
    DPS_FASTCALL(linear),
    DPS_FASTCALL(split_weights),
    DPS_FASTCALL(reconstruct),
    DPS_FASTCALL(moe_linear),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&g_module); }
