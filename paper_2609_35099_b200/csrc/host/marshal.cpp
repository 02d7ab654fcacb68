// The Python binding's inner loop in native code: what every call of the C ABI does per argument (is it a contiguous
// CUDA tensor of that type and shape, where does it start), the outputs' allocation and the call itself.  With small
// graphs the host side of a call is what it costs: forward and backward of 64 atoms and 8 channels convert 22 tensors,
// allocate six and pass 36 arguments (39 us a step in Python and ctypes, 23 us here).
//
// Nothing is decided here: a tensor that is not plainly what the entry point takes goes to the binding's own Python
// function, which raises the error (or copes with what this file does not know: subclasses, wrapped tensors).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

namespace {

PyObject *g_slow_ptr = nullptr, *g_slow_empty = nullptr;   // _dev_ptr and _empty of the binding

bool shape_is(const at::Tensor& t, PyObject* shape) {
    if (shape == Py_None) return true;
    if (!PyTuple_CheckExact(shape) || PyTuple_GET_SIZE(shape) != (Py_ssize_t)t.dim()) return false;
    for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(shape); ++i) {
        PyObject* n = PyTuple_GET_ITEM(shape, i);
        if (!PyLong_CheckExact(n) || PyLong_AsLongLong(n) != t.size(i)) return false;
    }
    return true;
}

// dev_ptr(tensor or None, dtype, shape or None, name) -> address or None
PyObject* dev_ptr(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 4) {
        PyErr_SetString(PyExc_TypeError, "dev_ptr takes a tensor, a dtype, a shape and a name");
        return nullptr;
    }
    if (args[0] == Py_None) Py_RETURN_NONE;
    if (THPVariable_CheckExact(args[0]) && THPDtype_Check(args[1])) {
        try {
            const at::Tensor& t = THPVariable_Unpack(args[0]);
            if (t.is_cuda() && t.layout() == at::kStrided && t.has_storage() &&
                t.scalar_type() == reinterpret_cast<THPDtype*>(args[1])->scalar_type && t.is_contiguous() &&
                !t.is_conj() && !t.is_neg() && shape_is(t, args[2]))
                return PyLong_FromUnsignedLongLong((unsigned long long)(uintptr_t)t.data_ptr());
        } catch (...) {   // (symbolic sizes, tensors without data)
        }
        PyErr_Clear();
    }
    return PyObject_Vectorcall(g_slow_ptr, args, 4, nullptr);
}

// empty(shape, dtype, like) -> an uninitialised tensor on like's device
PyObject* empty(PyObject*, PyObject* const* args, Py_ssize_t n) {
    constexpr Py_ssize_t kMostDims = 4;
    if (n != 3) {
        PyErr_SetString(PyExc_TypeError, "empty takes a shape, a dtype and a tensor");
        return nullptr;
    }
    if (PyTuple_CheckExact(args[0]) && PyTuple_GET_SIZE(args[0]) <= kMostDims && THPDtype_Check(args[1]) && THPVariable_CheckExact(args[2])) {
        int64_t sizes[kMostDims];
        const Py_ssize_t dims = PyTuple_GET_SIZE(args[0]);
        bool plain = true;
        for (Py_ssize_t i = 0; i < dims; ++i) {
            PyObject* v = PyTuple_GET_ITEM(args[0], i);
            plain = plain && PyLong_CheckExact(v);
            sizes[i] = plain ? PyLong_AsLongLong(v) : 0;
        }
        if (PyErr_Occurred()) PyErr_Clear(), plain = false;
        if (plain) {
            HANDLE_TH_ERRORS
            const auto options = at::TensorOptions().dtype(reinterpret_cast<THPDtype*>(args[1])->scalar_type).device(THPVariable_Unpack(args[2]).device());
            at::Tensor t;
            {
                pybind11::gil_scoped_release no_gil;   // (an allocation may wait for the device)
                t = at::empty(at::IntArrayRef(sizes, dims), options);
            }
            return THPVariable_Wrap(std::move(t));
            END_HANDLE_TH_ERRORS
        }
    }
    return PyObject_Vectorcall(g_slow_empty, args, 3, nullptr);
}

// call(address, arguments...) -> status, call_size for functions that return a size (of a plan and integers; where an entry
// point takes pointers and integers, the binding has formed the integers from shapes or computed with them).  Every parameter of the C ABI is an
// integer or a pointer and has a 64-bit slot of its own in the calling convention, so one signature serves all entry
// points; slots behind the last are not read.  None is NULL, for the first `pointers` arguments alone.
constexpr int kMostArgs = 24;
template <class R>
bool invoke(PyObject* const* args, Py_ssize_t n, Py_ssize_t pointers, R& result) {
    if (n < 1 || n > kMostArgs + 1) {
        PyErr_SetString(PyExc_TypeError, "an address and up to 24 arguments");
        return false;
    }
    uint64_t v[kMostArgs + 1] = {};
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (args[i] == Py_None && i > 0 && i <= pointers) continue;
        v[i] = PyLong_AsUnsignedLongLongMask(args[i]);
        if (v[i] == (uint64_t)-1 && PyErr_Occurred()) return false;
    }
    using U = uint64_t;
    using Entry = R (*)(U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U, U);
    const Entry f = reinterpret_cast<Entry>((uintptr_t)v[0]);
    Py_BEGIN_ALLOW_THREADS
    result = f(v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], v[10], v[11], v[12], v[13], v[14], v[15], v[16], v[17],
               v[18], v[19], v[20], v[21], v[22], v[23], v[24]);
    Py_END_ALLOW_THREADS
    return true;
}
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
    int status;
    return invoke(args, n, kMostArgs, status) ? PyLong_FromLong(status) : nullptr;
}
PyObject* call_size(PyObject*, PyObject* const* args, Py_ssize_t n) {
    size_t bytes;
    return invoke(args, n, 1, bytes) ? PyLong_FromSize_t(bytes) : nullptr;
}

// set_slow(dev_ptr, empty): what the two functions above fall back on
PyObject* set_slow(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 2) {
        PyErr_SetString(PyExc_TypeError, "set_slow takes two functions");
        return nullptr;
    }
    Py_INCREF(args[0]);
    Py_XSETREF(g_slow_ptr, args[0]);
    Py_INCREF(args[1]);
    Py_XSETREF(g_slow_empty, args[1]);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"dev_ptr", (PyCFunction)(void (*)(void))dev_ptr, METH_FASTCALL, nullptr},
    {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, nullptr},
    {"call_size", (PyCFunction)(void (*)(void))call_size, METH_FASTCALL, nullptr},
    {"empty", (PyCFunction)(void (*)(void))empty, METH_FASTCALL, nullptr},
    {"set_slow", (PyCFunction)(void (*)(void))set_slow, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// built_for: the torch and the interpreter whose object layouts are compiled in here; the binding uses the module with
// these alone.
PyMODINIT_FUNC PyInit__marshal() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", E3J_BUILT_FOR) != 0) Py_CLEAR(m);
    return m;
}
