// Argument marshalling of the Python binding: device pointers of tensors and 32-bit integers of lists, as the raw bytes of
// the C arrays that the entry points take.  One call per array: with two Python-level calls per tensor the 32 pointers
// and two length lists of a 16-participant aggregation took 11.2 us, of an 18.2 us call whose kernel takes 13.
//
// Anything out of the ordinary (a None, a tensor subclass, a tensor that is not contiguous, an int beyond 32 bits) is
// answered by None: the caller then takes its general path, which converts it or raises.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include <exception>

#include <torch/csrc/autograd/python_variable.h>

namespace {

// false: not a plain contiguous tensor
bool pointer_of(PyObject *o, uint64_t *out)
{
    if (!THPVariable_CheckExact(o)) return false;
    try {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_contiguous()) return false;
        *out = (uint64_t)(uintptr_t)t.data_ptr();
        return true;
    } catch (const std::exception &) {                          // no storage: the general path raises what it always raised
        return false;
    }
}

// pointer(tensor) -> int or None
PyObject *pointer(PyObject *, PyObject *o)
{
    uint64_t x;
    if (!pointer_of(o, &x)) Py_RETURN_NONE;
    return PyLong_FromUnsignedLongLong(x);
}

// pointers(list or tuple of tensors) -> bytes of void *[n], or None
PyObject *pointers(PyObject *, PyObject *seq)
{
    if (!PyList_CheckExact(seq) && !PyTuple_CheckExact(seq)) Py_RETURN_NONE;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    PyObject *bytes = PyBytes_FromStringAndSize(nullptr, n * (Py_ssize_t)sizeof(uint64_t));
    if (!bytes) return nullptr;
    uint64_t *out = reinterpret_cast<uint64_t *>(PyBytes_AS_STRING(bytes));
    for (Py_ssize_t i = 0; i < n; ++i)
        if (!pointer_of(PySequence_Fast_GET_ITEM(seq, i), out + i)) {
            Py_DECREF(bytes);
            Py_RETURN_NONE;
        }
    return bytes;
}

// int32s(list or tuple of int) -> bytes of int32_t[n], or None
PyObject *int32s(PyObject *, PyObject *seq)
{
    if (!PyList_CheckExact(seq) && !PyTuple_CheckExact(seq)) Py_RETURN_NONE;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    PyObject *bytes = PyBytes_FromStringAndSize(nullptr, n * (Py_ssize_t)sizeof(int32_t));
    if (!bytes) return nullptr;
    int32_t *out = reinterpret_cast<int32_t *>(PyBytes_AS_STRING(bytes));
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject *o = PySequence_Fast_GET_ITEM(seq, i);
        int overflow = 0;
        const long x = PyLong_CheckExact(o) ? PyLong_AsLongAndOverflow(o, &overflow) : 0;
        if (!PyLong_CheckExact(o) || overflow || x != (long)(int32_t)x) {
            Py_DECREF(bytes);
            Py_RETURN_NONE;
        }
        out[i] = (int32_t)x;
    }
    return bytes;
}

PyMethodDef methods[] = {{"pointer", pointer, METH_O, nullptr},
                         {"pointers", pointers, METH_O, nullptr},
                         {"int32s", int32s, METH_O, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fedattn_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fedattn_marshal(void) { return PyModule_Create(&module); }
