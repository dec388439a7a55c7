// The call from Python into the C ABI: one CPython function that turns its arguments into machine words and calls an entry
// point by address.  A pruning step on one image takes 12 us on the GPU and has 27 arguments; marshalled by ctypes they
// alone took 10 us of host time per call, so that the caller, not the GPU, set the pace.
//
//   call(address, scale, *args) -> int
//     address   of an entry point that returns int and takes pointers, integers and at most one float, which is `scale`
//     args      None -> null / 0, int -> itself, bytes -> pointer to its data (parameter structs), CUDA tensor -> data pointer
// On x86-64 (System V) the integer arguments of a call sit in order in six registers and then in 8-byte stack slots, whatever
// their widths, and a float argument sits in its own register file wherever it stands in the list; a caller may pass more
// than the callee takes.  So one signature serves every entry point.  The interpreter lock is released during the call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

#if !defined(__x86_64__)
#error "written for the System V calling convention of x86-64"
#endif

namespace {

constexpr int kMaxArgs = 36;
typedef int (*EntryPoint)(float, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t,
                          int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t,
                          int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t,
                          int64_t, int64_t, int64_t, int64_t);

bool to_word(PyObject* o, int64_t& v) {
    if (o == Py_None) {
        v = 0;
        return true;
    }
    if (PyLong_Check(o)) {
        v = PyLong_AsLongLong(o);
        return !(v == -1 && PyErr_Occurred());
    }
    if (THPVariable_Check(o)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda()) {
            PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor");
            return false;
        }
        if (!t.is_contiguous()) {
            PyErr_SetString(PyExc_ValueError, "expected a contiguous tensor");
            return false;
        }
        v = static_cast<int64_t>(reinterpret_cast<uintptr_t>(t.data_ptr()));
        return true;
    }
    if (PyBytes_Check(o)) {
        v = static_cast<int64_t>(reinterpret_cast<uintptr_t>(PyBytes_AS_STRING(o)));
        return true;
    }
    PyErr_Format(PyExc_TypeError, "expected a tensor, an int, bytes or None, got %.100s", Py_TYPE(o)->tp_name);
    return false;
}

PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n < 2 || n - 2 > kMaxArgs) {
        PyErr_SetString(PyExc_TypeError, "call(address, scale, *args): wrong number of arguments");
        return nullptr;
    }
    const unsigned long long address = PyLong_AsUnsignedLongLong(args[0]);
    if (PyErr_Occurred()) return nullptr;
    const double scale = PyFloat_AsDouble(args[1]);
    if (PyErr_Occurred()) return nullptr;
    int64_t a[kMaxArgs] = {};
    for (Py_ssize_t i = 2; i < n; ++i) {
        bool ok;
        try {
            ok = to_word(args[i], a[i - 2]);
        } catch (const std::exception& e) {
            PyErr_SetString(PyExc_RuntimeError, e.what());
            ok = false;
        }
        if (!ok) return nullptr;
    }
    const EntryPoint f = reinterpret_cast<EntryPoint>(static_cast<uintptr_t>(address));
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f(static_cast<float>(scale), a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13],
           a[14], a[15], a[16], a[17], a[18], a[19], a[20], a[21], a[22], a[23], a[24], a[25], a[26], a[27], a[28], a[29],
           a[30], a[31], a[32], a[33], a[34], a[35]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyMethodDef methods[] = {
    {"call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call)), METH_FASTCALL, "call(address, scale, *args) -> int"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", "Calls C entry points by address.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call(void) { return PyModule_Create(&module); }
