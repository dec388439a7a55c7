// The call from Python into the C ABI: one CPython function that turns its arguments into machine words and calls an entry
// point.  A pruning step on one image takes 9 us from Python and has 27 arguments; marshalled by ctypes they alone took 10 us
// of host time per call, so that the caller, not the GPU, set the pace.
//
//   bind(name, address) -> handle     of the entry point `name`, which the loaded library has at `address`
//   call(handle, scale, *args) -> int
//     args      the entry point's arguments in order, without its float argument if it has one, which is `scale`
//               None -> null / 0, int -> itself, bytes -> pointer to its data (parameter structs), CUDA tensor -> data pointer
// Every entry point is called through its own type (taken from the header), each word converted to the parameter's type, so
// nothing depends on a calling convention.  The interpreter lock is released during the call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <cstring>
#include <type_traits>
#include <utility>

#include "vitcop.h"

namespace {

constexpr int kMaxArgs = 36;

template <typename T>
T from_word(int64_t word, float scale) {
    if constexpr (std::is_floating_point_v<T>) return static_cast<T>(scale);
    else if constexpr (std::is_pointer_v<T>) return reinterpret_cast<T>(static_cast<uintptr_t>(word));
    else return static_cast<T>(word);
}

// How many of the first n parameters are integers or pointers: the word that parameter n takes.
template <typename... A>
constexpr int words_before(size_t n) {
    constexpr bool is_float[] = {std::is_floating_point_v<A>...};
    int w = 0;
    for (size_t i = 0; i < n; ++i) w += is_float[i] ? 0 : 1;
    return w;
}

template <typename... A, size_t... I>
int invoke(int (*f)(A...), const int64_t* words, float scale, std::index_sequence<I...>) {
    return f(from_word<A>(words[words_before<A...>(I) < kMaxArgs ? words_before<A...>(I) : 0], scale)...);
}

template <typename F>
struct Signature;
template <typename... A>
struct Signature<int(A...)> {
    static constexpr int kWords = words_before<A...>(sizeof...(A));
    static_assert(kWords <= kMaxArgs, "arguments of an entry point");
    static int call(uintptr_t address, const int64_t* words, float scale) {
        return invoke(reinterpret_cast<int (*)(A...)>(address), words, scale, std::index_sequence_for<A...>{});
    }
};

struct Entry {
    const char* name;
    int words;
    int (*call)(uintptr_t, const int64_t*, float);
    uintptr_t address;
};
#define ENTRY(name) {#name, Signature<decltype(name)>::kWords, Signature<decltype(name)>::call, 0}
Entry entries[] = {
    ENTRY(vitcop_knorm_score), ENTRY(vitcop_select), ENTRY(vitcop_compact_kv), ENTRY(vitcop_prune_step),
    ENTRY(vitcop_prune_step_static), ENTRY(vitcop_collaborative_step), ENTRY(vitcop_merge_clusters),
    ENTRY(vitcop_cls_saliency), ENTRY(vitcop_kproj_knorm), ENTRY(vitcop_redundancy_filter), ENTRY(vitcop_similarity_rows)};
constexpr int kEntries = sizeof(entries) / sizeof(entries[0]);

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

PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    const char* const name = n == 2 ? PyUnicode_AsUTF8(args[0]) : nullptr;
    if (!name) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "bind(name, address)");
        return nullptr;
    }
    const unsigned long long address = PyLong_AsUnsignedLongLong(args[1]);
    if (PyErr_Occurred()) return nullptr;
    for (int e = 0; e < kEntries; ++e) {
        if (std::strcmp(entries[e].name, name) == 0) {
            entries[e].address = static_cast<uintptr_t>(address);
            return PyLong_FromLong(e);
        }
    }
    PyErr_Format(PyExc_KeyError, "no such entry point: %.100s", name);
    return nullptr;
}

PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n < 2 || n - 2 > kMaxArgs) {
        PyErr_SetString(PyExc_TypeError, "call(handle, scale, *args): wrong number of arguments");
        return nullptr;
    }
    const long handle = PyLong_AsLong(args[0]);
    if (PyErr_Occurred()) return nullptr;
    if (handle < 0 || handle >= kEntries || entries[handle].address == 0) {
        PyErr_SetString(PyExc_ValueError, "call: not a handle of bind");
        return nullptr;
    }
    const Entry& e = entries[handle];
    const double scale = PyFloat_AsDouble(args[1]);
    if (PyErr_Occurred()) return nullptr;
    int64_t a[kMaxArgs] = {};
    for (Py_ssize_t i = 2; i < n; ++i) {
        bool ok;
        try {
            ok = to_word(args[i], a[i - 2]);
        } catch (const std::exception& ex) {
            PyErr_SetString(PyExc_RuntimeError, ex.what());
            ok = false;
        }
        if (!ok) return nullptr;
    }
    if (n - 2 != e.words) {
        PyErr_Format(PyExc_TypeError, "%s takes %d arguments, got %zd", e.name, e.words, n - 2);
        return nullptr;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = e.call(e.address, a, static_cast<float>(scale));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(bind)), METH_FASTCALL, "bind(name, address) -> handle"},
    {"call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call)), METH_FASTCALL, "call(handle, scale, *args) -> int"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", "Calls the entry points of the C ABI.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call(void) { return PyModule_Create(&module); }
