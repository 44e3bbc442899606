// CPython side of the calls a training or generation loop makes (binding.py has the signatures): arguments in the order of the C
// ABI, tensors turned into device pointers, one call, the status back.  ctypes took 11 - 13 us per call for the same -- more than
// the kernels of a few-token call run -- this takes 5 - 6 with the launches included (512 x 512, 64 tokens: 38 -> 28 us per step).
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <pthread.h>

#include <cstddef>
#include <cstdint>
#include <tuple>
#include <type_traits>
#include <utility>

#include "qlora.h"

namespace {

PyObject* g_desc_type = nullptr;                     // the ctypes structure of qlora_desc
PyObject *s_is_contiguous, *s_data_ptr, *s_cuda_stream, *s_numel, *s_element_size, *s_current_stream;
PyObject *g_torch_cuda = nullptr, *g_get_device = nullptr, *g_raw_stream = nullptr;
bool g_cuda_ready = false;                           // torch has initialised CUDA in this process

void in_child() { g_cuda_ready = false; }            // (a forked child goes through torch's own check again)

bool call_long(PyObject* callable_result, unsigned long long* out) {   // steals the reference
    if (callable_result == nullptr) return false;
    *out = PyLong_AsUnsignedLongLongMask(callable_result);
    Py_DECREF(callable_result);
    return !(*out == (unsigned long long)-1 && PyErr_Occurred());
}
bool method_long(PyObject* obj, PyObject* name, unsigned long long* out) { return call_long(PyObject_CallMethodNoArgs(obj, name), out); }

// A tensor's device pointer; None -> NULL; an int is passed through.
bool to_pointer(PyObject* t, void** out) {
    unsigned long long v = 0;
    if (t == Py_None) { *out = nullptr; return true; }
    if (PyLong_Check(t)) {
        v = PyLong_AsUnsignedLongLongMask(t);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) return false;
    } else {
        PyObject* c = PyObject_CallMethodNoArgs(t, s_is_contiguous);
        if (c == nullptr) return false;
        const int yes = PyObject_IsTrue(c);
        Py_DECREF(c);
        if (yes < 0) return false;
        if (!yes) { PyErr_SetString(PyExc_ValueError, "tensors must be contiguous (dense row-major)"); return false; }
        if (!method_long(t, s_data_ptr, &v)) return false;
    }
    *out = reinterpret_cast<void*>((uintptr_t)v);
    return true;
}

// None -> torch's current stream on the current device; an int is passed through; else an object with `cuda_stream`.
bool to_stream(PyObject* s, void** out) {
    unsigned long long v = 0;
    if (PyLong_Check(s)) {
        v = PyLong_AsUnsignedLongLongMask(s);
        if (v == (unsigned long long)-1 && PyErr_Occurred()) return false;
    } else if (s != Py_None) {
        if (!call_long(PyObject_GetAttr(s, s_cuda_stream), &v)) return false;
    } else if (g_cuda_ready) {
        PyObject* dev = PyObject_CallNoArgs(g_get_device);
        if (dev == nullptr) return false;
        PyObject* raw = PyObject_CallOneArg(g_raw_stream, dev);
        Py_DECREF(dev);
        if (!call_long(raw, &v)) return false;
    } else {                                         // the first time: torch's own way, which initialises CUDA or says why it cannot
        if (g_torch_cuda == nullptr && (g_torch_cuda = PyImport_ImportModule("torch.cuda")) == nullptr) return false;
        PyObject* cur = PyObject_CallMethodNoArgs(g_torch_cuda, s_current_stream);
        if (cur == nullptr) return false;
        const bool ok = call_long(PyObject_GetAttr(cur, s_cuda_stream), &v);
        Py_DECREF(cur);
        if (!ok) return false;
        PyObject* c = PyImport_ImportModule("torch._C");
        if (c != nullptr && g_raw_stream == nullptr) {
            g_get_device = PyObject_GetAttrString(c, "_cuda_getDevice");
            g_raw_stream = g_get_device ? PyObject_GetAttrString(c, "_cuda_getCurrentRawStream") : nullptr;
        }
        Py_XDECREF(c);
        PyErr_Clear();
        g_cuda_ready = g_get_device != nullptr && g_raw_stream != nullptr;
    }
    *out = reinterpret_cast<void*>((uintptr_t)v);
    return true;
}

// One argument of the C function from the Python argument at the same place.  The last pointer is the stream; a size is that of the
// tensor before it unless it is given.
template <typename T>
bool to_arg(PyObject* const* args, size_t i, size_t n, T* out) {
    PyObject* a = args[i];
    if constexpr (std::is_same_v<T, const qlora_desc*>) {
        const int is = PyObject_IsInstance(a, g_desc_type);
        if (is < 0) return false;
        Py_buffer view;
        if (!is) { PyErr_SetString(PyExc_TypeError, "the layer descriptor must come from desc()"); return false; }
        if (PyObject_GetBuffer(a, &view, PyBUF_SIMPLE) != 0) return false;
        *out = static_cast<const qlora_desc*>(view.buf);          // (the caller holds the object for the whole call)
        PyBuffer_Release(&view);
        return true;
    } else if constexpr (std::is_pointer_v<T>) {
        void* p = nullptr;
        if (!(i + 1 == n ? to_stream(a, &p) : to_pointer(a, &p))) return false;
        *out = static_cast<T>(p);
        return true;
    } else if constexpr (std::is_same_v<T, float>) {
        PyObject* f = PyNumber_Float(a);                              // (what float() takes, as the binding always did)
        if (f == nullptr) return false;
        *out = (float)PyFloat_AS_DOUBLE(f);
        Py_DECREF(f);
        return true;
    } else if constexpr (std::is_same_v<T, size_t>) {
        unsigned long long v = 0, e = 0;
        if (a != Py_None) {
            PyObject* l = PyNumber_Long(a);
            if (!call_long(l, &v)) return false;
        } else if (args[i - 1] != Py_None) {
            if (!method_long(args[i - 1], s_numel, &v) || !method_long(args[i - 1], s_element_size, &e)) return false;
            v *= e;
        }
        *out = (size_t)v;
        return true;
    } else {
        static_assert(std::is_same_v<T, int>);
        unsigned long long v = 0;
        if (PyLong_CheckExact(a)) {
            v = PyLong_AsUnsignedLongLongMask(a);
            if (v == (unsigned long long)-1 && PyErr_Occurred()) return false;
        } else if (!call_long(PyNumber_Long(a), &v)) {
            return false;
        }
        *out = (int)v;
        return true;
    }
}

template <typename... A, size_t... I>
PyObject* call_with(int (*fn)(A...), PyObject* const* args, std::index_sequence<I...>) {
    std::tuple<A...> v{};
    if (!(to_arg(args, I, sizeof...(A), &std::get<I>(v)) && ...)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(std::get<I>(v)...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <typename... A>
PyObject* checked_call(int (*fn)(A...), PyObject* const* args, Py_ssize_t n) {
    if (n != (Py_ssize_t)sizeof...(A)) {
        PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", (int)sizeof...(A), n);
        return nullptr;
    }
    return call_with(fn, args, std::index_sequence_for<A...>{});
}

template <auto Fn>
PyObject* py_call(PyObject*, PyObject* const* args, Py_ssize_t n) { return checked_call(Fn, args, n); }

PyObject* py_set_desc_type(PyObject*, PyObject* type) {
    Py_INCREF(type);
    Py_XSETREF(g_desc_type, type);
    Py_RETURN_NONE;
}

#define QLORA_PY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_call<&name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    QLORA_PY(qlora_fwd), QLORA_PY(qlora_bwd_input), QLORA_PY(qlora_bwd_input_db), QLORA_PY(qlora_bwd_lora),
    QLORA_PY(qlora_fwd_dropout), QLORA_PY(qlora_bwd_input_dropout), QLORA_PY(qlora_bwd_lora_dropout),
    QLORA_PY(qlora_gather_columns), QLORA_PY(qlora_lrec_loss), QLORA_PY(qlora_quantize_rtn),
    {"set_desc_type", py_set_desc_type, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pycall() {
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    s_current_stream = PyUnicode_InternFromString("current_stream");
    if (!s_is_contiguous || !s_data_ptr || !s_cuda_stream || !s_numel || !s_element_size || !s_current_stream) return nullptr;
    pthread_atfork(nullptr, nullptr, in_child);
    return PyModule_Create(&module);
}
