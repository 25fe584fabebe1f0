// CPython module `_native`: the device calls of the binding, with the arguments turned into C ones natively.
//
// A decode GEMV of a small layer runs for 3 to 4 us, and the same call through ctypes took 9 to 11 us of host time to issue:
// every tensor was asked three questions from Python, a stream object was made, twelve ctypes values were built.  Here the
// questions are field reads through torch's C++ interface.  One table describes the calls; a call is checked and
// converted in one pass over its arguments and made without the GIL, as ctypes made it.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <string.h>

#include <string>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/tilefuse.h"

namespace {

struct Arg {
    void* ptr;        // device address of a tensor (nullptr for None), or ...
    size_t bytes;     // ... with its size ...
    int value;        // ... or an integer
};

constexpr int kMaxArgs = 12;
struct Call {
    const char* name;
    int count;                                   // arguments before `stream`
    const char* kinds;                           // per argument: t = tensor, i = integer
    const char* names[kMaxArgs];
    tf_status (*make)(const Arg*, void* stream);
};

#define TF_LINEAR(fn)                                                                                                     \
    {#fn, 7, "tttiiit", {"packed", "a", "y", "M", "K", "N", "workspace"}, [](const Arg* x, void* s) {                     \
         return fn(x[0].ptr, x[1].ptr, x[2].ptr, x[3].value, x[4].value, x[5].value, x[6].ptr, x[6].bytes, s); }}
#define TF_GROUPED(fn)                                                                                                    \
    {#fn, 8, "tttiiiit", {"packed", "a", "y", "M", "K", "N", "group_size", "workspace"}, [](const Arg* x, void* s) {      \
         return fn(x[0].ptr, x[1].ptr, x[2].ptr, x[3].value, x[4].value, x[5].value, x[6].value, x[7].ptr, x[7].bytes, s); }}
#define TF_RAW(fn)                                                                                                        \
    {#fn, 10, "tttttiiiit", {"qweight", "scales_f16", "qzeros", "a", "y", "M", "K", "N", "group_size", "workspace"},      \
     [](const Arg* x, void* s) {                                                                                          \
         return fn(static_cast<const uint32_t*>(x[0].ptr), static_cast<const uint16_t*>(x[1].ptr),                        \
                   static_cast<const uint32_t*>(x[2].ptr), x[3].ptr, x[4].ptr, x[5].value, x[6].value, x[7].value,        \
                   x[8].value, x[9].ptr, x[9].bytes, s); }}

const Call kCalls[] = {
    TF_LINEAR(tf_gemv_w4a16), TF_LINEAR(tf_gemv_w8a16), TF_LINEAR(tf_gemm_w4a16), TF_LINEAR(tf_gemm_w8a16),
    TF_GROUPED(tf_gemv_w4a16_grouped), TF_GROUPED(tf_gemm_w4a16_grouped),
    TF_RAW(tf_gemv_awq_raw), TF_RAW(tf_gemm_awq_raw),
    {"tf_gemv_w4a16_static", 6, "tttiii", {"packed", "a", "y", "M", "K", "N"}, [](const Arg* x, void* s) {
         return tf_gemv_w4a16_static(x[0].ptr, x[1].ptr, x[2].ptr, x[3].value, x[4].value, x[5].value, s); }},
    {"tf_pack_awq_device", 7, "tttiiit", {"qweight", "scales_f16", "qzeros", "K", "N", "group_size", "out"},
     [](const Arg* x, void* s) {
         return tf_pack_awq_device(static_cast<const uint32_t*>(x[0].ptr), static_cast<const uint16_t*>(x[1].ptr),
                                   static_cast<const uint32_t*>(x[2].ptr), x[3].value, x[4].value, x[5].value, x[6].ptr,
                                   x[6].bytes, s); }},
};
constexpr int kNumCalls = sizeof(kCalls) / sizeof(kCalls[0]);

PyObject* g_raise = nullptr;                     // raise(name, status): the binding's exception for a status that is not TF_OK

bool convert_tensor(PyObject* o, Arg* out) {
    out->ptr = nullptr;
    out->bytes = 0;
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_AttributeError, "device buffers must be CUDA tensors, not '%.100s'", Py_TYPE(o)->tp_name);
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "device buffers must be contiguous CUDA tensors");
        return false;
    }
    out->ptr = t.data_ptr();
    out->bytes = t.nbytes();
    return true;
}

bool convert_int(PyObject* o, Arg* out) {
    PyObject* i = PyLong_CheckExact(o) ? Py_NewRef(o) : PyNumber_Index(o);
    if (i == nullptr) return false;
    out->value = static_cast<int>(PyLong_AsUnsignedLongMask(i));
    Py_DECREF(i);
    return !PyErr_Occurred();
}

bool convert_stream(PyObject* o, void** out) {
    if (o == nullptr || o == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (h == nullptr) return false;
    *out = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

// `self` is the call's number.
PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
    const Call& c = kCalls[PyLong_AsLong(self)];
    PyObject* given[kMaxArgs + 1] = {};          // the arguments, then `stream`
    if (nargs > c.count + 1) return PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", c.name, c.count + 1, nargs);
    for (Py_ssize_t i = 0; i < nargs; ++i) given[i] = args[i];
    const Py_ssize_t nkw = kwnames != nullptr ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
        const char* name = PyUnicode_AsUTF8(PyTuple_GET_ITEM(kwnames, k));
        if (name == nullptr) return nullptr;
        int at = 0;
        while (at < c.count && strcmp(name, c.names[at]) != 0) ++at;
        if (at == c.count && strcmp(name, "stream") != 0) return PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%s'", c.name, name);
        if (given[at] != nullptr) return PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", c.name, name);
        given[at] = args[nargs + k];
    }
    Arg x[kMaxArgs];
    void* stream = nullptr;
    try {
        for (int i = 0; i < c.count; ++i) {
            if (given[i] == nullptr) return PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", c.name, c.names[i]);
            if (!(c.kinds[i] == 't' ? convert_tensor(given[i], &x[i]) : convert_int(given[i], &x[i]))) return nullptr;
        }
        if (!convert_stream(given[c.count], &stream)) return nullptr;
    } catch (const std::exception& e) {          // torch: a tensor without memory of its own (under vmap), no device to ask for a stream
        return PyErr_Format(PyExc_RuntimeError, "%s(): %.500s", c.name, e.what());
    }
    PyThreadState* released = PyEval_SaveThread();
    const tf_status status = c.make(x, stream);  // C calls, which do not throw
    PyEval_RestoreThread(released);
    if (status != TF_OK) {
        PyObject* r = PyObject_CallFunction(g_raise, "si", c.name, static_cast<int>(status));
        Py_XDECREF(r);
        if (!PyErr_Occurred()) PyErr_Format(PyExc_RuntimeError, "%s -> %d", c.name, static_cast<int>(status));
        return nullptr;
    }
    Py_RETURN_NONE;
}

PyMethodDef g_defs[kNumCalls];
std::string g_docs[kNumCalls];                   // "name(arguments, stream=None)\n--\n\n...", which gives the function its signature
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, nullptr, nullptr, nullptr, nullptr, nullptr};

// calls(raise): {name: function} of every call of the table.
PyObject* calls(PyObject* module, PyObject* raise) {
    Py_XSETREF(g_raise, Py_NewRef(raise));
    PyObject* out = PyDict_New();
    for (int i = 0; out != nullptr && i < kNumCalls; ++i) {
        g_docs[i] = std::string(kCalls[i].name) + "(";
        for (int k = 0; k < kCalls[i].count; ++k) g_docs[i] += std::string(kCalls[i].names[k]) + ", ";
        g_docs[i] += "stream=None)\n--\n\nCUDA tensors and sizes as for the C call of this name; asynchronous on the stream.";
        g_defs[i] = {kCalls[i].name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(call)), METH_FASTCALL | METH_KEYWORDS, g_docs[i].c_str()};
        PyObject* index = PyLong_FromLong(i);
        PyObject* f = index != nullptr ? PyCFunction_NewEx(&g_defs[i], index, nullptr) : nullptr;
        if (f == nullptr || PyDict_SetItemString(out, kCalls[i].name, f) != 0) Py_CLEAR(out);
        Py_XDECREF(f);
        Py_XDECREF(index);
    }
    return out;
}

PyMethodDef g_calls_def = {"calls", calls, METH_O, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    PyObject* m = PyModule_Create(&g_module);
    if (m == nullptr) return nullptr;
    // the torch and the Python this file was compiled against; the build looks for it in the module before it is loaded
    if (PyModule_AddStringConstant(m, "TARGET", TF_NATIVE_TARGET) != 0) {
        Py_DECREF(m);
        return nullptr;
    }
    PyObject* f = PyCFunction_NewEx(&g_calls_def, nullptr, nullptr);
    if (f == nullptr || PyModule_AddObject(m, "calls", f) != 0) {
        Py_XDECREF(f);
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
