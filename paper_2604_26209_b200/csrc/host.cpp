// The Python side of the per-step calls: tensors, integers and the current stream handed to the C ABI of libhpd.
//
// A decode step of few prompts keeps the GPU busy for 20 to 40 us; marshalling its three calls (some fifty tensors) through
// ctypes objects took longer than that.  Every entry point here takes (geometry, arguments of the C function in order
// without the stream): tensors become device pointers (device-resident contiguous ones only), None a null pointer; the current
// stream is appended.  The functions' addresses come from the library that binding.load() has opened.
#include <Python.h>

#include <cstring>
#include <tuple>
#include <utility>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/hpd.h"

namespace {

bool read_geom(PyObject* o, hpd_geom& g)
{
    static PyObject* names[6];
    static const char* const text[6] = {"Hq", "Hkv", "D", "suffix_cap", "rope_theta", "sm_scale"};
    int32_t* const ints[4] = {&g.Hq, &g.Hkv, &g.D, &g.suffix_cap};
    float* const reals[2] = {&g.rope_theta, &g.sm_scale};
    for (int i = 0; i < 6; ++i) {
        if (!names[i] && !(names[i] = PyUnicode_InternFromString(text[i]))) return false;
        PyObject* v = PyObject_GetAttr(o, names[i]);
        if (!v) return false;
        PyObject* n = i < 4 ? PyNumber_Long(v) : PyNumber_Float(v);
        Py_DECREF(v);
        if (!n) return false;
        if (i < 4) *ints[i] = static_cast<int32_t>(PyLong_AsUnsignedLongLongMask(n));
        else *reals[i - 4] = static_cast<float>(PyFloat_AS_DOUBLE(n));
        Py_DECREF(n);
        if (PyErr_Occurred()) return false;
    }
    return true;
}

template <typename T> bool convert(PyObject* o, T& out)
{
    if constexpr (std::is_pointer_v<T>) {
        if (o == Py_None) { out = nullptr; return true; }
        if (!THPVariable_Check(o)) {
            PyErr_SetString(PyExc_TypeError, "a tensor or None is expected");
            return false;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device-resident contiguous tensors only");
            return false;
        }
        out = static_cast<T>(t.data_ptr());
        return true;
    } else {
        PyObject* n = PyNumber_Index(o);                             // integers and what stands for one (NumPy's, 0-d tensors); no floats
        if (!n) return false;
        out = static_cast<T>(PyLong_AsUnsignedLongLongMask(n));      // as ctypes does
        Py_DECREF(n);
        return !PyErr_Occurred();
    }
}

template <typename... A, size_t... I>
PyObject* invoke_with(int (*f)(const hpd_geom*, A...), PyObject* const* args, std::index_sequence<I...>)
{
    std::tuple<A...> v;
    hpd_geom g;
    if (!read_geom(args[0], g) || !(convert(args[1 + I], std::get<I>(v)) && ...)) return nullptr;
    std::get<sizeof...(A) - 1>(v) = c10::cuda::getCurrentCUDAStream().stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = std::apply([&](auto... a) { return f(&g, a...); }, v);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <typename... A>
PyObject* invoke(int (*f)(const hpd_geom*, A...), PyObject* const* args, Py_ssize_t n)
{
    if (!f) {
        PyErr_SetString(PyExc_RuntimeError, "the library has not been loaded");
        return nullptr;
    }
    if (n != static_cast<Py_ssize_t>(sizeof...(A))) {                // the geometry in the place of the stream
        PyErr_Format(PyExc_TypeError, "%zd arguments given, %zd expected", n, static_cast<Py_ssize_t>(sizeof...(A)));
        return nullptr;
    }
    try {
        return invoke_with(f, args, std::make_index_sequence<sizeof...(A) - 1>());
    } catch (const std::exception& e) {                              // a tensor without storage, no device
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define HPD_ENTRIES(X)                                                                                              \
    X(hpd_build_meta) X(hpd_build_meta_skeleton) X(hpd_rope) X(hpd_kv_append) X(hpd_rope_append) X(hpd_attn_decode)  \
    X(hpd_attn_decode_posorder) X(hpd_attn_decode_shared) X(hpd_advance) X(hpd_merge_lse) X(hpd_prefill_meta)        \
    X(hpd_prefill_attn)

#define X(name)                                                                                                     \
    decltype(&::name) at_##name = nullptr;                                                                          \
    PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n) { return invoke(at_##name, args, n); }
HPD_ENTRIES(X)
#undef X

PyObject* set_address(PyObject*, PyObject* args)
{
    const char* name;
    unsigned long long address;
    if (!PyArg_ParseTuple(args, "sK", &name, &address)) return nullptr;
#define X(entry) if (!strcmp(name, #entry)) { at_##entry = reinterpret_cast<decltype(at_##entry)>(address); Py_RETURN_NONE; }
    HPD_ENTRIES(X)
#undef X
    PyErr_Format(PyExc_KeyError, "%s", name);
    return nullptr;
}

PyMethodDef methods[] = {
#define X(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr},
    HPD_ENTRIES(X)
#undef X
    {"set_address", set_address, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host(void)
{
    PyObject* m = PyModule_Create(&module);
    if (!m) return nullptr;
    PyObject* names = PyTuple_New(0);
#define X(name) if (names) { PyObject* s = PyUnicode_FromString(#name); Py_ssize_t n = PyTuple_GET_SIZE(names); _PyTuple_Resize(&names, n + 1); if (names) PyTuple_SET_ITEM(names, n, s); }
    HPD_ENTRIES(X)
#undef X
    if (!names || PyModule_AddObject(m, "ENTRIES", names) < 0) return nullptr;
    if (PyModule_AddStringConstant(m, "BUILT_FOR", HPD_BUILT_FOR) < 0) return nullptr;
    return m;
}
