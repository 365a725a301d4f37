// Python side of the C ABI: each entry point as a function of positional arguments.  They convert as through ctypes: a whole number is
// an int or an object with __index__ (anything else is ctypes.ArgumentError), a float is what float() takes; a pointer is None, an
// address, or an object with data_ptr() (a torch tensor).  The GIL is released during the call.
//
// Why not ctypes: a step of the smallest layer is three calls whose kernels take 12 us together, and the host needed 30 us to
// issue them - 2 us and more a call to convert 9 to 22 arguments and 3 us for torch.cuda.current_stream().  With this module
// and the raw stream handle it needs 10 us, and the GPU is never idle between calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "../../include/sbp.h"

namespace {

PyObject* g_data_ptr = nullptr;            // the interned name "data_ptr"
PyObject* g_argument_error = nullptr;      // ctypes.ArgumentError

bool to_integer(PyObject* o, unsigned long long& v) {
    v = PyLong_AsUnsignedLongLongMask(o);
    if (v != (unsigned long long)-1 || !PyErr_Occurred()) return true;
    PyErr_Format(g_argument_error, "'%s' object cannot be interpreted as an integer", Py_TYPE(o)->tp_name);
    return false;
}

bool to_address(PyObject* o, unsigned long long& v) {
    if (o == Py_None) {
        v = 0;
        return true;
    }
    if (PyLong_Check(o)) return to_integer(o, v);
    PyObject* p = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (p == nullptr) return false;
    const bool ok = to_integer(p, v);
    Py_DECREF(p);
    return ok;
}

bool to_float(PyObject* o, double& v) {
    PyObject* f = PyNumber_Float(o);
    if (f == nullptr) return false;
    v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return true;
}

template <typename T>
bool convert(PyObject* o, T& out) {
    if constexpr (std::is_floating_point_v<T>) {
        double v = 0.0;
        if (!to_float(o, v)) return false;
        out = v;
        return true;
    } else {
        unsigned long long v = 0;
        if constexpr (std::is_pointer_v<T>) {
            if (!to_address(o, v)) return false;
            out = reinterpret_cast<T>(static_cast<uintptr_t>(v));
        } else {
            if (!to_integer(o, v)) return false;
            out = static_cast<T>(v);
        }
        return true;
    }
}

template <auto F>
struct Call;
template <typename R, typename... A, R (*F)(A...)>
struct Call<F> {
    template <size_t... I>
    static bool convert_all(PyObject* const* args, std::tuple<A...>& t, std::index_sequence<I...>) {
        return (convert(args[I], std::get<I>(t)) && ...);
    }
    static PyObject* run(PyObject*, PyObject* const* args, Py_ssize_t n) {
        if (n != (Py_ssize_t)sizeof...(A)) {
            PyErr_Format(PyExc_TypeError, "%zd arguments where %zd are expected", n, (Py_ssize_t)sizeof...(A));
            return nullptr;
        }
        std::tuple<A...> t;
        if (!convert_all(args, t, std::index_sequence_for<A...>())) return nullptr;
        long r;
        Py_BEGIN_ALLOW_THREADS
        r = (long)std::apply(F, t);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(r);
    }
};

#define SBP_CALL(name) {#name, (PyCFunction)(void (*)(void))Call<&name>::run, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    SBP_CALL(sbp_sample_keep),
    SBP_CALL(sbp_forward_cache),
    SBP_CALL(sbp_linear_forward),
    SBP_CALL(sbp_linear_backward),
    SBP_CALL(sbp_attention_backward),
    SBP_CALL(sbp_act_backward),
    SBP_CALL(sbp_patch_cache),
    SBP_CALL(sbp_patch_scatter),
    SBP_CALL(sbp_step_host),
    SBP_CALL(sbp_bias_grad_static),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    PyObject* ctypes = PyImport_ImportModule("ctypes");
    if (g_data_ptr == nullptr || ctypes == nullptr) return nullptr;
    g_argument_error = PyObject_GetAttrString(ctypes, "ArgumentError");
    Py_DECREF(ctypes);
    return g_argument_error == nullptr ? nullptr : PyModule_Create(&g_module);
}
