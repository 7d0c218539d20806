// Argument marshalling of the per-layer entry points and of the whole-model runs for Python, as a CPython extension module.
//
// A single layer's kernel runs for 3 - 6 us; the same call through ctypes spends ~2.5 us of host time converting a dozen
// arguments one Python object at a time, about as much as everything below it, and calls issued back to back are then
// bound by it.  The converters here do what binding.py's `_ptr` / `_stream` do (a torch tensor's data_ptr(), a stream's
// cuda_stream, integers, None); anything they do not know -- numpy arrays, keyword arguments -- goes to the Python
// function of the same name that the module was given.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>
#include <string.h>

#include "nnv.h"

namespace {

PyObject* s_data_ptr;
PyObject* s_cuda_stream;
PyObject* s_address;
PyObject* s_n;
PyObject* s_type;
PyObject* g_array;                                            // ctypes.Array and the binding's Choice
PyObject* g_choice;

// One converted argument; ok = false: not a kind that is handled here.
struct Arg {
    uint64_t v;
    bool ok;
};

Arg from_int(PyObject* o) {
    if (!PyLong_CheckExact(o)) return {0, false};
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(o);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) {
        PyErr_Clear();
        return {0, false};
    }
    return {(uint64_t)v, true};
}
Arg from_call(PyObject* r) {                                  // steals r
    if (!r) {
        PyErr_Clear();
        return {0, false};
    }
    const Arg a = from_int(r);
    Py_DECREF(r);
    return a;
}
Arg address(PyObject* o) {
    if (o == Py_None) return {0, true};
    if (PyLong_CheckExact(o)) return from_int(o);
    return from_call(PyObject_CallMethodNoArgs(o, s_data_ptr));
}
Arg stream(PyObject* o) {
    if (o == Py_None) return {0, true};
    if (PyLong_CheckExact(o)) return from_int(o);
    return from_call(PyObject_GetAttr(o, s_cuda_stream));
}
Arg plan(PyObject* o) { return from_call(PyObject_GetAttr(o, s_address)); }

// Address of the choices already laid out by choices_array: a ctypes array of Choice with one entry for each of the plan's layers.
// Nothing else that exports a buffer will do: a numpy array's rows are another layout, for the Python function to convert.
Arg choices(PyObject* o, PyObject* plan) {
    const Arg no{0, false};
    if (!PyType_IsSubtype(Py_TYPE(o), (PyTypeObject*)g_array)) return no;
    PyObject* type = PyObject_GetAttr((PyObject*)Py_TYPE(o), s_type);
    const Arg n = type == g_choice ? from_call(PyObject_GetAttr(plan, s_n)) : no;
    Py_XDECREF(type);
    Py_buffer b;
    if (!n.ok || PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
        PyErr_Clear();
        return no;
    }
    const Arg a{(uint64_t)(uintptr_t)b.buf, (uint64_t)b.len / sizeof(nnv_choice_t) >= n.v};
    PyBuffer_Release(&b);
    return a;
}

PyObject* g_fallback[6];                                      // the Python functions: conv_exec, transform_weights, transform_all, the three runs
PyObject* g_check;                                            // raises for a status that is not OK

PyObject* finish(nnv_status_t st) {
    if (st == NNV_OK) Py_RETURN_NONE;
    PyObject* code = PyLong_FromLong((long)st);
    if (!code) return nullptr;
    PyObject* r = PyObject_CallOneArg(g_check, code);
    Py_DECREF(code);
    return r;
}

// Converts args[0..n) by the letters of `kinds` (p plan, i integer, a address, s stream); an absent last stream is null.
bool convert(const char* kinds, PyObject* const* args, Py_ssize_t n, PyObject* kwnames, uint64_t* v) {
    if (kwnames && PyTuple_GET_SIZE(kwnames) != 0) return false;
    Py_ssize_t i = 0;
    for (; kinds[i]; ++i) {
        if (i >= n) {
            if (kinds[i] == 's' && !kinds[i + 1]) { v[i] = 0; continue; }
            return false;
        }
        const Arg a = kinds[i] == 'p' ? plan(args[i]) : kinds[i] == 'i' ? from_int(args[i]) : kinds[i] == 'a' ? address(args[i]) : stream(args[i]);
        if (!a.ok) return false;
        v[i] = a.v;
    }
    return n <= i;
}

void* P(uint64_t v) { return (void*)(uintptr_t)v; }

// nnv_conv_exec(plan, layer, variant, math, d_in, d_addend, d_wt, d_bias, d_out, d_ws, ws_bytes, stream=None)
PyObject* conv_exec(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    uint64_t v[12];
    if (!convert("piiiaaaaaais", args, n, kw, v)) return PyObject_Vectorcall(g_fallback[0], args, n, kw);
    nnv_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = nnv_conv_exec((nnv_plan_t*)P(v[0]), (int32_t)v[1], (int32_t)v[2], (int32_t)v[3], P(v[4]), P(v[5]), P(v[6]), P(v[7]), P(v[8]),
                       P(v[9]), v[10], P(v[11]));
    Py_END_ALLOW_THREADS
    return finish(st);
}

// nnv_transform_weights(plan, layer, variant, math, d_raw, d_out, stream=None)
PyObject* transform_weights(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    uint64_t v[7];
    if (!convert("piiiaas", args, n, kw, v)) return PyObject_Vectorcall(g_fallback[1], args, n, kw);
    nnv_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = nnv_transform_weights((nnv_plan_t*)P(v[0]), (int32_t)v[1], (int32_t)v[2], (int32_t)v[3], P(v[4]), P(v[5]), P(v[6]));
    Py_END_ALLOW_THREADS
    return finish(st);
}

// nnv_transform_all(plan, choices, d_weights, w_bytes, d_out, out_bytes, stream=None), choices as a ctypes array
PyObject* transform_all(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    uint64_t v[6];
    if (n < 6 || n > 7 || (kw && PyTuple_GET_SIZE(kw) != 0)) return PyObject_Vectorcall(g_fallback[2], args, n, kw);
    const Arg c = choices(args[1], args[0]);
    PyObject* rest[6] = {args[0], args[2], args[3], args[4], args[5], n == 7 ? args[6] : Py_None};
    if (!c.ok || !convert("paiais", rest, 6, nullptr, v)) return PyObject_Vectorcall(g_fallback[2], args, n, kw);
    nnv_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = nnv_transform_all((nnv_plan_t*)P(v[0]), (const nnv_choice_t*)P(c.v), P(v[1]), v[2], P(v[3]), v[4], P(v[5]));
    Py_END_ALLOW_THREADS
    return finish(st);
}

// The whole-model runs: plan, choices as a ctypes array, then `kinds`.  Calls that ask for timings are Python's.
bool convert_run(const char* kinds, PyObject* const* args, Py_ssize_t n, PyObject* kw, const nnv_choice_t** ch, uint64_t* v) {
    const Py_ssize_t m = (Py_ssize_t)strlen(kinds) + 1;
    if (n < m || n > m + 1 || (kw && PyTuple_GET_SIZE(kw) != 0) || (n == m + 1 && args[m] != Py_False)) return false;
    const Arg c = choices(args[1], args[0]);
    PyObject* rest[16];
    rest[0] = args[0];
    for (Py_ssize_t i = 2; i < m; ++i) rest[i - 1] = args[i];
    if (!c.ok || !convert(kinds, rest, m - 1, nullptr, v)) return false;
    *ch = (const nnv_choice_t*)P(c.v);
    return true;
}

// nnv_cold_run(plan, choices, h_weights, w_bytes, h_cached, c_bytes, h_input, h_output, d_arena, arena_bytes, s_copy, s_xform, s_exec, depth)
PyObject* cold_run(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    uint64_t v[13];
    const nnv_choice_t* ch;
    if (!convert_run("paiaiaaaisssi", args, n, kw, &ch, v)) return PyObject_Vectorcall(g_fallback[3], args, n, kw);
    nnv_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = nnv_cold_run((nnv_plan_t*)P(v[0]), ch, P(v[1]), v[2], P(v[3]), v[4], (const float*)P(v[5]), (float*)P(v[6]), P(v[7]), v[8], P(v[9]), P(v[10]),
                      P(v[11]), (int32_t)v[12], nullptr);
    Py_END_ALLOW_THREADS
    return finish(st);
}

// nnv_resident_run(plan, choices, d_weights, w_bytes, d_cached, c_bytes, d_input, d_output, d_arena, arena_bytes, s_xform, s_exec, depth)
PyObject* resident_run(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    uint64_t v[12];
    const nnv_choice_t* ch;
    if (!convert_run("paiaiaaaissi", args, n, kw, &ch, v)) return PyObject_Vectorcall(g_fallback[4], args, n, kw);
    nnv_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = nnv_resident_run((nnv_plan_t*)P(v[0]), ch, P(v[1]), v[2], P(v[3]), v[4], (const float*)P(v[5]), (float*)P(v[6]), P(v[7]), v[8], P(v[9]),
                          P(v[10]), (int32_t)v[11], nullptr);
    Py_END_ALLOW_THREADS
    return finish(st);
}

// nnv_warm_run(plan, warm, d_warm, warm_bytes, w_bytes, h_input, h_output, d_arena, arena_bytes, s_xform, s_exec)
PyObject* warm_run(PyObject*, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    uint64_t v[10];
    const nnv_choice_t* ch;
    if (!convert_run("paiiaaaiss", args, n, kw, &ch, v)) return PyObject_Vectorcall(g_fallback[5], args, n, kw);
    nnv_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = nnv_warm_run((nnv_plan_t*)P(v[0]), ch, P(v[1]), v[2], v[3], (const float*)P(v[4]), (float*)P(v[5]), P(v[6]), v[7], P(v[8]), P(v[9]), nullptr);
    Py_END_ALLOW_THREADS
    return finish(st);
}

PyObject* set_fallbacks(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != 9) {
        PyErr_SetString(PyExc_TypeError, "seven functions and two classes expected");
        return nullptr;
    }
    for (int i = 0; i < 6; ++i) Py_XSETREF(g_fallback[i], Py_NewRef(args[i]));
    Py_XSETREF(g_check, Py_NewRef(args[6]));
    Py_XSETREF(g_array, Py_NewRef(args[7]));
    Py_XSETREF(g_choice, Py_NewRef(args[8]));
    Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"nnv_conv_exec", (PyCFunction)(void (*)(void))conv_exec, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"nnv_transform_weights", (PyCFunction)(void (*)(void))transform_weights, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"nnv_transform_all", (PyCFunction)(void (*)(void))transform_all, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"nnv_cold_run", (PyCFunction)(void (*)(void))cold_run, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"nnv_resident_run", (PyCFunction)(void (*)(void))resident_run, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"nnv_warm_run", (PyCFunction)(void (*)(void))warm_run, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"set_fallbacks", (PyCFunction)(void (*)(void))set_fallbacks, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_nnvcall", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__nnvcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_address = PyUnicode_InternFromString("address");
    s_n = PyUnicode_InternFromString("n");
    s_type = PyUnicode_InternFromString("_type_");
    return PyModule_Create(&g_module);
}
