// The calls of the Python layer that a decode loop makes hundreds of times per token, as a CPython extension: reads
// pointers and sizes of the tensors it is given and calls the C ABI.  Argument marshalling only, like binding.py.
//
// Why native: with few tokens a loop is bound by what the host does per call.  Through ctypes a GEMM call took 10.8 us
// (3.3 of them torch.cuda.current_stream(), 1.4 ctypes' own conversions, 3 Python), of which the launch itself is
// 2.5; the kernels behind it take 4 to 10.  The functions are those of the libsbn.so that binding.py has loaded
// (bind() takes their addresses), so there is one library and one state.  The GIL is released around each call, as ctypes does.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "sbn.h"

namespace {

decltype(&sbn_quant_act) f_quant_act;
decltype(&sbn_quant_act_expand68) f_quant_act_expand68;
decltype(&sbn_norm_quant_act) f_norm_quant_act;
decltype(&sbn_norm_quant_act_expand68) f_norm_quant_act_expand68;
decltype(&sbn_sparse_bitlinear) f_sparse_bitlinear;
decltype(&sbn_bitlinear) f_bitlinear;
decltype(&sbn_sparse_bitlinear_packed) f_sparse_bitlinear_packed;
decltype(&sbn_quant_act_sparse_bitlinear) f_quant_act_sparse_bitlinear;
decltype(&sbn_quant_act_bitlinear) f_quant_act_bitlinear;

PyObject *s_data_ptr, *s_shape, *s_dtype, *s_numel, *s_element_size;      // interned names
PyObject *g_bfloat16, *g_get_device, *g_get_raw_stream;                   // torch.bfloat16, torch's current device / stream

// All conversions leave a Python error behind on failure and do nothing once there is one; run() looks before it calls
// the library.
void* ptr(PyObject* t) {
    if (t == Py_None || PyErr_Occurred()) return nullptr;
    PyObject* v = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!v) return nullptr;
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return p;
}

void shape2(PyObject* t, int& rows, int& cols) {
    rows = cols = 0;
    if (PyErr_Occurred()) return;
    PyObject* s = PyObject_GetAttr(t, s_shape);
    if (!s) return;
    if (!PyTuple_Check(s) || PyTuple_GET_SIZE(s) != 2) {
        PyErr_SetString(PyExc_ValueError, "expected a two-dimensional tensor");
    } else {
        rows = static_cast<int>(PyLong_AsLong(PyTuple_GET_ITEM(s, 0)));
        cols = static_cast<int>(PyLong_AsLong(PyTuple_GET_ITEM(s, 1)));
    }
    Py_DECREF(s);
}

long long call_ll(PyObject* t, PyObject* method) {
    if (PyErr_Occurred()) return 0;
    PyObject* v = PyObject_CallMethodNoArgs(t, method);
    if (!v) return 0;
    const long long n = PyLong_AsLongLong(v);
    Py_DECREF(v);
    return n;
}

// columns of the weight matrix: `per_element` of them in every element of t, over `rows` rows
int columns(PyObject* t, int per_element, int rows) {
    const long long n = call_ll(t, s_numel);
    if (PyErr_Occurred()) return 0;
    if (rows == 0) {
        PyErr_SetString(PyExc_ZeroDivisionError, "no output features");
        return 0;
    }
    return static_cast<int>(per_element * n / rows);
}

sbn_out_dtype out_dtype(PyObject* y) {
    if (PyErr_Occurred()) return SBN_OUT_F32;
    PyObject* d = PyObject_GetAttr(y, s_dtype);
    Py_XDECREF(d);                                        // torch keeps its dtype objects alive
    return d == g_bfloat16 ? SBN_OUT_BF16 : SBN_OUT_F32;
}

size_t bytes_of(PyObject* ws) {
    if (ws == Py_None) return 0;
    const long long n = call_ll(ws, s_numel);
    return static_cast<size_t>(n * call_ll(ws, s_element_size));
}

void* current_stream() {
    if (PyErr_Occurred()) return nullptr;
    PyObject* dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return nullptr;
    PyObject* s = PyObject_CallOneArg(g_get_raw_stream, dev);
    Py_DECREF(dev);
    if (!s) return nullptr;
    void* p = PyLong_AsVoidPtr(s);
    Py_DECREF(s);
    return p;
}

template <typename Fn>
PyObject* run(Fn fn) {
    if (PyErr_Occurred()) return nullptr;
    sbn_status st;
    Py_BEGIN_ALLOW_THREADS
    st = fn();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

bool expect(Py_ssize_t n, Py_ssize_t want) {
    if (n == want && f_quant_act) return true;
    PyErr_SetString(PyExc_TypeError, n != want ? "wrong number of arguments" : "bind() has not been called");
    return false;
}

// (x, xq, a_scale, expand68)
PyObject* py_quant_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 4)) return nullptr;
    int T, K;
    shape2(a[0], T, K);
    const void* x = ptr(a[0]);
    int8_t* xq = static_cast<int8_t*>(ptr(a[1]));
    float* sc = static_cast<float*>(ptr(a[2]));
    const auto f = a[3] == Py_True ? f_quant_act_expand68 : f_quant_act;
    void* s = current_stream();
    return run([=] { return f(x, T, K, xq, sc, s); });
}

// (x, xq, a_scale, gain, eps, expand68)
PyObject* py_norm_quant_act(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 6)) return nullptr;
    int T, K;
    shape2(a[0], T, K);
    const void* x = ptr(a[0]);
    int8_t* xq = static_cast<int8_t*>(ptr(a[1]));
    float* sc = static_cast<float*>(ptr(a[2]));
    const float* gain = static_cast<const float*>(ptr(a[3]));
    const float eps = PyErr_Occurred() ? 0.0f : static_cast<float>(PyFloat_AsDouble(a[4]));
    const int expand = PyErr_Occurred() ? 0 : PyObject_IsTrue(a[5]);
    const auto f = expand ? f_norm_quant_act_expand68 : f_norm_quant_act;
    void* s = current_stream();
    return run([=] { return f(x, T, K, gain, eps, xq, sc, s); });
}

// (xq, a_scale, vals, meta, w_scale, y, bias, acc_out, ws)
PyObject* py_sparse_bitlinear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 9)) return nullptr;
    int T, N;
    shape2(a[5], T, N);
    const int K = columns(a[2], 2, N);
    const int8_t* xq = static_cast<const int8_t*>(ptr(a[0]));
    const float* sc = static_cast<const float*>(ptr(a[1]));
    const int8_t* vals = static_cast<const int8_t*>(ptr(a[2]));
    const uint8_t* meta = static_cast<const uint8_t*>(ptr(a[3]));
    const float* w = static_cast<const float*>(ptr(a[4]));
    void* y = ptr(a[5]);
    const sbn_out_dtype dt = out_dtype(a[5]);
    const float* bias = static_cast<const float*>(ptr(a[6]));
    int32_t* acc = static_cast<int32_t*>(ptr(a[7]));
    void* ws = ptr(a[8]);
    const size_t wb = bytes_of(a[8]);
    void* s = current_stream();
    return run([=] { return f_sparse_bitlinear(xq, sc, T, vals, meta, w, N, K, bias, y, dt, acc, ws, wb, s); });
}

// (xq, a_scale, dense_q, w_scale, y, bias, acc_out, ws)
PyObject* py_bitlinear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 8)) return nullptr;
    int T, N;
    shape2(a[4], T, N);
    const int K = columns(a[2], 1, N);
    const int8_t* xq = static_cast<const int8_t*>(ptr(a[0]));
    const float* sc = static_cast<const float*>(ptr(a[1]));
    const int8_t* q = static_cast<const int8_t*>(ptr(a[2]));
    const float* w = static_cast<const float*>(ptr(a[3]));
    void* y = ptr(a[4]);
    const sbn_out_dtype dt = out_dtype(a[4]);
    const float* bias = static_cast<const float*>(ptr(a[5]));
    int32_t* acc = static_cast<int32_t*>(ptr(a[6]));
    void* ws = ptr(a[7]);
    const size_t wb = bytes_of(a[7]);
    void* s = current_stream();
    return run([=] { return f_bitlinear(xq, sc, T, q, w, N, K, bias, y, dt, acc, ws, wb, s); });
}

// (xq, a_scale, vals2, meta, w_scale, y, bias, acc_out)
PyObject* py_sparse_bitlinear_packed(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 8)) return nullptr;
    int T, N;
    shape2(a[5], T, N);
    const int K = columns(a[2], 8, N);
    const int8_t* xq = static_cast<const int8_t*>(ptr(a[0]));
    const float* sc = static_cast<const float*>(ptr(a[1]));
    const uint8_t* vals2 = static_cast<const uint8_t*>(ptr(a[2]));
    const uint8_t* meta = static_cast<const uint8_t*>(ptr(a[3]));
    const float* w = static_cast<const float*>(ptr(a[4]));
    void* y = ptr(a[5]);
    const sbn_out_dtype dt = out_dtype(a[5]);
    const float* bias = static_cast<const float*>(ptr(a[6]));
    int32_t* acc = static_cast<int32_t*>(ptr(a[7]));
    void* s = current_stream();
    return run([=] { return f_sparse_bitlinear_packed(xq, sc, T, vals2, meta, w, N, K, bias, y, dt, acc, s); });
}

// (x, vals, meta, w_scale, y, bias, acc_out, a_scale_out)
PyObject* py_quant_act_sparse_bitlinear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 8)) return nullptr;
    int T, K, T_y, N;
    shape2(a[0], T, K);
    shape2(a[4], T_y, N);
    const void* x = ptr(a[0]);
    const int8_t* vals = static_cast<const int8_t*>(ptr(a[1]));
    const uint8_t* meta = static_cast<const uint8_t*>(ptr(a[2]));
    const float* w = static_cast<const float*>(ptr(a[3]));
    void* y = ptr(a[4]);
    const sbn_out_dtype dt = out_dtype(a[4]);
    const float* bias = static_cast<const float*>(ptr(a[5]));
    int32_t* acc = static_cast<int32_t*>(ptr(a[6]));
    float* sc = static_cast<float*>(ptr(a[7]));
    void* s = current_stream();
    return run([=] { return f_quant_act_sparse_bitlinear(x, T, vals, meta, w, N, K, bias, y, dt, acc, sc, s); });
}

// (x, dense_q, w_scale, y, bias, acc_out, a_scale_out)
PyObject* py_quant_act_bitlinear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!expect(n, 7)) return nullptr;
    int T, K, T_y, N;
    shape2(a[0], T, K);
    shape2(a[3], T_y, N);
    const void* x = ptr(a[0]);
    const int8_t* q = static_cast<const int8_t*>(ptr(a[1]));
    const float* w = static_cast<const float*>(ptr(a[2]));
    void* y = ptr(a[3]);
    const sbn_out_dtype dt = out_dtype(a[3]);
    const float* bias = static_cast<const float*>(ptr(a[4]));
    int32_t* acc = static_cast<int32_t*>(ptr(a[5]));
    float* sc = static_cast<float*>(ptr(a[6]));
    void* s = current_stream();
    return run([=] { return f_quant_act_bitlinear(x, T, q, w, N, K, bias, y, dt, acc, sc, s); });
}

// bind(addresses: dict name -> int, torch.bfloat16, get_device, get_raw_stream)
template <typename F>
bool take(PyObject* addresses, const char* name, F& f) {
    PyObject* v = PyDict_GetItemString(addresses, name);                  // borrowed
    if (!v) {
        PyErr_SetString(PyExc_KeyError, name);
        return false;
    }
    f = reinterpret_cast<F>(PyLong_AsVoidPtr(v));
    return !PyErr_Occurred();
}
void keep(PyObject*& slot, PyObject* v) {
    Py_INCREF(v);
    Py_XSETREF(slot, v);
}
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 4 || !PyDict_Check(a[0])) {
        PyErr_SetString(PyExc_TypeError, "bind(addresses, bfloat16, get_device, get_raw_stream)");
        return nullptr;
    }
    PyObject* d = a[0];
    if (!take(d, "sbn_quant_act_expand68", f_quant_act_expand68) || !take(d, "sbn_norm_quant_act", f_norm_quant_act) ||
        !take(d, "sbn_norm_quant_act_expand68", f_norm_quant_act_expand68) || !take(d, "sbn_sparse_bitlinear", f_sparse_bitlinear) ||
        !take(d, "sbn_bitlinear", f_bitlinear) || !take(d, "sbn_sparse_bitlinear_packed", f_sparse_bitlinear_packed) ||
        !take(d, "sbn_quant_act_sparse_bitlinear", f_quant_act_sparse_bitlinear) ||
        !take(d, "sbn_quant_act_bitlinear", f_quant_act_bitlinear))
        return nullptr;
    keep(g_bfloat16, a[1]);
    keep(g_get_device, a[2]);
    keep(g_get_raw_stream, a[3]);
    if (!take(d, "sbn_quant_act", f_quant_act)) return nullptr;           // last: its presence means bound
    Py_RETURN_NONE;
}

#define SBN_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_##name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    SBN_METHOD(bind), SBN_METHOD(quant_act), SBN_METHOD(norm_quant_act), SBN_METHOD(sparse_bitlinear), SBN_METHOD(bitlinear),
    SBN_METHOD(sparse_bitlinear_packed), SBN_METHOD(quant_act_sparse_bitlinear), SBN_METHOD(quant_act_bitlinear),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_sbn_native", "Tensor arguments to the C ABI of libsbn.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sbn_native(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    if (!s_data_ptr || !s_shape || !s_dtype || !s_numel || !s_element_size) return nullptr;
    return PyModule_Create(&module_def);
}
