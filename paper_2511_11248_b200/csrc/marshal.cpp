// Argument marshalling of the hot entry points for Python, against the CPython C API.
//
// A decode call runs for 4 us on the GPU; issuing it through ctypes cost more than that on the host (a ctypes call
// of twelve arguments alone about 1.5 - 2.5 us, as much again for the Python that reads addresses and sizes).  Here
// one vectorcall reads the tensors' addresses and sizes and calls the C ABI.  The module holds no library of its
// own: binding.py hands it the addresses of the entry points it loaded (`bind`), so that whichever build
// TMAN_LIBRARY selects is the one that runs.  Every function takes the arguments of the Python wrapper of the same
// name with the stream as an integer last, and returns the tman_status.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include "tman.h"

namespace {

enum { F_GEMV, F_GROUPED, F_GEMM, F_QUANT, F_QUANT_I8, F_TERNARY, F_TERNARY_I8, F_PACK, F_COUNT };
void *g_fn[F_COUNT];
PyObject *g_data_ptr, *g_nbytes, *g_numel, *g_element_size;                // interned attribute names

// Address of a tensor (None: 0).  False with a Python error set when the object has none.
bool address(PyObject *t, void **out)
{
    if (t == Py_None) { *out = nullptr; return true; }
    PyObject *r = PyObject_CallMethodNoArgs(t, g_data_ptr);
    if (r && !PyLong_Check(r)) {                // another integer type, say of NumPy
        PyObject *n = PyNumber_Long(r);
        Py_DECREF(r);
        r = n;
    }
    if (!r) return false;
    *out = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return !PyErr_Occurred();
}
// Size of a tensor, or of any object with the numel() and element_size() of one.
bool bytes_of(PyObject *t, size_t *out)
{
    PyObject *r = PyObject_GetAttr(t, g_nbytes);
    if (!r) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
        PyErr_Clear();
        PyObject *n = PyObject_CallMethodNoArgs(t, g_numel), *e = n ? PyObject_CallMethodNoArgs(t, g_element_size) : nullptr;
        r = e ? PyNumber_Multiply(n, e) : nullptr;
        Py_XDECREF(n);
        Py_XDECREF(e);
        if (!r) return false;
    }
    *out = PyLong_AsSize_t(r);
    Py_DECREF(r);
    return !PyErr_Occurred();
}
bool integer(PyObject *o, int *out)
{
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    if (v == (unsigned long)-1 && PyErr_Occurred()) return false;
    *out = (int)(unsigned)v;                    // like ctypes' c_int: the low 32 bits
    return true;
}
// The same of whatever int() takes (an entry of N_list: a float, an element of an array or a tensor)
bool integer_of(PyObject *o, int *out)
{
    if (PyLong_Check(o)) return integer(o, out);
    PyObject *n = PyNumber_Long(o);
    const bool ok = n && integer(n, out);
    Py_XDECREF(n);
    return ok;
}
// Whatever float() takes
bool real_of(PyObject *o, double *out)
{
    PyObject *f = PyNumber_Float(o);
    if (!f) return false;
    *out = PyFloat_AsDouble(f);
    Py_DECREF(f);
    return !PyErr_Occurred();
}

// Reads arguments left to right; the first failure sticks.
struct Reader {
    PyObject *const *a;
    bool ok = true;
    explicit Reader(PyObject *const *args) : a(args) {}
    void *ptr() { void *p = nullptr; ok = ok && address(*a++, &p); return p; }
    void *buf(size_t *n) { void *p = nullptr; ok = ok && address(*a, &p) && bytes_of(*a, n); ++a; return p; }
    int num() { int v = 0; ok = ok && integer(*a++, &v); return v; }
    float real() { double v = 0.0; ok = ok && real_of(*a++, &v); return (float)v; }
    tman_stream_t stream() { void *p = nullptr; if (ok) { p = PyLong_AsVoidPtr(*a++); ok = !PyErr_Occurred(); } return (tman_stream_t)p; }
};

bool arity(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

#define TMAN_ISSUE(id, call_args)                                                   \
    do {                                                                            \
        if (!r.ok) return nullptr;                                                  \
        tman_status st;                                                             \
        Py_BEGIN_ALLOW_THREADS st = reinterpret_cast<decltype(&id)>(g_fn[f]) call_args; \
        Py_END_ALLOW_THREADS return PyLong_FromLong((long)st);                      \
    } while (0)

PyObject *matmul(int f, PyObject *const *args, Py_ssize_t n)
{
    if (!arity(n, 10)) return nullptr;
    Reader r(args);
    size_t pb = 0, wb = 0;
    void *pk = r.buf(&pb), *x = r.ptr(), *y = r.ptr();
    const int M = r.num(), K = r.num(), N = r.num(), bits = r.num(), group = r.num();
    void *ws = r.buf(&wb);
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_mpgemv, (pk, pb, x, y, M, K, N, bits, group, ws, wb, s));
}
PyObject *py_gemv(PyObject *, PyObject *const *args, Py_ssize_t n) { return matmul(F_GEMV, args, n); }
PyObject *py_gemm(PyObject *, PyObject *const *args, Py_ssize_t n) { return matmul(F_GEMM, args, n); }

PyObject *py_grouped(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    constexpr int f = F_GROUPED, MAX = 4;       // more matrices than the library takes are left to it to refuse
    if (!arity(n, 10)) return nullptr;
    PyObject *seq[3] = {nullptr, nullptr, nullptr};
    const int at[3] = {0, 2, 5};                // packed_list, y_list, N_list
    Py_ssize_t count = 0;
    bool ok = true;
    for (int i = 0; i < 3 && ok; ++i) {
        if (i == 0) {                           // packed_list needs a length, as it does for len()
            count = PyObject_Size(args[at[0]]);
            ok = count >= 0;
            if (!ok) break;
        }
        seq[i] = PySequence_Fast(args[at[i]], "expected a sequence");
        ok = seq[i] != nullptr;
        if (ok && PySequence_Fast_GET_SIZE(seq[i]) != count) {
            PyErr_SetString(PyExc_IndexError, "packed_list, y_list and N_list need an entry for every matrix and no more");
            ok = false;
        }
    }
    const void *pk[MAX] = {};
    void *y[MAX] = {};
    size_t pb[MAX] = {};
    int Ns[MAX] = {};
    for (Py_ssize_t i = 0; ok && i < count && i < MAX; ++i) {
        void *p = nullptr;
        ok = address(PySequence_Fast_GET_ITEM(seq[0], i), &p) && bytes_of(PySequence_Fast_GET_ITEM(seq[0], i), &pb[i]) &&
             address(PySequence_Fast_GET_ITEM(seq[1], i), &y[i]) && integer_of(PySequence_Fast_GET_ITEM(seq[2], i), &Ns[i]);
        pk[i] = p;
    }
    for (int i = 0; i < 3; ++i) Py_XDECREF(seq[i]);
    if (!ok) return nullptr;
    Reader r(args + 1);
    void *x = r.ptr();
    r.a = args + 3;
    const int M = r.num(), K = r.num();
    r.a = args + 6;
    const int bits = r.num(), group = r.num();
    size_t wb = 0;
    void *ws = r.buf(&wb);
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_mpgemv_grouped, ((int)count, pk, pb, x, y, M, K, Ns, bits, group, ws, wb, s));
}

PyObject *py_quant(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    constexpr int f = F_QUANT;
    if (!arity(n, 7)) return nullptr;
    Reader r(args);
    void *x = r.ptr();
    const int M = r.num(), K = r.num(), qmax = r.num();
    void *a = r.ptr(), *sc = r.ptr();
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_quantize_rows, (x, M, K, qmax, (int16_t *)a, (float *)sc, s));
}

PyObject *py_quant_i8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    constexpr int f = F_QUANT_I8;
    if (!arity(n, 6)) return nullptr;
    Reader r(args);
    void *x = r.ptr();
    const int M = r.num(), K = r.num();
    void *a = r.ptr(), *sc = r.ptr();
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_quantize_rows_i8, (x, M, K, (int8_t *)a, (float *)sc, s));
}

PyObject *py_ternary(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    constexpr int f = F_TERNARY;
    if (!arity(n, 12)) return nullptr;
    Reader r(args);
    size_t pb = 0, wb = 0;
    void *pk = r.buf(&pb), *a = r.ptr(), *sc = r.ptr();
    const float w = r.real();
    void *y = r.ptr(), *acc = r.ptr();
    const int M = r.num(), K = r.num(), N = r.num(), group = r.num();
    void *ws = r.buf(&wb);
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_mpgemv_ternary, (pk, pb, (const int16_t *)a, (const float *)sc, w, y, (int32_t *)acc, M, K, N, group, ws, wb, s));
}

PyObject *py_ternary_i8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    constexpr int f = F_TERNARY_I8;
    if (!arity(n, 11)) return nullptr;
    Reader r(args);
    size_t pb = 0, wb = 0;
    void *pk = r.buf(&pb), *a = r.ptr(), *sc = r.ptr();
    const float w = r.real();
    void *y = r.ptr();
    const int M = r.num(), K = r.num(), N = r.num(), group = r.num();
    void *ws = r.buf(&wb);
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_mpgemm_ternary_i8, (pk, pb, (const int8_t *)a, (const float *)sc, w, y, M, K, N, group, ws, wb, s));
}

PyObject *py_pack(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    constexpr int f = F_PACK;
    if (!arity(n, 9)) return nullptr;
    Reader r(args);
    void *codes = r.ptr(), *scales = r.ptr(), *zeros = r.ptr();
    const int K = r.num(), N = r.num(), bits = r.num(), group = r.num();
    size_t pb = 0;
    void *pk = r.buf(&pb);
    tman_stream_t s = r.stream();
    TMAN_ISSUE(tman_pack_weights, ((const uint8_t *)codes, scales, (const uint8_t *)zeros, K, N, bits, group, pk, pb, s));
}

// bind(addresses): the loaded library's entry points, in the order of the enumeration above
PyObject *py_bind(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (!arity(n, F_COUNT)) return nullptr;
    void *fn[F_COUNT];
    for (int i = 0; i < F_COUNT; ++i) {
        fn[i] = PyLong_AsVoidPtr(args[i]);
        if (PyErr_Occurred()) return nullptr;
        if (!fn[i]) { PyErr_SetString(PyExc_ValueError, "null entry point"); return nullptr; }
    }
    for (int i = 0; i < F_COUNT; ++i) g_fn[i] = fn[i];
    Py_RETURN_NONE;
}

#define TMAN_METHOD(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    TMAN_METHOD("bind", py_bind), TMAN_METHOD("mpgemv", py_gemv), TMAN_METHOD("mpgemv_grouped", py_grouped),
    TMAN_METHOD("mpgemm", py_gemm), TMAN_METHOD("quantize_rows", py_quant), TMAN_METHOD("quantize_rows_i8", py_quant_i8),
    TMAN_METHOD("mpgemv_ternary", py_ternary), TMAN_METHOD("mpgemm_ternary_i8", py_ternary_i8),
    TMAN_METHOD("pack_weights", py_pack), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void)
{
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_nbytes = PyUnicode_InternFromString("nbytes");
    g_numel = PyUnicode_InternFromString("numel");
    g_element_size = PyUnicode_InternFromString("element_size");
    if (!g_data_ptr || !g_nbytes || !g_numel || !g_element_size) return nullptr;
    return PyModule_Create(&module);
}
