// CPython side of the library's calls: one native function per C entry point that takes tensors, with the
// argument names of the Python interface.  It marshals and calls, nothing else.
//
// Why it is native: a decode call of one layer takes 4 to 8 us on the GPU, and marshalling its twelve arguments in
// Python (attribute look-ups, a numpy conversion of the level table, a torch Stream object per call, ctypes) took
// 10 us of host time, so calls made back to back waited for the host.  Here a call costs the driver's launch
// plus under a microsecond: pointers come from the tensors' data_ptr(), the level table from the buffer
// protocol, the current stream from torch's raw-stream query.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstring>
#include <initializer_list>

#include "lords.h"

namespace {

PyObject *g_error = nullptr;       // LordsError(status, what)
PyObject *g_table = nullptr;       // Python fall-back: (codebook, bits) -> contiguous float32 array
PyObject *g_data_ptr = nullptr;    // interned "data_ptr", "cuda_stream", "is_cuda"
PyObject *g_cuda_stream = nullptr;
PyObject *g_is_cuda = nullptr;
PyObject *g_get_device = nullptr;  // torch._C._cuda_getDevice / _cuda_getCurrentRawStream
PyObject *g_raw_stream = nullptr;

constexpr int kMaxArgs = 20;

// The arguments of one call by position, from positional and keyword arguments; `required` of them must be
// given, the others stay null.
bool gather(const char *fn, const char *const *names, int count, int required, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames,
            PyObject **out)
{
    if (nargs > count) {
        PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", fn, count, nargs);
        return false;
    }
    for (int k = 0; k < count; ++k) out[k] = k < nargs ? args[k] : nullptr;
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t j = 0; j < nkw; ++j) {
        PyObject *name = PyTuple_GET_ITEM(kwnames, j);
        int k = 0;
        while (k < count && PyUnicode_CompareWithASCIIString(name, names[k]) != 0) ++k;
        if (k == count) {
            PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", fn, name);
            return false;
        }
        if (out[k]) {
            PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", fn, names[k]);
            return false;
        }
        out[k] = args[nargs + j];
    }
    for (int k = 0; k < required; ++k)
        if (!out[k]) {
            PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", fn, names[k]);
            return false;
        }
    return true;
}

bool to_int(PyObject *o, int *v)
{
    const long l = PyLong_AsLong(o);
    if (l == -1 && PyErr_Occurred()) return false;
    *v = (int)l;
    return true;
}

// tensor.data_ptr(); `optional`: None is a null pointer
bool to_ptr(PyObject *o, bool optional, void **p)
{
    if (optional && (o == nullptr || o == Py_None)) {
        *p = nullptr;
        return true;
    }
    PyObject *v = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!v) return false;
    *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*p == nullptr && PyErr_Occurred());
}

bool to_stream(PyObject *o, void **p)
{
    PyObject *v;
    if (o && o != Py_None) {
        v = PyObject_GetAttr(o, g_cuda_stream);
    } else {
        if (!g_raw_stream) {
            PyObject *c = PyImport_ImportModule("torch._C");
            if (!c) return false;
            g_get_device = PyObject_GetAttrString(c, "_cuda_getDevice");
            g_raw_stream = g_get_device ? PyObject_GetAttrString(c, "_cuda_getCurrentRawStream") : nullptr;
            Py_DECREF(c);
            if (!g_raw_stream) return false;
        }
        PyObject *dev = PyObject_CallNoArgs(g_get_device);
        if (!dev) return false;
        v = PyObject_CallOneArg(g_raw_stream, dev);
        Py_DECREF(dev);
    }
    if (!v) return false;
    *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*p == nullptr && PyErr_Occurred());
}

// The level table as 2^bits floats: a contiguous float32 buffer of that size as it is, anything else through the
// Python conversion (which also reports a table of the wrong size).
struct Table {
    Py_buffer view;
    PyObject *owned = nullptr;
    bool held = false;
    ~Table()
    {
        if (held) PyBuffer_Release(&view);
        Py_XDECREF(owned);
    }
    bool take(PyObject *o)
    {
        if (PyObject_GetBuffer(o, &view, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS) != 0) return false;
        held = true;
        return true;
    }
    bool is(int bits) const
    {
        return view.itemsize == 4 && view.format && std::strcmp(view.format, "f") == 0 && bits >= 0 && bits < 16 && view.len == ((Py_ssize_t)4 << bits);
    }
    bool read(PyObject *o, int bits)
    {
        if (PyObject_CheckBuffer(o)) {
            if (take(o)) {
                if (is(bits)) return true;
                PyBuffer_Release(&view);
                held = false;
            } else {
                PyErr_Clear();
            }
        }
        owned = PyObject_CallFunction(g_table, "Oi", o, bits);
        if (!owned || !take(owned)) return false;
        if (is(bits)) return true;
        PyErr_SetString(PyExc_ValueError, "codebook must hold 2**bits floats");
        return false;
    }
    const float *data() const { return static_cast<const float *>(view.buf); }
};

PyObject *done(int status, const char *what)
{
    if (status == LORDS_OK) Py_RETURN_NONE;
    PyObject *e = PyObject_CallFunction(g_error, "is", status, what);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    return nullptr;
}

#define LORDS_ARGS(FN, COUNT, REQUIRED, ...)                                                    \
    static const char *const names[] = {__VA_ARGS__};                                           \
    static_assert(sizeof(names) / sizeof(names[0]) == (COUNT) && (COUNT) <= kMaxArgs, FN);      \
    PyObject *a[COUNT];                                                                         \
    if (!gather(FN, names, COUNT, REQUIRED, args, nargs, kwnames, a)) return nullptr

#define LORDS_CALL(EXPR)          \
    int status;                   \
    Py_BEGIN_ALLOW_THREADS        \
    status = (EXPR);              \
    Py_END_ALLOW_THREADS

typedef int (*ForwardFn)(const void *, const uint8_t *, const void *, const void *, const float *, int, int, int, int, int, void *, void *);

// x, Qpacked, B, A, codebook, bits, M, m, n, r, y, stream: the calls that share this list differ in y's name only
PyObject *forward_call(const char *fn, ForwardFn call, PyObject **a, bool host)
{
    int v[5];
    void *x, *q, *B, *A, *y, *s;
    Table cb;
    for (int k = 0; k < 5; ++k)
        if (!to_int(a[5 + k], &v[k])) return nullptr;
    if (!cb.read(a[4], v[0])) return nullptr;
    if (host)
        for (int k : {0, 10}) {
            PyObject *c = PyObject_GetAttr(a[k], g_is_cuda);
            if (!c) return nullptr;
            const int is = PyObject_IsTrue(c);
            Py_DECREF(c);
            if (is < 0) return nullptr;
            if (is) {
                PyErr_SetString(PyExc_ValueError, "x_host and y_host must be host tensors");
                return nullptr;
            }
        }
    if (!to_ptr(a[0], false, &x) || !to_ptr(a[1], false, &q) || !to_ptr(a[2], false, &B) || !to_ptr(a[3], false, &A) || !to_ptr(a[10], false, &y) ||
        !to_stream(a[11], &s))
        return nullptr;
    LORDS_CALL(call(x, static_cast<const uint8_t *>(q), B, A, cb.data(), v[0], v[1], v[2], v[3], v[4], y, s));
    return done(status, fn);
}

int forward_f32(const void *x, const uint8_t *q, const void *B, const void *A, const float *cb, int bits, int M, int m, int n, int r, void *y, void *s)
{
    return lords_linear_forward_f32(x, q, B, A, cb, bits, M, m, n, r, static_cast<float *>(y), s);
}
int backward_input_f32(const void *dy, const uint8_t *qt, const void *B, const void *A, const float *cb, int bits, int M, int m, int n, int r, void *dx, void *s)
{
    return lords_linear_backward_input_f32(dy, qt, B, A, cb, bits, M, m, n, r, static_cast<float *>(dx), s);
}

#define LORDS_FORWARD(NAME, CALL, HOST, X, Q, Y)                                                                        \
    PyObject *py_##NAME(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)                         \
    {                                                                                                                   \
        LORDS_ARGS(#NAME, 12, 11, X, Q, "B", "A", "codebook", "bits", "M", "m", "n", "r", Y, "stream");                 \
        return forward_call(#NAME, CALL, a, HOST);                                                                      \
    }

LORDS_FORWARD(lords_linear_forward_bits, lords_linear_forward_bits, false, "x", "Qpacked", "y")
LORDS_FORWARD(lords_linear_forward_f32, forward_f32, false, "x", "Qpacked", "y32")
LORDS_FORWARD(lords_linear_forward_host, lords_linear_forward_host, true, "x_host", "Qpacked", "y_host")
LORDS_FORWARD(lords_linear_forward_noalloc, lords_linear_forward_noalloc, false, "x", "Qpacked", "y")
LORDS_FORWARD(lords_linear_backward_input, lords_linear_backward_input, false, "dy", "Qt_packed", "dx")
LORDS_FORWARD(lords_linear_backward_input_f32, backward_input_f32, false, "dy", "Qt_packed", "dx32")

PyObject *py_lords_linear_forward(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_linear_forward", 11, 10, "x", "Qpacked", "B", "A", "codebook", "M", "m", "n", "r", "y", "stream");
    int v[4];
    void *x, *q, *B, *A, *y, *s;
    Table cb;
    for (int k = 0; k < 4; ++k)
        if (!to_int(a[5 + k], &v[k])) return nullptr;
    if (!cb.read(a[4], 4) || !to_ptr(a[0], false, &x) || !to_ptr(a[1], false, &q) || !to_ptr(a[2], false, &B) || !to_ptr(a[3], false, &A) ||
        !to_ptr(a[9], false, &y) || !to_stream(a[10], &s))
        return nullptr;
    LORDS_CALL(lords_linear_forward(x, static_cast<const uint8_t *>(q), B, A, cb.data(), v[0], v[1], v[2], v[3], y, s));
    return done(status, "lords_linear_forward");
}

PyObject *py_lords_quantize_codes(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_quantize_codes", 10, 9, "W", "B", "A", "codebook", "bits", "m", "n", "r", "Qpacked", "stream");
    int v[4];
    void *W, *B, *A, *q, *s;
    Table cb;
    for (int k = 0; k < 4; ++k)
        if (!to_int(a[4 + k], &v[k])) return nullptr;
    if (!cb.read(a[3], v[0]) || !to_ptr(a[0], false, &W) || !to_ptr(a[1], false, &B) || !to_ptr(a[2], false, &A) || !to_ptr(a[8], false, &q) ||
        !to_stream(a[9], &s))
        return nullptr;
    LORDS_CALL(lords_quantize_codes(W, B, A, cb.data(), v[0], v[1], v[2], v[3], static_cast<uint8_t *>(q), s));
    return done(status, "lords_quantize_codes");
}

PyObject *py_lords_transpose_codes(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_transpose_codes", 6, 5, "Qpacked", "bits", "m", "n", "Qt_packed", "stream");
    int v[3];
    void *q, *qt, *s;
    for (int k = 0; k < 3; ++k)
        if (!to_int(a[1 + k], &v[k])) return nullptr;
    if (!to_ptr(a[0], false, &q) || !to_ptr(a[4], false, &qt) || !to_stream(a[5], &s)) return nullptr;
    LORDS_CALL(lords_transpose_codes(static_cast<const uint8_t *>(q), v[0], v[1], v[2], static_cast<uint8_t *>(qt), s));
    return done(status, "lords_transpose_codes");
}

PyObject *py_lords_linear_backward_factors(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_linear_backward_factors", 14, 13, "dy", "x", "Qpacked", "B", "A", "codebook", "bits", "M", "m", "n", "r", "dB", "dA", "stream");
    int v[5];
    void *dy, *x, *q, *B, *A, *dB, *dA, *s;
    Table cb;
    for (int k = 0; k < 5; ++k)
        if (!to_int(a[6 + k], &v[k])) return nullptr;
    if (!cb.read(a[5], v[0]) || !to_ptr(a[0], false, &dy) || !to_ptr(a[1], false, &x) || !to_ptr(a[2], false, &q) || !to_ptr(a[3], false, &B) ||
        !to_ptr(a[4], false, &A) || !to_ptr(a[11], true, &dB) || !to_ptr(a[12], true, &dA) || !to_stream(a[13], &s))
        return nullptr;
    LORDS_CALL(lords_linear_backward_factors(dy, x, static_cast<const uint8_t *>(q), B, A, cb.data(), v[0], v[1], v[2], v[3], v[4],
                                             static_cast<float *>(dB), static_cast<float *>(dA), s));
    return done(status, "lords_linear_backward_factors");
}

PyObject *py_lords_linear_backward_qat(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_linear_backward_qat", 16, 15, "dy", "x", "W", "Qpacked", "B", "A", "codebook", "bits", "M", "m", "n", "r", "dW", "dB", "dA",
               "stream");
    int v[5];
    void *dy, *x, *W, *q, *B, *A, *dW, *dB, *dA, *s;
    Table cb;
    for (int k = 0; k < 5; ++k)
        if (!to_int(a[7 + k], &v[k])) return nullptr;
    if (!cb.read(a[6], v[0]) || !to_ptr(a[0], false, &dy) || !to_ptr(a[1], false, &x) || !to_ptr(a[2], false, &W) || !to_ptr(a[3], false, &q) ||
        !to_ptr(a[4], false, &B) || !to_ptr(a[5], false, &A) || !to_ptr(a[12], true, &dW) || !to_ptr(a[13], true, &dB) || !to_ptr(a[14], true, &dA) ||
        !to_stream(a[15], &s))
        return nullptr;
    LORDS_CALL(lords_linear_backward_qat(dy, x, W, static_cast<const uint8_t *>(q), B, A, cb.data(), v[0], v[1], v[2], v[3], v[4],
                                         static_cast<float *>(dW), static_cast<float *>(dB), static_cast<float *>(dA), s));
    return done(status, "lords_linear_backward_qat");
}

PyObject *py_lords_blockscale_forward(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_blockscale_forward", 12, 10, "x", "Qpacked", "scales", "codebook", "bits", "blk", "M", "m", "n", "y", "stream", "f32");
    int v[5];
    void *x, *q, *sc, *y, *s;
    Table cb;
    for (int k = 0; k < 5; ++k)
        if (!to_int(a[4 + k], &v[k])) return nullptr;
    const int f32 = a[11] ? PyObject_IsTrue(a[11]) : 0;
    if (f32 < 0 || !cb.read(a[3], v[0]) || !to_ptr(a[0], false, &x) || !to_ptr(a[1], false, &q) || !to_ptr(a[2], false, &sc) || !to_ptr(a[9], false, &y) ||
        !to_stream(a[10], &s))
        return nullptr;
    const uint8_t *q8 = static_cast<const uint8_t *>(q);
    LORDS_CALL(f32 ? lords_blockscale_forward_f32(x, q8, sc, cb.data(), v[0], v[1], v[2], v[3], v[4], static_cast<float *>(y), s)
                   : lords_blockscale_forward(x, q8, sc, cb.data(), v[0], v[1], v[2], v[3], v[4], y, s));
    return done(status, "lords_blockscale_forward");
}

PyObject *py_lords_adapter_forward(PyObject *, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    LORDS_ARGS("lords_adapter_forward", 15, 13, "x", "Qpacked", "scales", "A_l", "B_l", "codebook", "bits", "blk", "M", "m", "n", "r", "y", "stream", "f32");
    int v[6];
    void *x, *q, *sc, *Al, *Bl, *y, *s;
    Table cb;
    for (int k = 0; k < 6; ++k)
        if (!to_int(a[6 + k], &v[k])) return nullptr;
    const int f32 = a[14] ? PyObject_IsTrue(a[14]) : 0;
    if (f32 < 0 || !cb.read(a[5], v[0]) || !to_ptr(a[0], false, &x) || !to_ptr(a[1], false, &q) || !to_ptr(a[2], false, &sc) || !to_ptr(a[3], false, &Al) ||
        !to_ptr(a[4], false, &Bl) || !to_ptr(a[12], false, &y) || !to_stream(a[13], &s))
        return nullptr;
    const uint8_t *q8 = static_cast<const uint8_t *>(q);
    LORDS_CALL(f32 ? lords_adapter_forward_f32(x, q8, sc, Al, Bl, cb.data(), v[0], v[1], v[2], v[3], v[4], v[5], static_cast<float *>(y), s)
                   : lords_adapter_forward(x, q8, sc, Al, Bl, cb.data(), v[0], v[1], v[2], v[3], v[4], v[5], y, s));
    return done(status, "lords_adapter_forward");
}

PyObject *py_setup(PyObject *, PyObject *args)
{
    PyObject *error, *table;
    if (!PyArg_ParseTuple(args, "OO", &error, &table)) return nullptr;
    Py_INCREF(error);
    Py_INCREF(table);
    Py_XSETREF(g_error, error);
    Py_XSETREF(g_table, table);
    Py_RETURN_NONE;
}

#define LORDS_DEF(NAME, DOC) {#NAME, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(py_##NAME)), METH_FASTCALL | METH_KEYWORDS, DOC}

PyMethodDef g_methods[] = {
    {"setup", py_setup, METH_VARARGS, "setup(error_class, table_conversion)"},
    LORDS_DEF(lords_linear_forward, "lords_linear_forward(x, Qpacked, B, A, codebook, M, m, n, r, y, stream=None)\n--\n\n"
              "4-bit entry point: device tensors x[M,n], Qpacked[m,n/2], B[m,r], A[r,n] -> y[M,m] (bf16)."),
    LORDS_DEF(lords_linear_forward_bits, "lords_linear_forward_bits(x, Qpacked, B, A, codebook, bits, M, m, n, r, y, stream=None)\n--\n\n"
              "The same with an explicit code width."),
    LORDS_DEF(lords_linear_forward_f32, "lords_linear_forward_f32(x, Qpacked, B, A, codebook, bits, M, m, n, r, y32, stream=None)\n--\n\n"
              "The same with the fp32 accumulator stored."),
    LORDS_DEF(lords_linear_forward_host, "lords_linear_forward_host(x_host, Qpacked, B, A, codebook, bits, M, m, n, r, y_host, stream=None)\n--\n\n"
              "x_host / y_host are CPU tensors (pinned for asynchronous copies); weights are device tensors."),
    LORDS_DEF(lords_linear_forward_noalloc, "lords_linear_forward_noalloc(x, Qpacked, B, A, codebook, bits, M, m, n, r, y, stream=None)\n--\n\n"
              "Forward that never allocates and needs no lords_init (scratch lives in the library image)."),
    LORDS_DEF(lords_quantize_codes, "lords_quantize_codes(W, B, A, codebook, bits, m, n, r, Qpacked, stream=None)\n--\n\n"
              "Alg. 1 step 2.1 on the device: packed codes of the nearest levels of W / (B A)."),
    LORDS_DEF(lords_transpose_codes, "lords_transpose_codes(Qpacked, bits, m, n, Qt_packed, stream=None)\n--\n\n"
              "Packed codes of Q^T (n rows of m codes) from the packed codes of Q, on the device."),
    LORDS_DEF(lords_linear_backward_input, "lords_linear_backward_input(dy, Qt_packed, B, A, codebook, bits, M, m, n, r, dx, stream=None)\n--\n\n"
              "dx = dy W^ (bf16 [M, n]) for a layer whose transposed codes Qt_packed were made by lords_transpose_codes."),
    LORDS_DEF(lords_linear_backward_input_f32, "lords_linear_backward_input_f32(dy, Qt_packed, B, A, codebook, bits, M, m, n, r, dx32, stream=None)\n--\n\n"
              "The same with the fp32 accumulator stored (float [M, n])."),
    LORDS_DEF(lords_linear_backward_factors, "lords_linear_backward_factors(dy, x, Qpacked, B, A, codebook, bits, M, m, n, r, dB, dA, stream=None)\n--\n\n"
              "dB (float [m, r]) and dA (float [r, n]) of the layer with the codes fixed; either may be None."),
    LORDS_DEF(lords_linear_backward_qat, "lords_linear_backward_qat(dy, x, W, Qpacked, B, A, codebook, bits, M, m, n, r, dW, dB, dA, stream=None)\n--\n\n"
              "Straight-through gradients of quantisation-aware training (Eq. 4-5); any of dW, dB, dA may be None."),
    LORDS_DEF(lords_blockscale_forward, "lords_blockscale_forward(x, Qpacked, scales, codebook, bits, blk, M, m, n, y, stream=None, f32=False)\n--\n\n"
              "Comparator (Eq. 2): y = x (L[Q] (.) (s (x) 1))^T; y is bf16 [M, m], or float with f32=True."),
    LORDS_DEF(lords_adapter_forward, "lords_adapter_forward(x, Qpacked, scales, A_l, B_l, codebook, bits, blk, M, m, n, r, y, stream=None, f32=False)\n--\n\n"
              "Comparator (Sec. 3.4 / 4.4): the block-scaled layer plus an additive rank-r adapter, three launches."),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_native", "Native calls of the LoRDS library (see binding.py).", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void)
{
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    g_is_cuda = PyUnicode_InternFromString("is_cuda");
    return PyModule_Create(&g_module);
}
