/*
 * Argument marshalling of the Python binding (_lib.py) in C: one function per launching entry
 * point of libkeyless. An address argument is None, an int, or an object with data_ptr(); a shape or
 * options argument is the ctypes structure of _lib.py; an integer has __index__() or is a ctypes
 * c_int32; the stream is None (torch's current stream), an int, or an object with cuda_stream. Other
 * types are refused with ctypes' own exceptions. Each returns the kl_status.
 *
 * The module is not linked to libkeyless: bind() takes the entry points' addresses from the library
 * that _lib.py has loaded (and the structure classes), so that both always call the same copy, whatever
 * the loader's search path holds.
 *
 * A small decode takes the GPU 6 to 8 us and the C call 2, while ctypes with a c_void_p object per
 * argument and torch.cuda.current_stream() took 15 us of host time in front of it, plain ints and
 * the raw stream through ctypes 6, and this takes about 2.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "keyless.h"

static PyObject *s_data_ptr, *s_numel, *s_element_size, *s_cuda_stream;
static PyObject *s_value, *s_as_parameter;
static PyObject *g_argument_error, *g_cdata, *g_c_int, *g_sizeof;   /* ctypes: ArgumentError, _CData, c_int32, sizeof */
static PyObject *g_shape, *g_latent, *g_options;          /* the structure classes (bind()) */
static PyObject *g_initialized, *g_get_device, *g_raw_stream, *g_current_stream;   /* torch */

#define ENTRIES(X) \
    X(route_query) X(append_v) X(decode_attention) X(decode_attention_ex) X(decode_step) X(combine) \
    X(standard_decode) X(decode_attention_noalloc) X(append_v_chunk) X(prefill_attention) \
    X(append_v_fp8) X(quantize_cache_fp8) X(decode_attention_fp8) X(decode_step_fp8) \
    X(latent_decode) X(latent_decode_step)
#define POINTER(n) static __typeof__(kl_##n) *f_##n;
ENTRIES(POINTER)
#define SLOT(n) {"kl_" #n, &f_##n},
static const struct { const char *name; void *to; } slots[] = {ENTRIES(SLOT)};
enum { kEntries = sizeof slots / sizeof slots[0] };

/* The int `v`, as ctypes takes it (bits past the 64th dropped). */
static int to_u64(PyObject *v, uint64_t *out) {
    if (!PyLong_Check(v)) {
        PyErr_Format(PyExc_TypeError, "expected an int, got %.100s", Py_TYPE(v)->tp_name);
        return 0;
    }
    *out = PyLong_AsUnsignedLongLongMask(v);
    return !(*out == (uint64_t)-1 && PyErr_Occurred());
}

static int get_addr(PyObject *o, void **out) {
    uint64_t x = 0;
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    if (PyLong_Check(o)) {
        if (!to_u64(o, &x)) return 0;
    } else {
        PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
        if (!v) return 0;
        const int ok = v == Py_None || to_u64(v, &x);
        Py_DECREF(v);
        if (!ok) return 0;
    }
    *out = (void *)(uintptr_t)x;
    return 1;
}

static int get_i32(PyObject *o, int32_t *out) {
    if (PyIndex_Check(o)) {
        const unsigned long v = PyLong_AsUnsignedLongMask(o);
        if (v == (unsigned long)-1 && PyErr_Occurred()) return 0;
        *out = (int32_t)v;
        return 1;
    }
    const int is_c = PyObject_IsInstance(o, g_c_int);
    if (is_c < 0) return 0;
    PyObject *v = PyObject_GetAttr(o, is_c ? s_value : s_as_parameter);
    if (!v) {
        PyErr_Clear();
        PyErr_Format(g_argument_error, "expected an int, got %.100s", Py_TYPE(o)->tp_name);
        return 0;
    }
    int ok = !Py_EnterRecursiveCall(" in an integer argument");
    if (ok) {
        ok = get_i32(v, out);
        Py_LeaveRecursiveCall();
    }
    Py_DECREF(v);
    return ok;
}

/* The contents of an instance of the ctypes structure `type` (`size` bytes, or a subclass's more). */
static int get_struct(PyObject *o, void *out, Py_ssize_t size, PyObject *type) {
    Py_buffer b;
    if (!type) {
        PyErr_SetString(PyExc_RuntimeError, "bind() first");
        return 0;
    }
    int is = PyObject_IsInstance(o, type);
    if (is == 0) {
        is = PyObject_IsInstance(o, g_cdata);
        if (is >= 0)
            PyErr_Format(is ? g_argument_error : PyExc_TypeError, "expected %.100s, got %.100s",
                         ((PyTypeObject *)type)->tp_name, Py_TYPE(o)->tp_name);
        return 0;
    }
    if (is < 0 || PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) < 0) return 0;
    memcpy(out, b.buf, (size_t)size);
    PyBuffer_Release(&b);
    return 1;
}

/* bind({name: address}, shape, latent_shape, options): the library's entry points and the structure
 * classes that they take. */
static PyObject *py_bind(PyObject *m, PyObject *const *a, Py_ssize_t na) {
    (void)m;
    const Py_ssize_t size[3] = {sizeof(kl_shape), sizeof(kl_latent_shape), sizeof(kl_decode_options)};
    PyObject **to[3] = {&g_shape, &g_latent, &g_options};
    void *entry[kEntries];
    if (na != 4 || !PyDict_Check(a[0])) {
        PyErr_SetString(PyExc_TypeError, "bind takes a dict and 3 classes");
        return NULL;
    }
    for (int i = 0; i < kEntries; ++i) {
        PyObject *v = PyDict_GetItemString(a[0], slots[i].name);
        if (!v || !(entry[i] = PyLong_AsVoidPtr(v))) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, slots[i].name);
            return NULL;
        }
    }
    for (int i = 0; i < 3; ++i) {
        PyObject *n = PyObject_CallOneArg(g_sizeof, a[1 + i]);
        if (!n) return NULL;
        const Py_ssize_t have = PyLong_AsSsize_t(n);
        Py_DECREF(n);
        if (have != size[i] || !PyType_Check(a[1 + i])) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "a structure of another size");
            return NULL;
        }
    }
    for (int i = 0; i < kEntries; ++i) memcpy(slots[i].to, &entry[i], sizeof(void *));
    for (int i = 0; i < 3; ++i) {
        Py_INCREF(a[1 + i]);
        Py_XSETREF(*to[i], a[1 + i]);
    }
    Py_RETURN_NONE;
}

/* numel() * element_size() of a tensor, 0 of None. */
static int get_nbytes(PyObject *o, size_t *out) {
    uint64_t n, e;
    if (o == Py_None) {
        *out = 0;
        return 1;
    }
    PyObject *v = PyObject_CallMethodNoArgs(o, s_numel);
    if (!v) return 0;
    int ok = to_u64(v, &n);
    Py_DECREF(v);
    if (!ok) return 0;
    v = PyObject_CallMethodNoArgs(o, s_element_size);
    if (!v) return 0;
    ok = to_u64(v, &e);
    Py_DECREF(v);
    *out = (size_t)(n * e);
    return ok;
}

static int find_torch(void) {
    PyObject *cuda = PyImport_ImportModule("torch.cuda"), *c = PyImport_ImportModule("torch._C");
    int ok = cuda && c;
    ok = ok && (g_current_stream = PyObject_GetAttrString(cuda, "current_stream"));
    ok = ok && (g_get_device = PyObject_GetAttrString(c, "_cuda_getDevice"));
    ok = ok && (g_raw_stream = PyObject_GetAttrString(c, "_cuda_getCurrentRawStream"));
    ok = ok && (g_initialized = PyObject_GetAttrString(cuda, "is_initialized"));   /* last: the mark */
    Py_XDECREF(cuda);
    Py_XDECREF(c);
    return ok;
}

static int get_stream(PyObject *o, kl_stream_t *out) {
    uint64_t x = 0;
    PyObject *v;
    if (PyLong_Check(o)) {
        if (!to_u64(o, &x)) return 0;
    } else if (o != Py_None) {
        v = PyObject_GetAttr(o, s_cuda_stream);
        if (!v) return 0;
        const int ok = v == Py_None || to_u64(v, &x);
        Py_DECREF(v);
        if (!ok) return 0;
    } else {
        if (!g_initialized && !find_torch()) return 0;
        v = PyObject_CallNoArgs(g_initialized);
        if (!v) return 0;
        const int init = PyObject_IsTrue(v);
        Py_DECREF(v);
        if (init < 0) return 0;
        if (!init) {                       /* current_stream() initializes CUDA */
            v = PyObject_CallNoArgs(g_current_stream);
            if (!v) return 0;
            const int ok = get_stream(v, out);
            Py_DECREF(v);
            return ok;
        }
        PyObject *d = PyObject_CallNoArgs(g_get_device);
        if (!d) return 0;
        v = PyObject_CallOneArg(g_raw_stream, d);
        Py_DECREF(d);
        if (!v) return 0;
        const int ok = to_u64(v, &x);
        Py_DECREF(v);
        if (!ok) return 0;
    }
    *out = (kl_stream_t)(uintptr_t)x;
    return 1;
}

#define SHAPE(i) kl_shape sh; if (!get_struct(a[i], &sh, sizeof sh, g_shape)) return NULL
#define LATENT(i) kl_latent_shape sh; if (!get_struct(a[i], &sh, sizeof sh, g_latent)) return NULL
#define PTR(i, x) void *x; if (!get_addr(a[i], &x)) return NULL
#define INT(i, x) int32_t x; if (!get_i32(a[i], &x)) return NULL
#define OPTS(i) kl_decode_options o; const int has_o = a[i] != Py_None; \
    if (has_o && !get_struct(a[i], &o, sizeof o, g_options)) return NULL
#define WORK(i) void *ws; size_t wsn; if (!get_addr(a[i], &ws) || !get_nbytes(a[i], &wsn)) return NULL
#define STREAM(i) kl_stream_t st; if (!get_stream(a[i], &st)) return NULL
#define FN(name, n) static PyObject *py_##name(PyObject *m, PyObject *const *a, Py_ssize_t na) { \
    (void)m; \
    if (na != (n)) { PyErr_Format(PyExc_TypeError, #name " takes %d arguments", (n)); return NULL; }
#define CALL(expr) kl_status r; Py_BEGIN_ALLOW_THREADS r = (expr); Py_END_ALLOW_THREADS \
    return PyLong_FromLong((long)r); }

FN(route_query, 5) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, out); STREAM(4);
CALL(f_route_query(&sh, q, w, out, st))

FN(append_v, 7) SHAPE(0); PTR(1, v); PTR(2, bt); PTR(3, pos); PTR(4, c); PTR(5, e); STREAM(6);
CALL(f_append_v(&sh, v, bt, pos, c, e, st))

FN(decode_attention, 12) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, c); PTR(4, bt); PTR(5, sl); INT(6, ns);
PTR(7, out); INT(8, dt); WORK(9); PTR(10, e); STREAM(11);
CALL(f_decode_attention(&sh, q, w, c, bt, sl, ns, out, (kl_dtype)dt, ws, wsn, e, st))

FN(decode_attention_ex, 12) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, c); PTR(4, bt); PTR(5, sl); OPTS(6);
PTR(7, out); INT(8, dt); WORK(9); PTR(10, e); STREAM(11);
CALL(f_decode_attention_ex(&sh, q, w, c, bt, sl, has_o ? &o : NULL, out, (kl_dtype)dt, ws, wsn, e, st))

FN(decode_step, 14) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, v); PTR(4, pos); PTR(5, c); PTR(6, bt);
PTR(7, sl); OPTS(8); PTR(9, out); INT(10, dt); WORK(11); PTR(12, e); STREAM(13);
CALL(f_decode_step(&sh, q, w, v, pos, c, bt, sl, has_o ? &o : NULL, out, (kl_dtype)dt, ws, wsn, e, st))

FN(combine, 7) SHAPE(0); PTR(1, po); PTR(2, ml); INT(3, ns); PTR(4, out); INT(5, dt); STREAM(6);
CALL(f_combine(&sh, po, ml, ns, out, (kl_dtype)dt, st))

FN(standard_decode, 12) SHAPE(0); PTR(1, q); PTR(2, k); PTR(3, c); PTR(4, bt); PTR(5, sl); OPTS(6);
PTR(7, out); INT(8, dt); WORK(9); PTR(10, e); STREAM(11);
CALL(f_standard_decode(&sh, q, k, c, bt, sl, has_o ? &o : NULL, out, (kl_dtype)dt, ws, wsn, e, st))

FN(decode_attention_noalloc, 11) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, c); PTR(4, bt); PTR(5, sl);
INT(6, ns); PTR(7, out); INT(8, dt); PTR(9, e); STREAM(10);
CALL(f_decode_attention_noalloc(&sh, q, w, c, bt, sl, ns, out, (kl_dtype)dt, e, st))

FN(append_v_chunk, 10) SHAPE(0); PTR(1, v); PTR(2, bt); PTR(3, sl); PTR(4, cu); INT(5, tq); INT(6, mq);
PTR(7, c); PTR(8, e); STREAM(9);
CALL(f_append_v_chunk(&sh, v, bt, sl, cu, tq, mq, c, e, st))

FN(prefill_attention, 13) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, c); PTR(4, bt); PTR(5, sl); PTR(6, cu);
INT(7, tq); INT(8, mq); PTR(9, out); INT(10, dt); PTR(11, e); STREAM(12);
CALL(f_prefill_attention(&sh, q, w, c, bt, sl, cu, tq, mq, out, (kl_dtype)dt, e, st))

FN(append_v_fp8, 8) SHAPE(0); PTR(1, v); PTR(2, bt); PTR(3, pos); PTR(4, c); PTR(5, s); PTR(6, e);
STREAM(7);
CALL(f_append_v_fp8(&sh, v, bt, pos, c, s, e, st))

FN(quantize_cache_fp8, 5) SHAPE(0); PTR(1, v); PTR(2, c); PTR(3, s); STREAM(4);
CALL(f_quantize_cache_fp8(&sh, v, c, s, st))

FN(decode_attention_fp8, 13) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, c); PTR(4, s); PTR(5, bt); PTR(6, sl);
INT(7, ns); PTR(8, out); INT(9, dt); WORK(10); PTR(11, e); STREAM(12);
CALL(f_decode_attention_fp8(&sh, q, w, c, s, bt, sl, ns, out, (kl_dtype)dt, ws, wsn, e, st))

FN(decode_step_fp8, 15) SHAPE(0); PTR(1, q); PTR(2, w); PTR(3, v); PTR(4, pos); PTR(5, c); PTR(6, s);
PTR(7, bt); PTR(8, sl); INT(9, ns); PTR(10, out); INT(11, dt); WORK(12); PTR(13, e); STREAM(14);
CALL(f_decode_step_fp8(&sh, q, w, v, pos, c, s, bt, sl, ns, out, (kl_dtype)dt, ws, wsn, e, st))

FN(latent_decode, 13) LATENT(0); PTR(1, q); PTR(2, w); PTR(3, wp); PTR(4, c); PTR(5, bt); PTR(6, sl);
INT(7, ns); PTR(8, out); INT(9, dt); WORK(10); PTR(11, e); STREAM(12);
CALL(f_latent_decode(&sh, q, w, wp, c, bt, sl, ns, out, (kl_dtype)dt, ws, wsn, e, st))

FN(latent_decode_step, 15) LATENT(0); PTR(1, q); PTR(2, w); PTR(3, wp); PTR(4, v); PTR(5, pos); PTR(6, c);
PTR(7, bt); PTR(8, sl); INT(9, ns); PTR(10, out); INT(11, dt); WORK(12); PTR(13, e); STREAM(14);
CALL(f_latent_decode_step(&sh, q, w, wp, v, pos, c, bt, sl, ns, out, (kl_dtype)dt, ws, wsn, e, st))

#define M(name) {"kl_" #name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL},
static PyMethodDef methods[] = {
    ENTRIES(M) {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_keyless", NULL, -1, methods,
                                    NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__keyless(void) {
    PyObject *c = PyImport_ImportModule("ctypes");
    if (!c) return NULL;
    g_argument_error = PyObject_GetAttrString(c, "ArgumentError");
    g_c_int = PyObject_GetAttrString(c, "c_int32");
    g_sizeof = PyObject_GetAttrString(c, "sizeof");
    PyObject *st = PyObject_GetAttrString(c, "Structure");
    g_cdata = st ? PyObject_GetAttrString(st, "__base__") : NULL;
    Py_XDECREF(st);
    Py_DECREF(c);
    if (!g_argument_error || !g_c_int || !g_sizeof || !g_cdata) return NULL;
    if (!(s_data_ptr = PyUnicode_InternFromString("data_ptr")) ||
        !(s_numel = PyUnicode_InternFromString("numel")) ||
        !(s_element_size = PyUnicode_InternFromString("element_size")) ||
        !(s_cuda_stream = PyUnicode_InternFromString("cuda_stream")) ||
        !(s_value = PyUnicode_InternFromString("value")) ||
        !(s_as_parameter = PyUnicode_InternFromString("_as_parameter_")))
        return NULL;
    return PyModule_Create(&module);
}
