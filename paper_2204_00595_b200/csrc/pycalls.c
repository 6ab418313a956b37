/* Argument marshalling of the hot calls for CPython: the same checks and conversions as binding.py's helpers, without
 * ctypes.  A call on a few tokens takes the GPU 5 to 10 us, and ctypes with the checks written in Python took the host
 * 6 to 7 us of every call (4 attribute reads per tensor, 11 to 22 argument conversions); this takes about 1 us.
 *
 * Call(name, address, spec, names, float_types, on_error, stream_of) is a callable object.  spec has one letter per
 * positional argument, in the order of the C function's parameters:
 *   t  tensor of the storage dtype (the first one decides which)      f  float32 tensor       q  int64 tensor
 *   i  integer     w  workspace: object with ptr and nbytes, or (ptr, nbytes); two C parameters
 *   v  workspace pointer, or None     s  stream: None (the current one), an integer, or an object with cuda_stream
 *   D  (no argument) the dtype code
 * None as a tensor is a null pointer.  A non-zero status is given to on_error(status, name). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "monarch.h"

#define MAX_ARGS 24

typedef int (*apply_fn)(void *, const uint64_t *);
#define P(k) ((void *)(uintptr_t)a[k])
#define F(k) ((float *)(uintptr_t)a[k])
#define I(k) ((int32_t)a[k])
#define L(k) ((int64_t)a[k])
#define Z(k) ((size_t)a[k])
#define APPLY(name, ...) \
    static int apply_##name(void *fn, const uint64_t *a) { return ((__typeof__(name) *)fn)(__VA_ARGS__); }
APPLY(monarch_fwd, P(0), P(1), P(2), P(3), L(4), I(5), I(6), I(7), P(8), Z(9), P(10))
APPLY(monarch_bwd_dx, P(0), P(1), P(2), P(3), L(4), I(5), I(6), I(7), P(8), Z(9), P(10))
APPLY(monarch_bwd_dw, P(0), P(1), P(2), P(3), F(4), F(5), I(6), L(7), I(8), I(9), I(10), P(11), Z(12), P(13))
APPLY(monarch_bwd, P(0), P(1), P(2), P(3), P(4), P(5), F(6), F(7), I(8), L(9), I(10), I(11), I(12), P(13), Z(14), P(15))
APPLY(monarch_mlp_fwd, P(0), P(1), P(2), P(3), P(4), P(5), P(6), P(7), L(8), I(9), I(10), I(11), P(12), Z(13), P(14))
APPLY(monarch_mlp_bwd, P(0), P(1), P(2), P(3), P(4), P(5), P(6), P(7), F(8), F(9), F(10), F(11), F(12), F(13), I(14), L(15),
      I(16), I(17), I(18), P(19), Z(20), P(21))
APPLY(monarch_rect_fwd, P(0), P(1), P(2), P(3), L(4), I(5), I(6), I(7), I(8), I(9), P(10), Z(11), P(12))
APPLY(monarch_rect_bwd, P(0), P(1), P(2), P(3), P(4), P(5), F(6), F(7), I(8), L(9), I(10), I(11), I(12), I(13), I(14), P(15),
      Z(16), P(17))
APPLY(monarch_cplx_fwd, P(0), P(1), P(2), P(3), I(4), L(5), I(6), I(7), I(8), P(9), Z(10), P(11))
APPLY(monarch_dense, P(0), P(1), P(2), I(3), I(4), I(5), P(6))
APPLY(monarch_project, P(0), P(1), P(2), I(3), I(4), I(5), (unsigned long long *)P(6), P(7))

static const struct { const char *name; apply_fn apply; int params; } kCalls[] = {
    {"monarch_fwd", apply_monarch_fwd, 11},         {"monarch_bwd_dx", apply_monarch_bwd_dx, 11},
    {"monarch_bwd_dw", apply_monarch_bwd_dw, 14},   {"monarch_bwd", apply_monarch_bwd, 16},
    {"monarch_mlp_fwd", apply_monarch_mlp_fwd, 15}, {"monarch_mlp_bwd", apply_monarch_mlp_bwd, 22},
    {"monarch_rect_fwd", apply_monarch_rect_fwd, 13}, {"monarch_rect_bwd", apply_monarch_rect_bwd, 18},
    {"monarch_cplx_fwd", apply_monarch_cplx_fwd, 12}, {"monarch_dense", apply_monarch_dense, 7},
    {"monarch_project", apply_monarch_project, 8},
};

typedef struct {
    PyObject_HEAD
    vectorcallfunc vectorcall;
    void *fn;
    apply_fn apply;
    char spec[MAX_ARGS];
    int n_spec, n_args;
    PyObject *name, *names, *types, *on_error, *stream_of;   /* types: (float32, bfloat16, int64) */
} Call;

static PyObject *s_is_cuda, *s_is_contiguous, *s_dtype, *s_data_ptr, *s_ptr, *s_nbytes, *s_cuda_stream;

static int to_u64(PyObject *o, uint64_t *out)
{
    PyObject *n = PyNumber_Index(o);
    if (n == NULL) return -1;
    *out = PyLong_AsUnsignedLongLongMask(n);
    Py_DECREF(n);
    return *out == (uint64_t)-1 && PyErr_Occurred() ? -1 : 0;
}

static int attr_u64(PyObject *o, PyObject *attr, uint64_t *out)
{
    PyObject *v = PyObject_GetAttr(o, attr);
    if (v == NULL) return -1;
    const int r = to_u64(v, out);
    Py_DECREF(v);
    return r;
}

/* 1 / 0 / -1 for a truth-valued attribute (call: method) */
static int flag_of(PyObject *o, PyObject *attr, int call)
{
    PyObject *v = call ? PyObject_CallMethodNoArgs(o, attr) : PyObject_GetAttr(o, attr);
    if (v == NULL) return -1;
    const int r = PyObject_IsTrue(v);
    Py_DECREF(v);
    return r;
}

static int tensor_ptr(Call *c, int k, PyObject *t, char kind, PyObject **storage, int *code, uint64_t *out)
{
    PyObject *name = PyTuple_GET_ITEM(c->names, k), *f32 = PyTuple_GET_ITEM(c->types, 0);
    if (t == Py_None && !(kind == 't' && *storage == NULL)) {
        *out = 0;
        return 0;
    }
    PyObject *dt = PyObject_GetAttr(t, s_dtype);
    if (dt == NULL) return -1;
    int r = flag_of(t, s_is_cuda, 0);
    if (r == 0) PyErr_Format(PyExc_ValueError, "%U must be a CUDA tensor", name);
    if (r > 0 && (r = flag_of(t, s_is_contiguous, 1)) == 0) PyErr_Format(PyExc_ValueError, "%U must be contiguous", name);
    if (r > 0) {
        PyObject *want = kind == 'f' ? f32 : kind == 'q' ? PyTuple_GET_ITEM(c->types, 2) : *storage;
        if (want == NULL) {
            if (dt == f32) *code = MONARCH_F32;
            else if (dt == PyTuple_GET_ITEM(c->types, 1)) *code = MONARCH_BF16;
            else { PyErr_Format(PyExc_TypeError, "unsupported tensor dtype %S", dt); r = 0; }
            *storage = *code == MONARCH_F32 ? f32 : PyTuple_GET_ITEM(c->types, 1);
        } else if (dt != want) {
            PyErr_Format(PyExc_TypeError, "%U must have dtype %S, got %S", name, want, dt);
            r = 0;
        }
    }
    Py_DECREF(dt);
    if (r <= 0) return -1;
    PyObject *p = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (p == NULL) return -1;
    r = to_u64(p, out);
    Py_DECREF(p);
    return r;
}

static int workspace_of(PyObject *w, uint64_t *ptr, uint64_t *bytes)
{
    if (PyTuple_Check(w)) {
        if (PyTuple_GET_SIZE(w) != 2) { PyErr_SetString(PyExc_ValueError, "workspace is a Workspace or (pointer, bytes)"); return -1; }
        return to_u64(PyTuple_GET_ITEM(w, 0), ptr) || to_u64(PyTuple_GET_ITEM(w, 1), bytes) ? -1 : 0;
    }
    return attr_u64(w, s_ptr, ptr) || attr_u64(w, s_nbytes, bytes) ? -1 : 0;
}

static PyObject *call_it(PyObject *self, PyObject *const *args, size_t nargsf, PyObject *kw)
{
    Call *c = (Call *)self;
    const Py_ssize_t n = PyVectorcall_NARGS(nargsf);
    if (n != c->n_args || (kw != NULL && PyTuple_GET_SIZE(kw) != 0))
        return PyErr_Format(PyExc_TypeError, "%U takes %d positional arguments (%zd given)", c->name, c->n_args, n);
    uint64_t a[MAX_ARGS], ignored;
    PyObject *storage = NULL;
    int code = 0, out = 0, in = 0, dtype_at = -1;
    for (int i = 0; i < c->n_spec; ++i) {
        const char kind = c->spec[i];
        PyObject *v = kind == 'D' ? NULL : args[in];
        switch (kind) {
            case 'D': dtype_at = out++; break;
            case 'i': if (to_u64(v, &a[out++])) return NULL; break;
            case 'w': if (workspace_of(v, &a[out], &a[out + 1])) return NULL; out += 2; break;
            case 'v':
                a[out] = 0;
                if (v != Py_None && workspace_of(v, &a[out], &ignored)) return NULL;
                ++out;
                break;
            case 's':
                if (v == Py_None) {
                    PyObject *s = PyObject_CallNoArgs(c->stream_of);
                    if (s == NULL) return NULL;
                    const int r = to_u64(s, &a[out]);
                    Py_DECREF(s);
                    if (r) return NULL;
                } else if (PyLong_Check(v) ? to_u64(v, &a[out]) : attr_u64(v, s_cuda_stream, &a[out])) {
                    return NULL;
                }
                ++out;
                break;
            default: if (tensor_ptr(c, in, v, kind, &storage, &code, &a[out++])) return NULL;
        }
        if (kind != 'D') ++in;
    }
    if (dtype_at >= 0) a[dtype_at] = (uint64_t)code;
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = c->apply(c->fn, a);
    Py_END_ALLOW_THREADS
    if (status != 0) return PyObject_CallFunction(c->on_error, "iO", status, c->name);
    Py_RETURN_NONE;
}

static PyObject *call_new(PyTypeObject *type, PyObject *args, PyObject *kw)
{
    PyObject *name, *names, *types, *on_error, *stream_of;
    unsigned long long fn;
    const char *spec;
    Py_ssize_t len;
    if (kw != NULL && PyDict_GET_SIZE(kw) != 0) { PyErr_SetString(PyExc_TypeError, "Call takes no keywords"); return NULL; }
    if (!PyArg_ParseTuple(args, "UKs#O!O!OO", &name, &fn, &spec, &len, &PyTuple_Type, &names, &PyTuple_Type, &types, &on_error, &stream_of))
        return NULL;
    if (len > MAX_ARGS || PyTuple_GET_SIZE(types) != 3) { PyErr_SetString(PyExc_ValueError, "bad spec"); return NULL; }
    int n_args = 0, params = 0;
    for (Py_ssize_t i = 0; i < len; ++i) {
        if (strchr("tfqiwvsD", spec[i]) == NULL) { PyErr_SetString(PyExc_ValueError, "bad spec"); return NULL; }
        n_args += spec[i] != 'D';
        params += spec[i] == 'w' ? 2 : 1;
    }
    apply_fn apply = NULL;
    for (size_t k = 0; k < sizeof(kCalls) / sizeof(kCalls[0]); ++k)
        if (PyUnicode_CompareWithASCIIString(name, kCalls[k].name) == 0 && kCalls[k].params == params) apply = kCalls[k].apply;
    if (apply == NULL || fn == 0 || PyTuple_GET_SIZE(names) != n_args) { PyErr_SetString(PyExc_ValueError, "spec does not fit the function"); return NULL; }
    Call *c = (Call *)type->tp_alloc(type, 0);
    if (c == NULL) return NULL;
    c->vectorcall = call_it;
    c->fn = (void *)(uintptr_t)fn;
    c->apply = apply;
    memcpy(c->spec, spec, (size_t)len);
    c->n_spec = (int)len;
    c->n_args = n_args;
    c->name = Py_NewRef(name);
    c->names = Py_NewRef(names);
    c->types = Py_NewRef(types);
    c->on_error = Py_NewRef(on_error);
    c->stream_of = Py_NewRef(stream_of);
    return (PyObject *)c;
}

static void call_dealloc(PyObject *self)
{
    Call *c = (Call *)self;
    Py_XDECREF(c->name);
    Py_XDECREF(c->names);
    Py_XDECREF(c->types);
    Py_XDECREF(c->on_error);
    Py_XDECREF(c->stream_of);
    Py_TYPE(self)->tp_free(self);
}

static PyTypeObject CallType = {
    PyVarObject_HEAD_INIT(NULL, 0)
    .tp_name = "paper_2204_00595_b200._pycalls.Call",
    .tp_basicsize = sizeof(Call),
    .tp_dealloc = call_dealloc,
    .tp_vectorcall_offset = offsetof(Call, vectorcall),
    .tp_call = PyVectorcall_Call,
    .tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL,
    .tp_new = call_new,
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycalls", "native argument marshalling", -1, NULL, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycalls(void)
{
    if (PyType_Ready(&CallType) < 0) return NULL;
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_ptr = PyUnicode_InternFromString("ptr");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    PyObject *m = PyModule_Create(&module);
    if (m == NULL || PyModule_AddObjectRef(m, "Call", (PyObject *)&CallType) < 0) return NULL;
    return m;
}
