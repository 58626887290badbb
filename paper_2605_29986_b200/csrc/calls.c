/* The per-step calls of include/cfgzip.h as Python functions: argument marshalling only. A decode step of a small batch
 * takes 5 us on the GPU, and handing it eighteen arguments through ctypes took 3 to 6 us of the caller's time; this takes
 * under 1. Device buffers are objects with data_ptr() (torch tensors), host buffers those or numpy arrays; raw integer
 * addresses are accepted everywhere and None is a null pointer. A stream is None, an integer, or an object with cuda_stream.
 * The functions come in through bind() by address, so that this module and the ctypes handle share one library. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "cfgzip.h"

enum { MAX_ARGS = 24 };

/* One call: the names of its arguments, their kinds ('p' address, 's' stream, 'i' integer, 'f' number) and how many have to
 * be given; what is left out is a null pointer, the null stream or 0 (CFGZIP_AUTO). */
typedef struct {
    const char* name;
    const char* kinds;
    int required;
    const char* args[MAX_ARGS];
    void* fn;
} Call;

typedef union {
    void* p;
    int64_t i;
    float f;
} Value;

static PyObject *s_data_ptr, *s_ctypes, *s_data, *s_cuda_stream;
static PyObject* g_raise; /* raises the package's error for (status, call) */

static int as_address(PyObject* o, void** out) {
    PyObject* v;
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return PyErr_Occurred() ? -1 : 0;
    }
    v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) {
        PyObject* c;
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
        PyErr_Clear();
        c = PyObject_GetAttr(o, s_ctypes);
        if (!c) {
            PyErr_Clear();
            PyErr_Format(PyExc_TypeError, "cannot take the address of %R", (PyObject*)Py_TYPE(o));
            return -1;
        }
        v = PyObject_GetAttr(c, s_data);
        Py_DECREF(c);
        if (!v) return -1;
    }
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static int as_stream(PyObject* o, void** out) {
    PyObject* v;
    if (o == Py_None || PyLong_Check(o)) return as_address(o, out);
    v = PyObject_GetAttr(o, s_cuda_stream);
    if (!v) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

/* Positional and keyword arguments in the order of the call, converted. */
static int take(const Call* c, PyObject* const* args, Py_ssize_t n, PyObject* kwnames, Value* v) {
    PyObject* given[MAX_ARGS] = {NULL};
    const int count = (int)strlen(c->kinds);
    Py_ssize_t k, n_kw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    int i;
    if (!c->fn) {
        PyErr_SetString(PyExc_RuntimeError, "the CFGzip library is not loaded");
        return -1;
    }
    if (n > count) {
        PyErr_Format(PyExc_TypeError, "%s() takes %d arguments (%zd given)", c->name, count, n);
        return -1;
    }
    for (i = 0; i < n; ++i) given[i] = args[i];
    for (k = 0; k < n_kw; ++k) {
        PyObject* name = PyTuple_GET_ITEM(kwnames, k);
        for (i = 0; i < count; ++i)
            if (PyUnicode_CompareWithASCIIString(name, c->args[i]) == 0) break;
        if (i == count || given[i]) {
            PyErr_Format(PyExc_TypeError, "%s() got an unexpected or repeated argument '%U'", c->name, name);
            return -1;
        }
        given[i] = args[n + k];
    }
    for (i = 0; i < count; ++i) {
        if (!given[i]) {
            if (i < c->required) {
                PyErr_Format(PyExc_TypeError, "%s() is missing the argument '%s'", c->name, c->args[i]);
                return -1;
            }
            v[i].i = 0;
            continue;
        }
        switch (c->kinds[i]) {
            case 'p':
                if (as_address(given[i], &v[i].p) != 0) return -1;
                break;
            case 's':
                if (as_stream(given[i], &v[i].p) != 0) return -1;
                break;
            case 'f': {
                const double d = PyFloat_AsDouble(given[i]);
                if (d == -1.0 && PyErr_Occurred()) return -1;
                v[i].f = (float)d;
                break;
            }
            default:
                v[i].i = PyLong_AsLongLong(given[i]);
                if (v[i].i == -1 && PyErr_Occurred()) return -1;
        }
    }
    return 0;
}

static PyObject* done(const Call* c, int status) {
    if (status == CFGZIP_OK) Py_RETURN_NONE;
    return PyObject_CallFunction(g_raise, "is", status, c->name); /* NULL: it raised */
}

enum { EXPAND_MASK, MASK_LOGITS, FUSED, SAMPLE, SAMPLE_FILTERED, MULTI_MASK, PLAN_ROWS, MAP_TOKENS, STEP_HOST, N_CALLS };

#define STEP_ARGS                                                                                                     \
    "ctx", "part0", "row_part", "class_mask", "class_stride_words", "logits", "dtype", "row_stride_elems", "B", "vocab_mask", \
        "vocab_stride_words"

static Call calls[N_CALLS] = {
    {"cfgzip_expand_mask", "pippipiiis", 8,
     {"ctx", "part0", "row_part", "class_mask", "class_stride_words", "vocab_mask", "vocab_stride_words", "B", "mode", "stream"},
     NULL},
    {"cfgzip_mask_logits", "ppiiiipis", 8,
     {"ctx", "logits", "dtype", "row_stride_elems", "B", "V", "vocab_mask", "vocab_stride_words", "stream"}, NULL},
    {"cfgzip_masked_logsoftmax_argmax", "pippipiiipipppppis", 12,
     {STEP_ARGS, "argmax", "rep", "logp_argmax", "lse", "logp_full", "mode", "stream"}, NULL},
    {"cfgzip_masked_sample", "pippipiiipipfppppis", 14,
     {STEP_ARGS, "u", "inv_temperature", "token", "rep", "logp_token", "lse", "mode", "stream"}, NULL},
    {"cfgzip_masked_sample_filtered", "pippipiiipipfifppppis", 16,
     {STEP_ARGS, "u", "inv_temperature", "top_k", "top_p", "token", "rep", "logp_token", "lse", "mode", "stream"}, NULL},
    {"cfgzip_multi_mask_logsoftmax_argmax", "pipiipiiipipppps", 12,
     {"ctx", "part0", "class_masks", "class_stride_words", "masks_per_row", "logits", "dtype", "row_stride_elems", "B",
      "vocab_masks", "vocab_stride_words", "argmax", "rep", "logp_argmax", "lse", "stream"}, NULL},
    {"cfgzip_plan_rows", "pipis", 4, {"ctx", "part0", "row_part", "B", "stream"}, NULL},
    {"cfgzip_map_tokens", "pipppis", 6, {"ctx", "part0", "row_part", "tokens", "reps", "B", "stream"}, NULL},
    {"cfgzip_decode_step_host", "pippipiippppppis", 8,
     {"ctx", "part0", "row_part_host", "class_mask_host", "class_stride_words", "logits_host", "dtype", "B", "masked_logits",
      "vocab_mask_host", "argmax", "rep", "logp_argmax", "lse", "mode", "stream"}, NULL},
};

#define I(k) ((int32_t)v[k].i)
#define L(k) (v[k].i)
#define P(k) (v[k].p)
#define F(k) (v[k].f)
#define CTX ((cfgzip_ctx*)v[0].p)
#define CALL(index, function, ...)                                                                       \
    Value v[MAX_ARGS];                                                                               \
    int status;                                                                                      \
    (void)self;                                                                                      \
    if (take(&calls[index], args, n, kw, v) != 0) return NULL;                                       \
    Py_BEGIN_ALLOW_THREADS                                                                           \
    status = ((__typeof__(&function))calls[index].fn)(__VA_ARGS__);                                                   \
    Py_END_ALLOW_THREADS                                                                             \
    return done(&calls[index], status)


static PyObject* py_cfgzip_expand_mask(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(EXPAND_MASK, cfgzip_expand_mask, CTX, I(1), P(2), P(3), L(4), P(5), L(6), I(7), I(8), P(9));
}

static PyObject* py_cfgzip_mask_logits(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(MASK_LOGITS, cfgzip_mask_logits, CTX, P(1), I(2), L(3), I(4), I(5), P(6), L(7), P(8));
}

static PyObject* py_cfgzip_masked_logsoftmax_argmax(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(FUSED, cfgzip_masked_logsoftmax_argmax, CTX, I(1), P(2), P(3), L(4), P(5), I(6), L(7), I(8), P(9), L(10),
         P(11), P(12), P(13), P(14), P(15), I(16), P(17));
}

static PyObject* py_cfgzip_masked_sample(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(SAMPLE, cfgzip_masked_sample, CTX, I(1), P(2), P(3), L(4), P(5), I(6), L(7), I(8), P(9), L(10), P(11), F(12),
         P(13), P(14), P(15), P(16), I(17), P(18));
}

static PyObject* py_cfgzip_masked_sample_filtered(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(SAMPLE_FILTERED, cfgzip_masked_sample_filtered, CTX, I(1), P(2), P(3), L(4), P(5), I(6), L(7), I(8), P(9),
         L(10), P(11), F(12), I(13), F(14), P(15), P(16), P(17), P(18), I(19), P(20));
}

static PyObject* py_cfgzip_multi_mask_logsoftmax_argmax(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(MULTI_MASK, cfgzip_multi_mask_logsoftmax_argmax, CTX, I(1), P(2), L(3), I(4), P(5), I(6), L(7), I(8), P(9),
         L(10), P(11), P(12), P(13), P(14), P(15));
}

static PyObject* py_cfgzip_plan_rows(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(PLAN_ROWS, cfgzip_plan_rows, CTX, I(1), P(2), I(3), P(4));
}

static PyObject* py_cfgzip_map_tokens(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(MAP_TOKENS, cfgzip_map_tokens, CTX, I(1), P(2), P(3), P(4), I(5), P(6));
}

static PyObject* py_cfgzip_decode_step_host(PyObject* self, PyObject* const* args, Py_ssize_t n, PyObject* kw) {
    CALL(STEP_HOST, cfgzip_decode_step_host, CTX, I(1), P(2), P(3), L(4), P(5), I(6), I(7), P(8), P(9), P(10), P(11),
         P(12), P(13), I(14), P(15));
}

/* bind(addresses by name, raise): where the functions are, and what to call with (status, call) when one fails */
static PyObject* py_bind(PyObject* self, PyObject* args) {
    PyObject *addresses, *raise;
    int i;
    (void)self;
    if (!PyArg_ParseTuple(args, "O!O", &PyDict_Type, &addresses, &raise)) return NULL;
    for (i = 0; i < N_CALLS; ++i) {
        PyObject* a = PyDict_GetItemString(addresses, calls[i].name);
        if (!a) {
            PyErr_Format(PyExc_KeyError, "%s", calls[i].name);
            return NULL;
        }
        calls[i].fn = PyLong_AsVoidPtr(a);
        if (PyErr_Occurred()) return NULL;
    }
    Py_INCREF(raise);
    Py_XSETREF(g_raise, raise);
    Py_RETURN_NONE;
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL | METH_KEYWORDS, NULL}
static PyMethodDef methods[] = {
    METHOD(cfgzip_expand_mask),
    METHOD(cfgzip_mask_logits),
    METHOD(cfgzip_masked_logsoftmax_argmax),
    METHOD(cfgzip_masked_sample),
    METHOD(cfgzip_masked_sample_filtered),
    METHOD(cfgzip_multi_mask_logsoftmax_argmax),
    METHOD(cfgzip_plan_rows),
    METHOD(cfgzip_map_tokens),
    METHOD(cfgzip_decode_step_host),
    {"bind", py_bind, METH_VARARGS, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_ctypes = PyUnicode_InternFromString("ctypes");
    s_data = PyUnicode_InternFromString("data");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
