/*
 * pycalls.c -- argument conversion of the binding's per-step calls as a CPython extension.
 *
 * A decode step is a few dozen calls of a few microseconds of device work each; in a small step, or one layer per call,
 * the host is what the device waits for.  Converting a verification call's arguments in Python (a pointer per tensor, a
 * ctypes structure per cache, a ctypes call) took 6.1 us, here it takes 2.5 us: a float32 step of seven calls takes 73 us
 * instead of 89.  Nothing is kept between calls: every pointer and size is read from the objects of the call.  The
 * library is called without the interpreter lock, as ctypes does.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/specpv.h"

/* Argument kinds: G specpv_config structure, i int, P tensor or None, C cache (the binding's Cache, or anything else whose
 * desc() gives a specpv_paged_kv structure) -> specpv_paged_kv, W workspace tensor -> pointer and bytes, S stream or None (the
 * current one). */
typedef struct {
    const char *name, *kinds;
    int (*call)(const uint64_t *v);
} Spec;

enum { kMaxValues = 20, kMaxCaches = 2 };

#define P(i) ((void *)(uintptr_t)v[i])
#define I(i) ((int)v[i])
static int call_summaries(const uint64_t *v) {
    return specpv_update_block_summaries(P(0), I(1), I(2), P(3), P(4), I(5), P(6), P(7), P(8), (size_t)v[9], P(10));
}
static int call_scores(const uint64_t *v) {
    return specpv_score_blocks(P(0), I(1), I(2), P(3), P(4), I(5), P(6), P(7), P(8), P(9), P(10), P(11), (size_t)v[12], P(13));
}
static int call_select(const uint64_t *v) {
    return specpv_select_partial_kv(P(0), I(1), P(2), P(3), I(4), I(5), P(6), P(7), P(8), (size_t)v[9], P(10));
}
static int call_refresh(const uint64_t *v) {
    return specpv_refresh_partial(P(0), P(1), P(2), P(3), P(4), P(5), P(6), (size_t)v[7], P(8));
}
static int call_verify_partial(const uint64_t *v) {
    return specpv_verify_partial(P(0), I(1), I(2), P(3), P(4), P(5), P(6), P(7), I(8), P(9), P(10), P(11), P(12), (size_t)v[13], P(14));
}
static int call_verify_full(const uint64_t *v) {
    return specpv_verify_full(P(0), I(1), I(2), P(3), P(4), P(5), P(6), P(7), I(8), P(9), P(10), P(11), P(12), (size_t)v[13], P(14));
}
static int call_verify_static(const uint64_t *v) {
    return specpv_verify_partial_static(P(0), I(1), I(2), P(3), P(4), P(5), P(6), P(7), I(8), P(9), P(10), P(11), P(12), P(13));
}
static int call_verify_host(const uint64_t *v) {
    return specpv_verify_host(P(0), I(1), I(2), I(3), P(4), P(5), P(6), P(7), I(8), P(9), P(10), P(11), P(12), (size_t)v[13], P(14));
}
static int call_commit(const uint64_t *v) {
    return specpv_commit_accepted(P(0), I(1), I(2), P(3), P(4), I(5), P(6), P(7), I(8), P(9), P(10), P(11), P(12), (size_t)v[13], P(14));
}
static int call_qkv(const uint64_t *v) {
    return specpv_qkv_rope(P(0), I(1), I(2), P(3), I(4), P(5), P(6), I(7), I(8), P(9), P(10), P(11), P(12), (size_t)v[13], P(14));
}
static int call_o_proj(const uint64_t *v) {
    return specpv_o_proj(P(0), I(1), I(2), P(3), P(4), I(5), P(6), I(7), I(8), P(9), P(10), (size_t)v[11], P(12));
}

/* set once by init(): torch.Tensor, the binding's converters, torch's current device and stream, the binding's Cache and
 * ctypes' structures and simple values */
static PyObject *tensor_type, *convert, *convert_stream, *get_device, *raw_stream, *cache_type, *structure_type, *simple_type;
static PyObject *s_data_ptr, *s_is_contiguous, *s_size, *s_numel, *s_k_pool, *s_v_pool, *s_block_table, *s_seq_lens, *s_max_seq_len, *s_desc, *s_value;
static PyObject *zero, *one;

static int take_u64(PyObject *number, uint64_t *out) {  /* steals the reference */
    if (!number) return -1;
    *out = number == Py_None ? 0 : (uint64_t)PyLong_AsUnsignedLongLongMask(number);
    Py_DECREF(number);
    return PyErr_Occurred() ? -1 : 0;
}

static int take_int(PyObject *number, int32_t *out) {  /* steals the reference */
    if (!number) return -1;
    *out = (int32_t)PyLong_AsLong(number);
    Py_DECREF(number);
    return PyErr_Occurred() ? -1 : 0;
}

static int data_ptr(PyObject *tensor, uint64_t *out) { return take_u64(PyObject_CallMethodNoArgs(tensor, s_data_ptr), out); }

static int pointer_of(PyObject *arg, uint64_t *out) {
    if (arg == Py_None) {
        *out = 0;
        return 0;
    }
    if (!PyObject_TypeCheck(arg, (PyTypeObject *)tensor_type)) return take_u64(PyObject_CallOneArg(convert, arg), out);
    PyObject *r = PyObject_CallMethodNoArgs(arg, s_is_contiguous);
    if (!r) return -1;
    const int ok = r == Py_True;
    Py_DECREF(r);
    if (!ok) {
        PyErr_SetString(PyExc_AssertionError, "tensors passed to the C ABI must be contiguous");
        return -1;
    }
    return data_ptr(arg, out);
}

/* The memory of a ctypes structure of at least `size` bytes; it lives as long as the structure does. */
static int structure_of(PyObject *arg, size_t size, const void **out) {
    Py_buffer view;
    if (!PyObject_TypeCheck(arg, (PyTypeObject *)structure_type)) {
        PyErr_Format(PyExc_TypeError, "a ctypes structure was expected, not %.80s", Py_TYPE(arg)->tp_name);
        return -1;
    }
    if (PyObject_GetBuffer(arg, &view, PyBUF_SIMPLE)) return -1;
    const int ok = view.len >= (Py_ssize_t)size;
    *out = view.buf;
    PyBuffer_Release(&view);
    if (!ok) PyErr_Format(PyExc_TypeError, "%.80s is too small", Py_TYPE(arg)->tp_name);
    return ok ? 0 : -1;
}

/* Read straight from the attributes of a Cache; another type's own desc() is asked. */
static int cache_of(PyObject *cache, specpv_paged_kv *kv) {
    if ((PyObject *)Py_TYPE(cache) != cache_type) {
        const void *desc = NULL;
        PyObject *d = PyObject_CallMethodNoArgs(cache, s_desc);
        const int bad = !d || structure_of(d, sizeof *kv, &desc);
        if (!bad) *kv = *(const specpv_paged_kv *)desc;
        Py_XDECREF(d);
        return bad ? -1 : 0;
    }
    PyObject *k = PyObject_GetAttr(cache, s_k_pool), *v = PyObject_GetAttr(cache, s_v_pool);
    PyObject *table = PyObject_GetAttr(cache, s_block_table), *lens = PyObject_GetAttr(cache, s_seq_lens);
    PyObject *limit = PyObject_GetAttr(cache, s_max_seq_len);
    uint64_t p[4];
    int st = k && v && table && lens && limit ? 0 : -1;
    if (!st) st = data_ptr(k, &p[0]) || data_ptr(v, &p[1]) || data_ptr(table, &p[2]) || data_ptr(lens, &p[3]) ||
                  take_int(PyObject_CallMethodOneArg(table, s_size, zero), &kv->batch) ||
                  take_int(PyObject_CallMethodOneArg(table, s_size, one), &kv->max_blocks) ||
                  take_int(PyObject_CallMethodOneArg(k, s_size, one), &kv->n_pages) ||
                  take_int(PyNumber_Long(limit), &kv->max_seq_len) ? -1 : 0;
    if (!st) {
        kv->k_pool = (void *)(uintptr_t)p[0];
        kv->v_pool = (void *)(uintptr_t)p[1];
        kv->block_table = (const int32_t *)(uintptr_t)p[2];
        kv->seq_lens = (const int32_t *)(uintptr_t)p[3];
    }
    Py_XDECREF(k);
    Py_XDECREF(v);
    Py_XDECREF(table);
    Py_XDECREF(lens);
    Py_XDECREF(limit);
    return st;
}

static int config_of(PyObject *arg, uint64_t *out) {
    const void *cfg = NULL;
    if (structure_of(arg, sizeof(specpv_config), &cfg)) return -1;
    *out = (uint64_t)(uintptr_t)cfg;
    return 0;
}

static int int_of(PyObject *arg, uint64_t *out) {
    PyObject *value = NULL;  /* of a c_int and the like */
    if (PyObject_TypeCheck(arg, (PyTypeObject *)simple_type)) {
        if (!(value = PyObject_GetAttr(arg, s_value))) return -1;
        arg = value;
    }
    const long x = PyLong_AsLong(arg);
    Py_XDECREF(value);
    *out = (uint64_t)x;
    return x == -1 && PyErr_Occurred() ? -1 : 0;
}

static int stream_of(PyObject *arg, uint64_t *out) {
    if (arg != Py_None || raw_stream == Py_None) return take_u64(PyObject_CallOneArg(convert_stream, arg), out);
    PyObject *device = PyObject_CallNoArgs(get_device);
    if (!device) return -1;
    PyObject *handle = PyObject_CallOneArg(raw_stream, device);
    Py_DECREF(device);
    return take_u64(handle, out);
}

static PyObject *invoke(const Spec *spec, PyObject *const *args, Py_ssize_t n) {
    uint64_t v[kMaxValues];
    specpv_paged_kv caches[kMaxCaches];
    int n_v = 0, n_caches = 0;
    if (n != (Py_ssize_t)strlen(spec->kinds) || !tensor_type) {
        PyErr_Format(PyExc_TypeError, "%s: wrong number of arguments", spec->name);
        return NULL;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        int st = 0;
        switch (spec->kinds[i]) {
            case 'i': st = int_of(args[i], &v[n_v]); break;
            case 'G': st = config_of(args[i], &v[n_v]); break;
            case 'C':
                st = cache_of(args[i], &caches[n_caches]);
                v[n_v] = (uint64_t)(uintptr_t)&caches[n_caches++];
                break;
            case 'S': st = stream_of(args[i], &v[n_v]); break;
            case 'W':
                st = pointer_of(args[i], &v[n_v]);
                if (!st) st = take_u64(PyObject_CallMethodNoArgs(args[i], s_numel), &v[++n_v]);
                break;
            default: st = pointer_of(args[i], &v[n_v]); break;
        }
        if (st) return NULL;
        ++n_v;
    }
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = spec->call(v);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

#define CALLS(X)                                                        \
    X(specpv_update_block_summaries, "GiiCPiPPWS", call_summaries)      \
    X(specpv_score_blocks, "GiiPPiPPPCPWS", call_scores)                \
    X(specpv_select_partial_kv, "GiPPiiPPWS", call_select)              \
    X(specpv_refresh_partial, "GCPPCPWS", call_refresh)                 \
    X(specpv_verify_partial, "GiiPPPPPiCPPWS", call_verify_partial)     \
    X(specpv_verify_full, "GiiPPPPPiCPPWS", call_verify_full)           \
    X(specpv_verify_partial_static, "GiiPPPPPiCPPPS", call_verify_static) \
    X(specpv_verify_host, "GiiiPPPPiCPPWS", call_verify_host)           \
    X(specpv_commit_accepted, "GiiPPiPPiCPPWS", call_commit)            \
    X(specpv_qkv_rope, "GiiPiPPiiPPPWS", call_qkv)                      \
    X(specpv_o_proj, "GiiPPiPiiPWS", call_o_proj)

#define WRAPPER(name, kinds, call)                                                       \
    static PyObject *py_##name(PyObject *self, PyObject *const *args, Py_ssize_t n) {    \
        static const Spec spec = {#name, kinds, call};                                   \
        (void)self;                                                                      \
        return invoke(&spec, args, n);                                                   \
    }
CALLS(WRAPPER)

static PyObject *py_init(PyObject *self, PyObject *const *args, Py_ssize_t n) {
    (void)self;
    PyObject **slots[] = {&tensor_type, &convert, &convert_stream, &get_device, &raw_stream, &cache_type, &structure_type, &simple_type};
    if (n != 8 || !PyType_Check(args[0]) || !PyType_Check(args[6]) || !PyType_Check(args[7])) {
        PyErr_SetString(PyExc_TypeError, "init takes eight objects, the first and the last two of them types");
        return NULL;
    }
    for (int i = 0; i < 8; ++i) {
        Py_INCREF(args[i]);
        Py_XSETREF(*slots[i], args[i]);
    }
    Py_RETURN_NONE;
}

#define METHOD(name, kinds, call) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL},
static PyMethodDef methods[] = {CALLS(METHOD){"init", (PyCFunction)(void (*)(void))py_init, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "pycalls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit_pycalls(void) {
    struct {
        PyObject **slot;
        const char *text;
    } names[] = {{&s_data_ptr, "data_ptr"},       {&s_is_contiguous, "is_contiguous"}, {&s_size, "size"},
                 {&s_numel, "numel"},             {&s_k_pool, "k_pool"},               {&s_v_pool, "v_pool"},
                 {&s_block_table, "block_table"}, {&s_seq_lens, "seq_lens"},           {&s_max_seq_len, "max_seq_len"},
                 {&s_desc, "desc"},               {&s_value, "value"}};
    for (size_t i = 0; i < sizeof(names) / sizeof(names[0]); ++i)
        if (!(*names[i].slot = PyUnicode_InternFromString(names[i].text))) return NULL;
    if (!(zero = PyLong_FromLong(0)) || !(one = PyLong_FromLong(1))) return NULL;
    return PyModule_Create(&module);
}
