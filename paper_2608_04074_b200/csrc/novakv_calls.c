/* Python entry to the per-step calls of libnovakv.so: takes tensors, forms the C arguments and calls the library without
 * the interpreter lock.
 *
 * A decode step of one short sequence runs 17 us on the device; marshalled through ctypes, its two calls took the host 27 us
 * (7 us a call for the foreign-function layer, another 2 for the stream object).  Nothing is computed or kept here.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stdint.h>

#include "novakv.h"

/* How a C argument is formed from Python argument `arg` (the context handle comes first and is not listed):
 *   L an integer   I int(x)   F float(x)   P data_ptr() of a tensor, 0 for None   0, 1 shape[0], shape[1]   n, m the same, 0 for None
 *   T 1 if its dtype is float32   B its size in bytes   S the current CUDA stream (no argument) */
typedef struct { char kind; signed char arg; } param;
#define MAX_ARGS 28

enum { ENCODE, ENCODE_SCALED, ENCODE_DEPLOYED, DECODE, DECODE_SCALED, DECODE_SINK, DECODE_BANDED, DECODE_DEPLOYED, BAND_APPEND,
       WINDOW, STEP_HOST, STEP_HOST_ASYNC, N_ENTRIES };

static const struct { const char* name; int n_args; param p[MAX_ARGS]; } entries[N_ENTRIES] = {
    /* layer, k_new, v_new, tok_seq, tok_pos, k_pages, v_pages, page_table, seq_lens */
    [ENCODE] = {"novakv_encode_append", 9,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'n', 1}, {'P', 5}, {'P', 6}, {'0', 5}, {'P', 7}, {'1', 7}, {'0', 7}, {'P', 8}, {'S', 0}}},
    /* ... k_pages, v_pages, k_scales, page_table, seq_lens */
    [ENCODE_SCALED] = {"novakv_encode_append_scaled", 10,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'n', 1}, {'P', 5}, {'P', 6}, {'P', 7}, {'0', 5}, {'P', 8}, {'1', 8}, {'0', 8}, {'P', 9}, {'S', 0}}},
    /* ... k_pages, v_pages, k_scales, v_meta, page_table, seq_lens */
    [ENCODE_DEPLOYED] = {"novakv_encode_append_deployed", 11,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'n', 1}, {'P', 5}, {'P', 6}, {'P', 7}, {'P', 8}, {'0', 5}, {'P', 9}, {'1', 9}, {'0', 9}, {'P', 10}, {'S', 0}}},
    /* layer, q, k_pages, v_pages, page_table, seq_lens, out, workspace, sm_scale */
    [DECODE] = {"novakv_decode_attention", 9,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'0', 2}, {'P', 4}, {'1', 4}, {'P', 5}, {'0', 1}, {'F', 8}, {'P', 6}, {'T', 6}, {'P', 7}, {'B', 7}, {'S', 0}}},
    /* layer, q, k_pages, v_pages, k_scales, page_table, seq_lens, out, workspace, sm_scale */
    [DECODE_SCALED] = {"novakv_decode_attention_scaled", 10,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'0', 2}, {'P', 5}, {'1', 5}, {'P', 6}, {'0', 1}, {'F', 9}, {'P', 7}, {'T', 7}, {'P', 8}, {'B', 8}, {'S', 0}}},
    /* layer, q, k_pages, v_pages, k_scales, sink_logits, page_table, seq_lens, out, workspace, sm_scale */
    [DECODE_SINK] = {"novakv_decode_attention_sink", 11,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'P', 5}, {'0', 2}, {'P', 6}, {'1', 6}, {'P', 7}, {'0', 1}, {'F', 10}, {'P', 8}, {'T', 8}, {'P', 9}, {'B', 9}, {'S', 0}}},
    /* layer, q, k_pages, v_pages, k_scales, sink_logits, page_table, quant_lens, band_k, band_v, n_sink, band_meta, out, workspace, sm_scale */
    [DECODE_BANDED] = {"novakv_decode_attention_banded", 15,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'P', 5}, {'0', 2}, {'P', 6}, {'1', 6}, {'P', 7}, {'P', 8}, {'P', 9}, {'1', 8}, {'I', 10}, {'P', 11},
         {'0', 1}, {'F', 14}, {'P', 12}, {'T', 12}, {'P', 13}, {'B', 13}, {'S', 0}}},
    /* layer, q, k_pages, v_pages, k_scales, v_meta, sink_logits, page_table, quant_lens, band_k, band_v, n_sink, band_meta, out, workspace, sm_scale */
    [DECODE_DEPLOYED] = {"novakv_decode_attention_deployed", 16,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'P', 5}, {'P', 6}, {'0', 2}, {'P', 7}, {'1', 7}, {'P', 8}, {'P', 9}, {'P', 10}, {'m', 9}, {'I', 11}, {'P', 12},
         {'0', 1}, {'F', 15}, {'P', 13}, {'T', 13}, {'P', 14}, {'B', 14}, {'S', 0}}},
    /* layer, k_new, v_new, band_k, band_v, n_sink, n_rec, block, band_meta, quant_lens, k_pages, v_pages, k_scales, v_meta, page_table, seq_lens, staging */
    [BAND_APPEND] = {"novakv_band_append", 17,
        {{'L', 0}, {'P', 1}, {'P', 2}, {'0', 1}, {'P', 3}, {'P', 4}, {'1', 3}, {'I', 5}, {'I', 6}, {'I', 7}, {'P', 8}, {'P', 9}, {'P', 10}, {'P', 11}, {'P', 12}, {'P', 13},
         {'0', 10}, {'P', 14}, {'1', 14}, {'P', 15}, {'P', 16}, {'B', 16}, {'S', 0}}},
    /* q, k_pages, v_pages, page_table, seq_lens, out, workspace, sm_scale, window */
    [WINDOW] = {"novakv_bf16_decode_attention", 9,
        {{'P', 0}, {'P', 1}, {'P', 2}, {'0', 1}, {'P', 3}, {'1', 3}, {'P', 4}, {'0', 0}, {'F', 7}, {'I', 8}, {'P', 5}, {'T', 5}, {'P', 6}, {'B', 6}, {'S', 0}}},
    /* layer, k_new, v_new, tok_seq, tok_pos, q, k_pages, v_pages, page_table, seq_lens, out, staging, workspace, sm_scale */
#define HOST_PARAMS {{'L', 0}, {'P', 1}, {'P', 2}, {'P', 3}, {'P', 4}, {'n', 1}, {'P', 5}, {'P', 6}, {'P', 7}, {'0', 6}, {'P', 8}, {'1', 8}, {'P', 9}, {'0', 5}, {'F', 13}, \
         {'P', 10}, {'P', 11}, {'B', 11}, {'P', 12}, {'B', 12}, {'S', 0}}
    [STEP_HOST] = {"novakv_step_host", 14, HOST_PARAMS},
    [STEP_HOST_ASYNC] = {"novakv_step_host_async", 14, HOST_PARAMS},
};

static PyObject *s_data_ptr, *s_shape, *s_dtype, *s_nbytes;
static PyObject *get_stream, *get_device, *float32;        /* given by setup() */

typedef struct {
    PyObject_HEAD
    vectorcallfunc vectorcall;
    int entry;
    void* fn;
} Entry;

/* shape[dim] as int(x.shape[dim]) gives it; -1 with an exception set */
static long long shape_of(PyObject* x, int dim) {
    PyObject* shape = PyObject_GetAttr(x, s_shape);
    if (!shape) return -1;
    PyObject* item = PySequence_GetItem(shape, dim);
    Py_DECREF(shape);
    if (!item) return -1;
    const long long v = PyLong_AsLongLong(item);
    Py_DECREF(item);
    return v;
}
static int as_int(PyObject* x, int exact, long long* v) {
    PyObject* n = exact ? PyNumber_Index(x) : PyNumber_Long(x);
    if (!n) return -1;
    *v = PyLong_AsLongLong(n);
    Py_DECREF(n);
    return *v == -1 && PyErr_Occurred() ? -1 : 0;
}
static int pointer_of(PyObject* x, unsigned long long* v) {
    if (x == Py_None) { *v = 0; return 0; }
    PyObject* n = PyObject_CallMethodNoArgs(x, s_data_ptr);
    if (!n) return -1;
    *v = PyLong_AsUnsignedLongLong(n);
    Py_DECREF(n);
    return PyErr_Occurred() ? -1 : 0;
}
static int current_stream(unsigned long long* v) {
    PyObject* dev = PyObject_CallNoArgs(get_device);
    if (!dev) return -1;
    PyObject* s = PyObject_CallOneArg(get_stream, dev);
    Py_DECREF(dev);
    if (!s) return -1;
    *v = PyLong_AsUnsignedLongLong(s);
    Py_DECREF(s);
    return PyErr_Occurred() ? -1 : 0;
}

static novakv_status call(int entry, void* fn, novakv_ctx* c, const long long* a, float f) {
#define I(i) ((int)a[i])
#define V(i) ((void*)(uintptr_t)a[i])
#define Z(i) ((size_t)a[i])
    switch (entry) {
        case ENCODE:
            return ((__typeof__(&novakv_encode_append))fn)(c, I(0), V(1), V(2), V(3), V(4), I(5), V(6), V(7), I(8), V(9), I(10), I(11), V(12), V(13));
        case ENCODE_SCALED:
            return ((__typeof__(&novakv_encode_append_scaled))fn)(c, I(0), V(1), V(2), V(3), V(4), I(5), V(6), V(7), V(8), I(9), V(10), I(11), I(12), V(13), V(14));
        case ENCODE_DEPLOYED:
            return ((__typeof__(&novakv_encode_append_deployed))fn)(c, I(0), V(1), V(2), V(3), V(4), I(5), V(6), V(7), V(8), V(9), I(10), V(11), I(12), I(13), V(14), V(15));
        case DECODE:
            return ((__typeof__(&novakv_decode_attention))fn)(c, I(0), V(1), V(2), V(3), I(4), V(5), I(6), V(7), I(8), f, V(10), I(11), V(12), Z(13), V(14));
        case DECODE_SCALED:
            return ((__typeof__(&novakv_decode_attention_scaled))fn)(c, I(0), V(1), V(2), V(3), V(4), I(5), V(6), I(7), V(8), I(9), f, V(11), I(12), V(13), Z(14), V(15));
        case DECODE_SINK:
            return ((__typeof__(&novakv_decode_attention_sink))fn)(c, I(0), V(1), V(2), V(3), V(4), V(5), I(6), V(7), I(8), V(9), I(10), f, V(12), I(13), V(14), Z(15), V(16));
        case DECODE_BANDED:
            return ((__typeof__(&novakv_decode_attention_banded))fn)(c, I(0), V(1), V(2), V(3), V(4), V(5), I(6), V(7), I(8), V(9), V(10), V(11), I(12), I(13), V(14), I(15), f,
                                                                     V(17), I(18), V(19), Z(20), V(21));
        case DECODE_DEPLOYED:
            return ((__typeof__(&novakv_decode_attention_deployed))fn)(c, I(0), V(1), V(2), V(3), V(4), V(5), V(6), I(7), V(8), I(9), V(10), V(11), V(12), I(13), I(14), V(15),
                                                                       I(16), f, V(18), I(19), V(20), Z(21), V(22));
        case BAND_APPEND:
            return ((__typeof__(&novakv_band_append))fn)(c, I(0), V(1), V(2), I(3), V(4), V(5), I(6), I(7), I(8), I(9), V(10), V(11), V(12), V(13), V(14), V(15), I(16), V(17),
                                                         I(18), V(19), V(20), Z(21), V(22));
        case WINDOW:
            return ((__typeof__(&novakv_bf16_decode_attention))fn)(c, V(0), V(1), V(2), I(3), V(4), I(5), V(6), I(7), f, I(9), V(10), I(11), V(12), Z(13), V(14));
        default:
            return ((__typeof__(&novakv_step_host))fn)(c, I(0), V(1), V(2), V(3), V(4), I(5), V(6), V(7), V(8), I(9), V(10), I(11), V(12), I(13), f, V(15), V(16), Z(17), V(18),
                                                       Z(19), V(20));
    }
#undef I
#undef V
#undef Z
}

/* entry(handle, arguments...) -> status */
static PyObject* entry_call(PyObject* self, PyObject* const* args, size_t nargsf, PyObject* kwnames) {
    Entry* e = (Entry*)self;
    const Py_ssize_t n = PyVectorcall_NARGS(nargsf);
    if (kwnames || n != entries[e->entry].n_args + 1) {
        PyErr_Format(PyExc_TypeError, "%s: a context and %d positional arguments", entries[e->entry].name, entries[e->entry].n_args);
        return NULL;
    }
    const unsigned long long ctx = args[0] == Py_None ? 0 : PyLong_AsUnsignedLongLong(args[0]);
    if (PyErr_Occurred()) return NULL;
    long long a[MAX_ARGS];
    float f = 0.f;
    const param* p = entries[e->entry].p;
    for (int i = 0; i < MAX_ARGS && p[i].kind; ++i) {
        PyObject* x = args[1 + p[i].arg];
        unsigned long long u = 0;
        a[i] = 0;
        switch (p[i].kind) {
            case 'L': if (as_int(x, 1, &a[i])) return NULL; break;
            case 'I': if (as_int(x, 0, &a[i])) return NULL; break;
            case 'F': f = (float)PyFloat_AsDouble(x); break;
            case 'P': if (pointer_of(x, &u)) return NULL; a[i] = (long long)u; break;
            case '0': a[i] = shape_of(x, 0); break;
            case '1': a[i] = shape_of(x, 1); break;
            case 'n': if (x != Py_None) a[i] = shape_of(x, 0); break;
            case 'm': if (x != Py_None) a[i] = shape_of(x, 1); break;
            case 'T': { PyObject* d = PyObject_GetAttr(x, s_dtype); a[i] = d == float32; Py_XDECREF(d); break; }
            case 'B': { PyObject* b = PyObject_GetAttr(x, s_nbytes); if (!b) return NULL; a[i] = PyLong_AsLongLong(b); Py_DECREF(b); break; }
            default: if (current_stream(&u)) return NULL; a[i] = (long long)u;
        }
        if (PyErr_Occurred()) return NULL;
    }
    novakv_status st;
    Py_BEGIN_ALLOW_THREADS
    st = call(e->entry, e->fn, (novakv_ctx*)(uintptr_t)ctx, a, f);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

static PyTypeObject EntryType = {
    PyVarObject_HEAD_INIT(NULL, 0).tp_name = "_novakv_calls.Entry",
    .tp_basicsize = sizeof(Entry),
    .tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL,
    .tp_vectorcall_offset = offsetof(Entry, vectorcall),
    .tp_call = PyVectorcall_Call,
};

/* setup(current stream of a device, current device, torch.float32): what the calls ask torch for */
static PyObject* setup(PyObject* self, PyObject* args) {
    PyObject *a, *b, *c;
    if (!PyArg_ParseTuple(args, "OOO", &a, &b, &c)) return NULL;
    Py_INCREF(a); Py_INCREF(b); Py_INCREF(c);
    Py_XSETREF(get_stream, a);
    Py_XSETREF(get_device, b);
    Py_XSETREF(float32, c);
    Py_RETURN_NONE;
}
/* bind(handle of the opened library) -> {name: entry} */
static PyObject* bind(PyObject* self, PyObject* handle) {
    void* h = PyLong_AsVoidPtr(handle);
    if (PyErr_Occurred()) return NULL;
    if (!get_stream) { PyErr_SetString(PyExc_RuntimeError, "setup() comes first"); return NULL; }
    PyObject* d = PyDict_New();
    for (int i = 0; d && i < N_ENTRIES; ++i) {
        void* fn = dlsym(h, entries[i].name);
        Entry* e = fn ? PyObject_New(Entry, &EntryType) : NULL;
        if (!fn) PyErr_Format(PyExc_RuntimeError, "the library lacks %s", entries[i].name);
        if (e) { e->vectorcall = entry_call; e->entry = i; e->fn = fn; }
        if (!e || PyDict_SetItemString(d, entries[i].name, (PyObject*)e)) Py_CLEAR(d);
        Py_XDECREF((PyObject*)e);
    }
    return d;
}

static PyMethodDef methods[] = {{"setup", setup, METH_VARARGS, NULL}, {"bind", bind, METH_O, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_novakv_calls", NULL, -1, methods};

PyMODINIT_FUNC PyInit__novakv_calls(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    if (!s_data_ptr || !s_shape || !s_dtype || !s_nbytes || PyType_Ready(&EntryType) < 0) return NULL;
    return PyModule_Create(&module);
}
