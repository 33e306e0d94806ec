/* The library's calls as functions of a CPython module, for the binding (binding.py): the same names without the prefix,
 * the same arguments, the return code as an int.  A shape is the address of a pevlm_shape_t; a pointer is None, an address
 * or anything with a data_ptr() (a torch tensor).  A call costs about a microsecond less per six arguments than through
 * ctypes, which is what a decode step or a tiny layer is made of.  The interpreter lock is released during the call. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/pevlm.h"

static PyObject* g_data_ptr; /* interned "data_ptr" */

/* Both do nothing once an argument was bad: its exception is pending. */
static void* as_pointer(PyObject* o, int* bad) {
    if (*bad || o == Py_None) return NULL;
    if (PyLong_Check(o)) {
        void* p = PyLong_AsVoidPtr(o);
        if (!p && PyErr_Occurred()) *bad = 1;
        return p;
    }
    PyObject* v = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!v) {
        *bad = 1;
        return NULL;
    }
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (!p && PyErr_Occurred()) *bad = 1;
    return p;
}

static int64_t as_int(PyObject* o, int* bad) {
    if (*bad) return 0;
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) *bad = 1;
    return v;
}

#define P(i) as_pointer(a[i], &bad)
#define I(i) as_int(a[i], &bad)
/* BEGIN(name, number of arguments) ...decode the arguments... END(the call) */
#define BEGIN(name, count)                                                                                        \
    static PyObject* py_##name(PyObject* self, PyObject* const* a, Py_ssize_t n) {                                \
        (void)self;                                                                                               \
        if (n != (count)) return PyErr_Format(PyExc_TypeError, #name " takes %d arguments, got %zd", (count), n); \
        int bad = 0, rc;                                                                                          \
        const pevlm_shape_t* s = (const pevlm_shape_t*)P(0);
#define END(...)                       \
        if (bad) return NULL;          \
        Py_BEGIN_ALLOW_THREADS         \
        rc = (__VA_ARGS__);            \
        Py_END_ALLOW_THREADS           \
        return PyLong_FromLong(rc);    \
    }

BEGIN(rope_qk, 9)
    void *qi = P(1), *ki = P(2), *qo = P(3), *ko = P(4); int64_t first = I(5), tokens = I(6); void *pos = P(7), *st = P(8);
END(pevlm_rope_qk(s, qi, ki, qo, ko, first, tokens, (const int32_t*)pos, st))

BEGIN(rope_qkv, 11)
    void *qi = P(1), *ki = P(2), *vi = P(3), *qo = P(4), *ko = P(5), *vo = P(6); int64_t first = I(7), tokens = I(8);
    void *pos = P(9), *st = P(10);
END(pevlm_rope_qkv(s, qi, ki, vi, qo, ko, vo, first, tokens, (const int32_t*)pos, st))

BEGIN(rope_qk_mrope, 11)
    void *qi = P(1), *ki = P(2), *qo = P(3), *ko = P(4); int64_t tokens = I(5); void* pos = P(6);
    int32_t sec[3] = {(int32_t)I(7), (int32_t)I(8), (int32_t)I(9)}; void* st = P(10);
END(pevlm_rope_qk_mrope(s, qi, ki, qo, ko, tokens, (const int32_t*)pos, sec, st))

BEGIN(parallel_prefill_attn, 9)
    void *q = P(1), *k = P(2), *v = P(3), *o = P(4), *lse = P(5), *ws = P(6); int64_t wb = I(7); void* st = P(8);
END(pevlm_parallel_prefill_attn(s, q, k, v, o, (float*)lse, ws, (size_t)wb, st))

BEGIN(block_attn, 11)
    void *q = P(1), *k = P(2), *v = P(3); int64_t row = I(4), rows = I(5); void *o = P(6), *lse = P(7), *ws = P(8);
    int64_t wb = I(9); void* st = P(10);
END(pevlm_block_attn(s, q, k, v, row, rows, o, (float*)lse, ws, (size_t)wb, st))

BEGIN(assemble_kv, 8)
    void *kv = P(1), *vv = P(2), *kq = P(3), *vq = P(4), *kc = P(5), *vc = P(6), *st = P(7);
END(pevlm_assemble_kv(s, kv, vv, kq, vq, kc, vc, st))

BEGIN(query_attn, 9)
    void *q = P(1), *k = P(2), *v = P(3), *o = P(4), *lse = P(5), *ws = P(6); int64_t wb = I(7); void* st = P(8);
END(pevlm_query_attn(s, q, k, v, o, (float*)lse, ws, (size_t)wb, st))

BEGIN(query_attn_noalloc, 7)
    void *q = P(1), *k = P(2), *v = P(3), *o = P(4), *lse = P(5), *st = P(6);
END(pevlm_query_attn_noalloc(s, q, k, v, o, (float*)lse, st))

BEGIN(layer_forward, 18)
    int64_t last = I(1); void *q = P(2), *k = P(3), *v = P(4), *qv = P(5), *qq = P(6), *kc = P(7), *vc = P(8), *ov = P(9),
    *lv = P(10), *oq = P(11), *lq = P(12), *wp = P(13); int64_t wpb = I(14); void* wq = P(15);
    int64_t wqb = I(16); void* st = P(17);
END(pevlm_layer_forward(s, (int32_t)last, q, k, v, qv, qq, kc, vc, ov, (float*)lv, oq, (float*)lq, wp, (size_t)wpb, wq, (size_t)wqb, st))

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {METHOD(rope_qk), METHOD(rope_qkv), METHOD(rope_qk_mrope), METHOD(parallel_prefill_attn),
                                METHOD(block_attn), METHOD(assemble_kv), METHOD(query_attn), METHOD(query_attn_noalloc),
                                METHOD(layer_forward), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pevlm_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pevlm_call(void) {
    g_data_ptr = PyUnicode_InternFromString("data_ptr");
    if (!g_data_ptr) return NULL;
    return PyModule_Create(&module);
}
