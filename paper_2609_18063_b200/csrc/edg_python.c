/* CPython entry points of the calls a decoder makes per layer and token: argument marshalling in C.
 *
 * ctypes and the Python around it took most of a call's host time: a layer-step of the small layer 12.7 us, now 5.9 (on the GPU it is
 * under 9); the sigmoid-group gate 10.9, now 5.2 (200 calls issued one after the other).  Semantics are those of the Python helpers of binding.py
 * -- a buffer is None, an int, a torch tensor or a numpy array, contiguous; a stream None (torch's current one), an int or an
 * object with cuda_stream -- and the interpreter lock is released around the call, as ctypes does.  The addresses of the
 * library's functions and the Python helpers for the unusual cases come from binding.py (init). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>
#include <string.h>

#include "edg_moe.h"

static struct {
    __typeof__(&prerouter_topk) prerouter_topk;
    __typeof__(&prerouter_topk_tokens) prerouter_topk_tokens;
    __typeof__(&softmax_topk_rows) softmax_topk_rows;
    __typeof__(&sigmoid_group_topk_rows) sigmoid_group_topk_rows;
    __typeof__(&prerouter_mlp_topk) prerouter_mlp_topk;
    __typeof__(&moe_expert_ffn_int4_lora) moe_expert_ffn_int4_lora;
    __typeof__(&moe_layer_decode) moe_layer_decode;
    __typeof__(&moe_layer_decode_dependent) moe_layer_decode_dependent;
    __typeof__(&edg_stack_decode_token) edg_stack_decode_token;
    __typeof__(&edg_next_hidden_state) edg_next_hidden_state;
} F;
static PyObject *py_ptr, *py_stream, *py_check;               /* binding._ptr, binding._stream, binding._check */
static PyObject *t_desc, *t_lora, *t_int, *t_size;            /* binding.LayerDesc, binding.Lora, ctypes.c_int32, ctypes.c_size_t */
static PyObject *raw_stream, *raw_device;                     /* torch's current raw stream of a device, current device; or NULL */
static PyObject *s_data_ptr, *s_is_contiguous, *s_cuda_stream, *s_value, *s_numel, *s_element_size;

/* integer result of a Python callable's object; consumes it */
static int take_u64(PyObject* o, uint64_t* v) {
    if (o == NULL) return -1;
    if (o == Py_None) { *v = 0; Py_DECREF(o); return 0; }
    *v = PyLong_AsUnsignedLongLongMask(o);
    Py_DECREF(o);
    return (*v == (uint64_t)-1 && PyErr_Occurred()) ? -1 : 0;
}

static int as_ptr(PyObject* o, void** p) {
    uint64_t v = 0;
    *p = NULL;
    if (o == Py_None) return 0;
    if (PyLong_Check(o)) {
        v = PyLong_AsUnsignedLongLongMask(o);
        if (v == (uint64_t)-1 && PyErr_Occurred()) return -1;
        *p = (void*)(uintptr_t)v;
        return 0;
    }
    PyObject* c = PyObject_CallMethodNoArgs(o, s_is_contiguous);
    if (c == NULL) {                                          /* a numpy array, or nothing with an address: the Python helper knows */
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
        PyErr_Clear();
        if (take_u64(PyObject_CallOneArg(py_ptr, o), &v) != 0) return -1;
        *p = (void*)(uintptr_t)v;
        return 0;
    }
    const int yes = PyObject_IsTrue(c);
    Py_DECREF(c);
    if (yes < 0) return -1;
    if (!yes) {
        PyErr_SetString(PyExc_ValueError, "tensor must be contiguous");
        return -1;
    }
    if (take_u64(PyObject_CallMethodNoArgs(o, s_data_ptr), &v) != 0) return -1;
    *p = (void*)(uintptr_t)v;
    return 0;
}

static int as_stream(PyObject* o, void** p) {
    uint64_t v = 0;
    *p = NULL;
    if (o == Py_None) {
        if (raw_stream != NULL) {
            PyObject* dev = PyObject_CallNoArgs(raw_device);
            if (dev == NULL) return -1;
            PyObject* st = PyObject_CallOneArg(raw_stream, dev);
            Py_DECREF(dev);
            if (take_u64(st, &v) != 0) return -1;
        } else if (take_u64(PyObject_CallOneArg(py_stream, o), &v) != 0) return -1;
    } else if (PyLong_Check(o)) {
        v = PyLong_AsUnsignedLongLongMask(o);
        if (v == (uint64_t)-1 && PyErr_Occurred()) return -1;
    } else if (take_u64(PyObject_GetAttr(o, s_cuda_stream), &v) != 0) return -1;
    *p = (void*)(uintptr_t)v;
    return 0;
}

/* what ctypes takes for an integer argument: anything with an index, cut to the type's bits, or an instance of the type itself */
static int as_bits(PyObject* o, PyObject* type, uint64_t* v) {
    PyObject* i;
    if (!PyLong_Check(o) && PyObject_TypeCheck(o, (PyTypeObject*)type)) i = PyObject_GetAttr(o, s_value);
    else i = PyNumber_Index(o);
    if (i == NULL) return -1;
    *v = PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return *v == (uint64_t)-1 && PyErr_Occurred() ? -1 : 0;
}

static int as_int(PyObject* o, int32_t* p) {
    uint64_t v = 0;
    const int rc = as_bits(o, t_int, &v);
    *p = (int32_t)(uint32_t)v;
    return rc;
}

static int as_float(PyObject* o, float* p) {
    PyObject* f = PyNumber_Float(o);
    if (f == NULL) return -1;
    *p = (float)PyFloat_AsDouble(f);
    Py_DECREF(f);
    return PyErr_Occurred() ? -1 : 0;
}

/* a ctypes structure of the given type (or, for `opt`, None), by value */
static int as_struct(PyObject* o, PyObject* type, void* dst, size_t bytes, int opt, int* present) {
    if (present != NULL) *present = o != Py_None;
    if (opt && o == Py_None) return 0;
    if (!PyObject_TypeCheck(o, (PyTypeObject*)type)) {
        PyErr_Format(PyExc_TypeError, "%s expected instead of %s", ((PyTypeObject*)type)->tp_name, Py_TYPE(o)->tp_name);
        return -1;
    }
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return -1;
    const int ok = (size_t)b.len >= bytes;                    /* (more for a subclass with fields of its own) */
    if (ok) memcpy(dst, b.buf, bytes);
    PyBuffer_Release(&b);
    if (!ok) PyErr_SetString(PyExc_TypeError, "not the expected structure");
    return ok ? 0 : -1;
}

/* a ctypes.c_void_p, or None */
static int as_handle(PyObject* o, void** p) {
    uint64_t v = 0;
    *p = NULL;
    if (o == Py_None) return 0;
    if (take_u64(PyObject_GetAttr(o, s_value), &v) != 0) return -1;
    *p = (void*)(uintptr_t)v;
    return 0;
}

/* workspace_bytes, or None: all of the workspace */
static int as_bytes(PyObject* o, PyObject* workspace, size_t* n) {
    uint64_t a, b;
    if (o != Py_None) {
        if (as_bits(o, t_size, &a) != 0) return -1;
        *n = (size_t)a;
        return 0;
    }
    if (take_u64(PyObject_CallMethodNoArgs(workspace, s_numel), &a) != 0 ||
        take_u64(PyObject_CallMethodNoArgs(workspace, s_element_size), &b) != 0)
        return -1;
    *n = (size_t)(a * b);
    return 0;
}

static PyObject* done(int32_t rc, const char* what) {
    if (rc != 0) return PyObject_CallFunction(py_check, "is", (int)rc, what);      /* raises EdgError */
    Py_RETURN_NONE;
}

#define ARGS(name, n)                                                                                     \
    if (nargs != (n)) return PyErr_Format(PyExc_TypeError, name ": %zd arguments instead of %d", nargs, n)
#define CALL(expr) Py_BEGIN_ALLOW_THREADS rc = expr; Py_END_ALLOW_THREADS

static PyObject* py_prerouter_topk(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("prerouter_topk", 9);
    edg_layer_desc d;
    void *W, *s, *inds, *gates, *logits, *mirror, *st;
    int32_t n, rc;
    if (as_struct(a[0], t_desc, &d, sizeof d, 0, NULL) || as_ptr(a[1], &W) || as_ptr(a[2], &s) || as_int(a[3], &n) || as_ptr(a[4], &inds) ||
        as_ptr(a[5], &gates) || as_ptr(a[6], &logits) || as_ptr(a[7], &mirror) || as_stream(a[8], &st))
        return NULL;
    CALL(F.prerouter_topk(&d, W, s, n, inds, gates, logits, mirror, st))
    return done(rc, "prerouter_topk");
}

static PyObject* py_prerouter_topk_tokens(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("prerouter_topk_tokens", 8);
    edg_layer_desc d;
    void *W, *s, *inds, *gates, *logits, *st;
    int32_t T, rc;
    if (as_struct(a[0], t_desc, &d, sizeof d, 0, NULL) || as_ptr(a[1], &W) || as_ptr(a[2], &s) || as_int(a[3], &T) || as_ptr(a[4], &inds) ||
        as_ptr(a[5], &gates) || as_ptr(a[6], &logits) || as_stream(a[7], &st))
        return NULL;
    CALL(F.prerouter_topk_tokens(&d, W, s, T, inds, gates, logits, st))
    return done(rc, "prerouter_topk_tokens");
}

static PyObject* py_softmax_topk_rows(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("softmax_topk_rows", 6);
    edg_layer_desc d;
    void *logits, *inds, *gates, *st;
    int32_t T, rc;
    if (as_struct(a[0], t_desc, &d, sizeof d, 0, NULL) || as_ptr(a[1], &logits) || as_int(a[2], &T) || as_ptr(a[3], &inds) || as_ptr(a[4], &gates) ||
        as_stream(a[5], &st))
        return NULL;
    CALL(F.softmax_topk_rows(&d, logits, T, inds, gates, st))
    return done(rc, "softmax_topk_rows");
}

static PyObject* py_sigmoid_group_topk_rows(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("sigmoid_group_topk_rows", 11);
    void *logits, *bias, *inds, *gates, *st;
    int32_t T, E, K, groups, keep, rc;
    float scale;
    if (as_ptr(a[0], &logits) || as_int(a[1], &T) || as_int(a[2], &E) || as_int(a[3], &K) || as_int(a[4], &groups) || as_int(a[5], &keep) ||
        as_float(a[6], &scale) || as_ptr(a[7], &bias) || as_ptr(a[8], &inds) || as_ptr(a[9], &gates) || as_stream(a[10], &st))
        return NULL;
    CALL(F.sigmoid_group_topk_rows(logits, T, E, K, groups, keep, scale, bias, inds, gates, st))
    return done(rc, "sigmoid_group_topk_rows");
}

static PyObject* py_prerouter_mlp_topk(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("prerouter_mlp_topk", 15);
    edg_layer_desc d;
    edg_mlp_head h;
    void *W1, *b1, *W2, *b2, *Wr, *s, *cur, *prev, *inds, *gates, *logits, *st;
    int32_t width, n, rc;
    if (as_struct(a[0], t_desc, &d, sizeof d, 0, NULL) || as_ptr(a[1], &W1) || as_ptr(a[2], &b1) || as_ptr(a[3], &W2) || as_ptr(a[4], &b2) ||
        as_ptr(a[5], &Wr) || as_int(a[6], &width) || as_ptr(a[7], &s) || as_ptr(a[8], &cur) || as_ptr(a[9], &prev) || as_int(a[10], &n) ||
        as_ptr(a[11], &inds) || as_ptr(a[12], &gates) || as_ptr(a[13], &logits) || as_stream(a[14], &st))
        return NULL;
    memset(&h, 0, sizeof h);
    h.W1 = W1; h.b1 = b1; h.W2 = W2; h.b2 = b2; h.W_res = Wr; h.width = width;
    CALL(F.prerouter_mlp_topk(&d, &h, s, cur, prev, n, inds, gates, logits, st))
    return done(rc, "prerouter_mlp_topk");
}

static PyObject* py_moe_expert_ffn(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("moe_expert_ffn_int4_lora", 13);
    edg_layer_desc d;
    edg_lora lo;
    void *pool, *table, *slots, *experts, *gates, *x, *y, *ws, *st;
    size_t bytes;
    int32_t T, rc;
    int has;
    if (as_struct(a[0], t_desc, &d, sizeof d, 0, NULL) || as_ptr(a[1], &pool) || as_ptr(a[2], &table) || as_int(a[3], &T) || as_ptr(a[4], &slots) ||
        as_ptr(a[5], &experts) || as_ptr(a[6], &gates) || as_ptr(a[7], &x) || as_struct(a[8], t_lora, &lo, sizeof lo, 1, &has) || as_ptr(a[9], &y) ||
        as_ptr(a[10], &ws) || as_bytes(a[11], a[10], &bytes) || as_stream(a[12], &st))
        return NULL;
    CALL(F.moe_expert_ffn_int4_lora(&d, pool, table, T, slots, experts, gates, x, has ? &lo : NULL, y, ws, bytes, st))
    return done(rc, "moe_expert_ffn_int4_lora");
}

static PyObject* py_moe_layer_decode(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("moe_layer_decode", 14);
    void *h, *x, *ic, *gc, *W, *in, *gn, *ln, *mirror, *y, *ws, *st;
    size_t bytes;
    int32_t layer, rc;
    if (as_handle(a[0], &h) || as_int(a[1], &layer) || as_ptr(a[2], &x) || as_ptr(a[3], &ic) || as_ptr(a[4], &gc) || as_ptr(a[5], &W) ||
        as_ptr(a[6], &in) || as_ptr(a[7], &gn) || as_ptr(a[8], &ln) || as_ptr(a[9], &mirror) || as_ptr(a[10], &y) || as_ptr(a[11], &ws) ||
        as_bytes(a[12], a[11], &bytes) || as_stream(a[13], &st))
        return NULL;
    CALL(F.moe_layer_decode(h, layer, x, ic, gc, W, in, gn, ln, mirror, y, ws, bytes, st))
    return done(rc, "moe_layer_decode");
}

static PyObject* py_moe_layer_decode_dependent(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("moe_layer_decode_dependent", 16);
    void *h, *x, *ic, *gc, *W, *in, *gn, *ln, *mirror, *y, *xn, *ws, *st;
    size_t bytes;
    int32_t layer, rc;
    float eps;
    if (as_handle(a[0], &h) || as_int(a[1], &layer) || as_ptr(a[2], &x) || as_ptr(a[3], &ic) || as_ptr(a[4], &gc) || as_ptr(a[5], &W) ||
        as_ptr(a[6], &in) || as_ptr(a[7], &gn) || as_ptr(a[8], &ln) || as_ptr(a[9], &mirror) || as_ptr(a[10], &y) || as_ptr(a[11], &xn) ||
        as_float(a[12], &eps) || as_ptr(a[13], &ws) || as_bytes(a[14], a[13], &bytes) || as_stream(a[15], &st))
        return NULL;
    CALL(F.moe_layer_decode_dependent(h, layer, x, ic, gc, W, in, gn, ln, mirror, y, xn, eps, ws, bytes, st))
    return done(rc, "moe_layer_decode_dependent");
}

static PyObject* py_stack_decode_token(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("stack_decode_token", 15);
    void *h, *x, *ic, *gc, *W, *in, *gn, *ln, *mc, *mn, *y, *ws, *st;
    size_t bytes;
    int32_t rc, miss = 0;
    int prefetch;
    if (as_handle(a[0], &h) || as_ptr(a[1], &x) || as_ptr(a[2], &ic) || as_ptr(a[3], &gc) || as_ptr(a[4], &W) || as_ptr(a[5], &in) ||
        as_ptr(a[6], &gn) || as_ptr(a[7], &ln) || as_ptr(a[8], &mc) || as_ptr(a[9], &mn) || as_ptr(a[10], &y) || as_ptr(a[11], &ws) ||
        as_bytes(a[12], a[11], &bytes) || as_stream(a[13], &st) || (prefetch = PyObject_IsTrue(a[14])) < 0)
        return NULL;
    CALL(F.edg_stack_decode_token(h, x, ic, gc, W, in, gn, ln, mc, mn, y, ws, bytes, st, prefetch, &miss))
    if (rc != 0) return done(rc, "edg_stack_decode_token");
    return PyLong_FromLong(miss);
}

static PyObject* py_next_hidden_state(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("next_hidden_state", 6);
    edg_layer_desc d;
    void *x, *y, *xn, *st;
    float eps;
    int32_t rc;
    if (as_struct(a[0], t_desc, &d, sizeof d, 0, NULL) || as_ptr(a[1], &x) || as_ptr(a[2], &y) || as_ptr(a[3], &xn) || as_float(a[4], &eps) ||
        as_stream(a[5], &st))
        return NULL;
    CALL(F.edg_next_hidden_state(&d, x, y, xn, eps, st))
    return done(rc, "edg_next_hidden_state");
}

/* init(addresses: dict name -> int, _ptr, _stream, _check, LayerDesc, Lora, c_int32, c_size_t) */
static PyObject* py_init(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("init", 8);
#define TAKE(name)                                                                                        \
    do {                                                                                                  \
        PyObject* v = PyDict_GetItemString(a[0], #name);                                                  \
        if (v == NULL) return PyErr_Format(PyExc_KeyError, "%s", #name);                                  \
        F.name = (__typeof__(F.name))PyLong_AsVoidPtr(v);                                                 \
        if (PyErr_Occurred()) return NULL;                                                                \
    } while (0)
    TAKE(prerouter_topk); TAKE(prerouter_topk_tokens); TAKE(softmax_topk_rows); TAKE(sigmoid_group_topk_rows); TAKE(prerouter_mlp_topk);
    TAKE(moe_expert_ffn_int4_lora); TAKE(moe_layer_decode); TAKE(moe_layer_decode_dependent); TAKE(edg_stack_decode_token);
    TAKE(edg_next_hidden_state);
    py_ptr = Py_NewRef(a[1]);
    py_stream = Py_NewRef(a[2]);
    py_check = Py_NewRef(a[3]);
    for (int i = 4; i < 8; ++i)
        if (!PyType_Check(a[i])) return PyErr_Format(PyExc_TypeError, "init: argument %d is no type", i);
    t_desc = Py_NewRef(a[4]);
    t_lora = Py_NewRef(a[5]);
    t_int = Py_NewRef(a[6]);
    t_size = Py_NewRef(a[7]);
    Py_RETURN_NONE;
}

/* streams(current device, raw current stream of a device): from here on the current stream is asked for without torch.cuda's wrappers */
static PyObject* py_streams(PyObject* self, PyObject* const* a, Py_ssize_t nargs) {
    ARGS("streams", 2);
    if (raw_stream != NULL) Py_RETURN_NONE;
    raw_device = Py_NewRef(a[0]);
    raw_stream = Py_NewRef(a[1]);
    Py_RETURN_NONE;
}

#define M(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    M("init", py_init), M("streams", py_streams), M("prerouter_topk", py_prerouter_topk), M("prerouter_topk_tokens", py_prerouter_topk_tokens),
    M("softmax_topk_rows", py_softmax_topk_rows), M("sigmoid_group_topk_rows", py_sigmoid_group_topk_rows),
    M("prerouter_mlp_topk", py_prerouter_mlp_topk), M("moe_expert_ffn_int4_lora", py_moe_expert_ffn), M("moe_layer_decode", py_moe_layer_decode),
    M("moe_layer_decode_dependent", py_moe_layer_decode_dependent), M("stack_decode_token", py_stack_decode_token),
    M("next_hidden_state", py_next_hidden_state), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_edgcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__edgcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_value = PyUnicode_InternFromString("value");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    return PyModule_Create(&module);
}
