/* The three calls of a decoding step, marshalled natively.  Small calls are bound by the host: spec_verify of
 * a small problem took 7.4 us with the tensor checks in Python and a ctypes call of 13 arguments, 4.9 so; in two kernels
 * 9.5 and 6.8.  Each function here
 * looks at its tensors (device, type, contiguity, shape) and calls the library through the address it was given; on
 * anything out of the ordinary it returns None and touches nothing: the caller then goes through its own checks, which know
 * what to say.  The interpreter's lock is released around the call. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "spec_b200.h"

typedef int (*verify_fn)(const int32_t *, const void *, int, int, int, int, int, int32_t *, int32_t *, int32_t *, void *,
                         size_t, void *);
typedef int (*next_ctx_fn)(const void *, const int32_t *, const int32_t *, int, int, int, int, void *, int32_t *, void *);
typedef int (*draft_fn)(spec_handle_t, const void *, const int32_t *, int, const int32_t *, int, int32_t *, float *, void *,
                        size_t, void *);
static verify_fn f_verify, f_verify_early;
static next_ctx_fn f_next_ctx;
static draft_fn f_draft;
static PyObject *t_i32, *t_bf16, *t_f32;   /* torch dtypes */
static PyObject *get_device, *get_raw_stream;   /* of the current device */
static PyObject *s_cuda_stream, *s_is_cuda, *s_dtype, *s_is_contiguous, *s_shape, *s_data_ptr, *s_numel, *s_get_device;

/* Contiguous CUDA tensor of `dtype` (null: bf16 or fp32, which is told in *bf16): fills `dim` with its nd sizes. */
static int look(PyObject *t, PyObject *dtype, int nd, long long *dim, uintptr_t *ptr, int *bf16) {
    int ok = 0;
    PyObject *o = PyObject_GetAttr(t, s_is_cuda);
    if (!o) return 0;
    ok = o == Py_True;
    Py_DECREF(o);
    if (!ok || !(o = PyObject_GetAttr(t, s_dtype))) return 0;
    ok = dtype ? o == dtype : (o == t_bf16 || o == t_f32);
    if (bf16) *bf16 = o == t_bf16;
    Py_DECREF(o);
    if (!ok || !(o = PyObject_CallMethodNoArgs(t, s_is_contiguous))) return 0;
    ok = o == Py_True;
    Py_DECREF(o);
    if (!ok || !(o = PyObject_GetAttr(t, s_shape))) return 0;
    ok = PyTuple_Check(o) && PyTuple_GET_SIZE(o) == nd;
    for (int i = 0; ok && i < nd; ++i) {
        dim[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(o, i));
        ok = dim[i] > 0 && dim[i] <= INT32_MAX;
    }
    Py_DECREF(o);
    if (!ok || !(o = PyObject_CallMethodNoArgs(t, s_data_ptr))) return 0;
    *ptr = (uintptr_t)PyLong_AsUnsignedLongLong(o);
    Py_DECREF(o);
    return !PyErr_Occurred();
}

static int number(PyObject *t, PyObject *method, long long *out) {
    PyObject *o = PyObject_CallMethodNoArgs(t, method);
    if (!o) return 0;
    *out = PyLong_AsLongLong(o);
    Py_DECREF(o);
    return !PyErr_Occurred();
}

static int bytes_of(PyObject *t, uintptr_t *ptr, long long *n) {   /* a workspace: its address and elements */
    PyObject *o = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!o) return 0;
    *ptr = (uintptr_t)PyLong_AsUnsignedLongLong(o);
    Py_DECREF(o);
    return !PyErr_Occurred() && number(t, s_numel, n);
}

static int vec_i32(PyObject *t, long long n, uintptr_t *ptr) {
    long long d[1];
    return look(t, t_i32, 1, d, ptr, NULL) && d[0] == n;
}

static int stream_of(PyObject *stream, uintptr_t *st) {   /* a stream object, or None: the current one */
    PyObject *o, *dev;
    if (stream != Py_None) {
        o = PyObject_GetAttr(stream, s_cuda_stream);
    } else {
        if (!(dev = PyObject_CallNoArgs(get_device))) return 0;
        o = PyObject_CallOneArg(get_raw_stream, dev);
        Py_DECREF(dev);
    }
    if (!o) return 0;
    *st = (uintptr_t)PyLong_AsUnsignedLongLong(o);
    Py_DECREF(o);
    return !PyErr_Occurred();
}

static PyObject *unusual(void) {
    PyErr_Clear();
    Py_RETURN_NONE;
}

/* verify(cand_tok, base_logits, accept_len, best_cand, next_tok, workspace, stream, early) -> status or None */
static PyObject *py_verify(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    long long c[3], l[4], wn;
    uintptr_t pc, pl, pa, pb, pn, pw, st;
    int bf16 = 0, status;
    if (n != 8 || !look(a[0], t_i32, 3, c, &pc, NULL) || !look(a[1], NULL, 4, l, &pl, &bf16) || l[0] != c[0] || l[1] != c[1] ||
        l[2] != c[2] + 1 || !vec_i32(a[2], c[0], &pa) || !vec_i32(a[3], c[0], &pb) || !vec_i32(a[4], c[0], &pn) ||
        !bytes_of(a[5], &pw, &wn) || !stream_of(a[6], &st))
        return unusual();
    const int early = PyObject_IsTrue(a[7]);
    if (early < 0) return unusual();
    const verify_fn f = early ? f_verify_early : f_verify;
    Py_BEGIN_ALLOW_THREADS
    status = f((const int32_t *)pc, (const void *)pl, bf16 ? SPEC_BF16 : SPEC_F32, (int)c[0], (int)c[1], (int)c[2], (int)l[3],
               (int32_t *)pa, (int32_t *)pb, (int32_t *)pn, (void *)pw, (size_t)wn, (void *)st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

/* next_ctx(base_state, best_cand, accept_len, ctx_state, err_workspace, stream) -> status or None */
static PyObject *py_next_ctx(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    long long s[4], x[2], on;
    PyObject *dev;
    uintptr_t ps, pb, pa, px, pe = 0, st;
    int status;
    if (n != 6 || !look(a[0], t_bf16, 4, s, &ps, NULL) || !vec_i32(a[1], s[0], &pb) || !vec_i32(a[2], s[0], &pa) ||
        !look(a[3], t_bf16, 2, x, &px, NULL) || x[0] != s[0] || x[1] != s[3] || s[2] < 2 ||
        !number(a[0], s_get_device, &on) || !(dev = PyObject_CallNoArgs(get_device)))
        return unusual();
    const int here = PyLong_AsLongLong(dev) == on;   /* the tensors' device is current */
    Py_DECREF(dev);
    if (!here || !stream_of(a[5], &st)) return unusual();
    if (a[4] != Py_None) {
        PyObject *o = PyObject_CallMethodNoArgs(a[4], s_data_ptr);
        if (!o) return unusual();
        pe = (uintptr_t)PyLong_AsUnsignedLongLong(o);
        Py_DECREF(o);
        if (PyErr_Occurred()) return unusual();
    }
    Py_BEGIN_ALLOW_THREADS
    status = f_next_ctx((const void *)ps, (const int32_t *)pb, (const int32_t *)pa, (int)s[0], (int)s[1], (int)s[2] - 1,
                        (int)s[3], (void *)px, (int32_t *)pe, (void *)st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

/* draft(handle, n_heads, d_base, ctx_state, last_tok, topk, K, cand_tok, cand_logp, workspace, stream) -> status or None */
static PyObject *py_draft(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    long long x[2], c[3], p[2], wn;
    uintptr_t h, px, pt, pc, pp, pw, st;
    int32_t topk[SPEC_MAX_HEADS];
    int status;
    if (n != 11 || !PyTuple_CheckExact(a[5])) return unusual();
    h = (uintptr_t)PyLong_AsUnsignedLongLong(a[0]);
    const long long heads = PyLong_AsLongLong(a[1]), d_base = PyLong_AsLongLong(a[2]), K = PyLong_AsLongLong(a[6]);
    if (PyErr_Occurred() || heads < 1 || heads > SPEC_MAX_HEADS || PyTuple_GET_SIZE(a[5]) != heads || K < 1 || K > INT32_MAX ||
        !look(a[3], t_bf16, 2, x, &px, NULL) || x[1] != d_base || !vec_i32(a[4], x[0], &pt) ||
        !look(a[7], t_i32, 3, c, &pc, NULL) || c[0] != x[0] || c[1] != K || c[2] != heads ||
        !look(a[8], t_f32, 2, p, &pp, NULL) || p[0] != x[0] || p[1] != K || !bytes_of(a[9], &pw, &wn))
        return unusual();
    for (int l = 0; l < heads; ++l) {
        const long long k = PyLong_AsLongLong(PyTuple_GET_ITEM(a[5], l));
        if (k < 0 || k > INT32_MAX) return unusual();
        topk[l] = (int32_t)k;
    }
    if (PyErr_Occurred() || !stream_of(a[10], &st)) return unusual();
    Py_BEGIN_ALLOW_THREADS
    status = f_draft((spec_handle_t)h, (const void *)px, (const int32_t *)pt, (int)x[0], topk, (int)K, (int32_t *)pc,
                     (float *)pp, (void *)pw, (size_t)wn, (void *)st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

/* bind(spec_verify, spec_verify_early, spec_next_ctx, spec_draft, int32, bfloat16, float32, get_device, get_raw_stream): addresses, dtypes
 * and the callables that tell the current device and its current stream */
static PyObject *py_bind(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    if (n != 9) {
        PyErr_SetString(PyExc_TypeError, "bind() takes four addresses, three dtypes and two callables");
        return NULL;
    }
    f_verify = (verify_fn)(uintptr_t)PyLong_AsUnsignedLongLong(a[0]);
    f_verify_early = (verify_fn)(uintptr_t)PyLong_AsUnsignedLongLong(a[1]);
    f_next_ctx = (next_ctx_fn)(uintptr_t)PyLong_AsUnsignedLongLong(a[2]);
    f_draft = (draft_fn)(uintptr_t)PyLong_AsUnsignedLongLong(a[3]);
    if (PyErr_Occurred()) return NULL;
    Py_XSETREF(t_i32, Py_NewRef(a[4]));
    Py_XSETREF(t_bf16, Py_NewRef(a[5]));
    Py_XSETREF(t_f32, Py_NewRef(a[6]));
    Py_XSETREF(get_device, Py_NewRef(a[7]));
    Py_XSETREF(get_raw_stream, Py_NewRef(a[8]));
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, NULL},
                                {"verify", (PyCFunction)(void (*)(void))py_verify, METH_FASTCALL, NULL},
                                {"next_ctx", (PyCFunction)(void (*)(void))py_next_ctx, METH_FASTCALL, NULL},
                                {"draft", (PyCFunction)(void (*)(void))py_draft, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void) {
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_shape = PyUnicode_InternFromString("shape");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_get_device = PyUnicode_InternFromString("get_device");
    return PyModule_Create(&module);
}
