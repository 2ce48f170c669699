/* CPython entry points of the calls a training loop makes: argument marshalling only, in C because the loop's small
 * calls are bound by it (an advantage scan of 5 us on the device took 10 us to enqueue through ctypes: 3 for the
 * current stream, 2.5 for pointers and conversions, 1.5 for the foreign call).  Every function takes the arguments of
 * the Python function of the same name positionally, the stream last; pointers are torch tensors, C-contiguous numpy
 * arrays, integers or None, and contexts integers, c_void_p or None: nothing else that has an address of its own (a
 * numpy scalar, bytes) is taken for one.  A non-zero status raises the exception type handed to init(). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include "hts.h"

static PyObject *g_error;                              /* HtsError(status, what) */
static PyObject *g_raw_stream, *g_get_device;          /* torch._C._cuda_getCurrentRawStream, _cuda_getDevice */
static PyTypeObject *g_ndarray, *g_void_p;             /* numpy.ndarray, ctypes.c_void_p */
static PyObject *g_argument_error;                     /* ctypes.ArgumentError */
static PyObject *s_data_ptr, *s_is_contiguous, *s_cuda_stream, *s_value;
static PyObject *s_weights[12];
static const char *const kWeights[12] = {"conv1_w", "conv1_b", "conv2_w", "conv2_b", "conv3_w", "conv3_b",
                                         "fc_w", "fc_b", "pi_w", "pi_b", "v_w", "v_b"};

static int not_contiguous(void)
{
    PyErr_Clear();
    PyErr_SetString(PyExc_AssertionError, "tensors and arrays must be contiguous");
    return 0;
}

static int int_ptr(PyObject *l, void **out)            /* takes the reference */
{
    if (!l) return 0;
    *out = PyLong_AsVoidPtr(l);
    Py_DECREF(l);
    return !PyErr_Occurred();
}

/* address of a tensor, array, integer or None; 0 with an exception set on failure */
static int to_ptr(PyObject *x, void **out)
{
    if (x == Py_None) { *out = NULL; return 1; }
    if (PyLong_Check(x)) return int_ptr(Py_NewRef(x), out);
    if (PyObject_TypeCheck(x, g_ndarray)) {
        Py_buffer b;
        if (PyObject_GetBuffer(x, &b, PyBUF_C_CONTIGUOUS) != 0) return not_contiguous();
        *out = b.buf;
        PyBuffer_Release(&b);                          /* the caller keeps the object for the duration of the call */
        return 1;
    }
    PyObject *c = PyObject_CallMethodNoArgs(x, s_is_contiguous);
    if (!c) return 0;
    const int ok = PyObject_IsTrue(c);
    Py_DECREF(c);
    if (ok <= 0) return ok < 0 ? 0 : not_contiguous();
    return int_ptr(PyObject_CallMethodNoArgs(x, s_data_ptr), out);
}

/* a context: what hts_policy_create returned */
static int to_ctx(PyObject *x, void **out)
{
    if (x == Py_None) { *out = NULL; return 1; }
    if (PyLong_Check(x)) return int_ptr(Py_NewRef(x), out);
    if (PyObject_TypeCheck(x, g_void_p)) {
        PyObject *v = PyObject_GetAttr(x, s_value);
        if (v != Py_None) return int_ptr(v, out);
        Py_DECREF(v);
        *out = NULL;
        return 1;
    }
    PyErr_SetString(g_argument_error, "argument 1: a context is an integer, c_void_p or None");
    return 0;
}

static int to_u64(PyObject *x, uint64_t *out)          /* int(x), wrapped to 64 bits */
{
    PyObject *l = PyLong_Check(x) ? Py_NewRef(x) : PyNumber_Long(x);
    if (!l) return 0;
    *out = PyLong_AsUnsignedLongLongMask(l);
    Py_DECREF(l);
    return !PyErr_Occurred();
}
static int to_i32(PyObject *x, int32_t *out)
{
    uint64_t v;
    if (!to_u64(x, &v)) return 0;
    *out = (int32_t)v;
    return 1;
}
static int to_i64(PyObject *x, int64_t *out) { return to_u64(x, (uint64_t *)out); }
static int to_f32(PyObject *x, float *out)
{
    PyObject *f = PyFloat_Check(x) ? Py_NewRef(x) : PyNumber_Float(x);       /* float(x) */
    if (!f) return 0;
    *out = (float)PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return 1;
}

/* None: torch's current stream; else an integer handle or an object with .cuda_stream */
static int to_stream(PyObject *x, void **out)
{
    PyObject *h;
    if (x == Py_None) {
        if (!g_raw_stream) {
            PyObject *torch = PyImport_ImportModule("torch"), *cuda = torch ? PyObject_GetAttrString(torch, "cuda") : NULL;
            PyObject *st = cuda ? PyObject_CallMethod(cuda, "current_stream", NULL) : NULL;   /* initialises CUDA, or says why not */
            PyObject *c = st ? PyObject_GetAttrString(torch, "_C") : NULL;
            PyObject *raw = c ? PyObject_GetAttrString(c, "_cuda_getCurrentRawStream") : NULL;
            PyObject *dev = raw ? PyObject_GetAttrString(c, "_cuda_getDevice") : NULL;
            h = st ? PyObject_GetAttr(st, s_cuda_stream) : NULL;
            if (dev) { g_get_device = dev; g_raw_stream = raw; }
            else { Py_XDECREF(raw); if (h) PyErr_Clear(); }
            Py_XDECREF(torch); Py_XDECREF(cuda); Py_XDECREF(st); Py_XDECREF(c);
        } else {
            PyObject *d = PyObject_CallNoArgs(g_get_device);
            h = d ? PyObject_CallOneArg(g_raw_stream, d) : NULL;
            Py_XDECREF(d);
        }
    } else
        h = PyLong_Check(x) ? Py_NewRef(x) : PyObject_GetAttr(x, s_cuda_stream);
    if (!h) return 0;
    *out = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

static int weights_of(PyObject *map, void **p)
{
    for (int i = 0; i < 12; ++i) {
        PyObject *v = PyObject_GetItem(map, s_weights[i]);
        if (!v) return 0;
        const int ok = to_ptr(v, p + i);
        Py_DECREF(v);                                  /* the mapping keeps it */
        if (!ok) return 0;
    }
    return 1;
}

static PyObject *done(hts_status st, const char *what)
{
    if (st == HTS_OK) Py_RETURN_NONE;
    PyObject *e = PyObject_CallFunction(g_error, "is", (int)st, what);
    if (e) { PyErr_SetObject(g_error, e); Py_DECREF(e); }
    return NULL;
}

#define ARGS(count) \
    if (nargs != (count)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return NULL; }
#define PTR(name, i) void *name; if (!to_ptr(a[i], &name)) return NULL
#define CTX() void *ctx; if (!to_ctx(a[0], &ctx)) return NULL
#define I32(name, i) int32_t name; if (!to_i32(a[i], &name)) return NULL
#define I64(name, i) int64_t name; if (!to_i64(a[i], &name)) return NULL
#define U64(name, i) uint64_t name; if (!to_u64(a[i], &name)) return NULL
#define F32(name, i) float name; if (!to_f32(a[i], &name)) return NULL
#define STREAM(i) void *stream; if (!to_stream(a[i], &stream)) return NULL
#define CALL(expr, what) \
    hts_status st; Py_BEGIN_ALLOW_THREADS st = (expr); Py_END_ALLOW_THREADS return done(st, what)
#define FN(name) static PyObject *name(PyObject *self, PyObject *const *a, Py_ssize_t nargs)

static PyObject *step(PyObject *const *a, Py_ssize_t nargs, int host)
{
    ARGS(13);
    CTX(); PTR(obs, 1); PTR(ids, 2); PTR(tpe, 3); I32(t, 4); U64(seed, 5); I32(n, 6);
    PTR(act, 7); PTR(logp, 8); PTR(val, 9); PTR(ent, 10); PTR(logits, 11); STREAM(12);
    CALL((host ? hts_policy_step_host : hts_policy_step)(ctx, obs, ids, tpe, t, seed, n, act, logp, val, ent, logits, stream),
         host ? "hts_policy_step_host" : "hts_policy_step");
}
FN(policy_step) { (void)self; return step(a, nargs, 0); }
FN(policy_step_host) { (void)self; return step(a, nargs, 1); }
FN(policy_step_indexed)
{
    (void)self;
    ARGS(14);
    CTX(); PTR(buf, 1); I32(pool, 2); PTR(slots, 3); PTR(ids, 4); PTR(tpe, 5); I32(t, 6); U64(seed, 7); I32(n, 8);
    PTR(act, 9); PTR(logp, 10); PTR(val, 11); PTR(ent, 12); STREAM(13);
    CALL(hts_policy_step_indexed(ctx, buf, pool, slots, ids, tpe, t, seed, n, act, logp, val, ent, stream), "hts_policy_step_indexed");
}
FN(policy_evaluate)
{
    (void)self;
    ARGS(9);
    CTX(); PTR(obs, 1); PTR(act, 2); I32(n, 3); PTR(logp, 4); PTR(val, 5); PTR(ent, 6); PTR(logits, 7); STREAM(8);
    CALL(hts_policy_evaluate(ctx, obs, act, n, logp, val, ent, logits, stream), "hts_policy_evaluate");
}
FN(policy_gradient)
{
    (void)self;
    ARGS(12);
    hts_grads g;
    CTX(); PTR(obs, 1); PTR(act, 2); PTR(adv, 3); PTR(ret, 4); PTR(old, 5); F32(vc, 6); F32(ec, 7); F32(clip, 8); I32(n, 9);
    if (!weights_of(a[10], (void **)&g)) return NULL;
    STREAM(11);
    CALL(hts_policy_gradient(ctx, obs, act, adv, ret, old, vc, ec, clip, n, &g, stream), "hts_policy_gradient");
}
FN(policy_load_weights)
{
    (void)self;
    ARGS(3);
    hts_weights w;
    CTX();
    if (!weights_of(a[1], (void **)&w)) return NULL;
    STREAM(2);
    CALL(hts_policy_load_weights(ctx, &w, stream), "hts_policy_load_weights");
}
FN(a2c_terms)
{
    (void)self;
    ARGS(7);
    PTR(logp, 0); PTR(val, 1); PTR(ent, 2); PTR(ret, 3); I64(count, 4); PTR(out, 5); STREAM(6);
    CALL(hts_a2c_terms(logp, val, ent, ret, count, out, stream), "hts_a2c_terms");
}
FN(ppo_terms)
{
    (void)self;
    ARGS(11);
    PTR(ln, 0); PTR(lo, 1); PTR(val, 2); PTR(ent, 3); PTR(adv, 4); PTR(ret, 5); I64(count, 6); F32(clip, 7);
    const int norm = PyObject_IsTrue(a[8]);
    if (norm < 0) return NULL;
    PTR(out, 9); STREAM(10);
    CALL(hts_ppo_terms(ln, lo, val, ent, adv, ret, count, clip, norm, out, stream), "hts_ppo_terms");
}
FN(delayed_update)
{
    (void)self;
    ARGS(9);
    PTR(theta, 0); PTR(grad, 1); PTR(sq, 2); I64(count, 3); F32(lr, 4); F32(alpha, 5); F32(eps, 6); PTR(half, 7); STREAM(8);
    CALL(hts_delayed_update(theta, grad, sq, count, lr, alpha, eps, half, stream), "hts_delayed_update");
}
static PyObject *scan(PyObject *const *a, Py_ssize_t nargs, int host)
{
    ARGS(11);
    PTR(r, 0); PTR(v, 1); PTR(d, 2); PTR(b, 3); F32(gamma, 4); F32(lambda, 5); I32(T, 6); I32(N, 7); PTR(adv, 8); PTR(ret, 9); STREAM(10);
    CALL((host ? hts_gae_host : hts_gae)(r, v, d, b, gamma, lambda, T, N, adv, ret, stream), host ? "hts_gae_host" : "hts_gae");
}
FN(gae) { (void)self; return scan(a, nargs, 0); }
FN(gae_host) { (void)self; return scan(a, nargs, 1); }
FN(vtrace)
{
    (void)self;
    ARGS(14);
    PTR(lr, 0); PTR(r, 1); PTR(v, 2); PTR(d, 3); PTR(b, 4); F32(gamma, 5); F32(lambda, 6); F32(rho, 7); F32(c, 8); I32(T, 9); I32(N, 10);
    PTR(vs, 11); PTR(pg, 12); STREAM(13);
    CALL(hts_vtrace(lr, r, v, d, b, gamma, lambda, rho, c, T, N, vs, pg, stream), "hts_vtrace");
}
static PyObject *init(PyObject *self, PyObject *error)
{
    (void)self;
    Py_XSETREF(g_error, Py_NewRef(error));
    Py_RETURN_NONE;
}

#define M(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef kMethods[] = {
    M(policy_step), M(policy_step_host), M(policy_step_indexed), M(policy_evaluate), M(policy_gradient), M(policy_load_weights),
    M(a2c_terms), M(ppo_terms), M(delayed_update), M(gae), M(gae_host), M(vtrace), {"init", init, METH_O, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, kMethods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_value = PyUnicode_InternFromString("value");
    for (int i = 0; i < 12; ++i) s_weights[i] = PyUnicode_InternFromString(kWeights[i]);
    PyObject *np = PyImport_ImportModule("numpy"), *ct = np ? PyImport_ImportModule("ctypes") : NULL;
    g_ndarray = np ? (PyTypeObject *)PyObject_GetAttrString(np, "ndarray") : NULL;
    g_void_p = ct ? (PyTypeObject *)PyObject_GetAttrString(ct, "c_void_p") : NULL;
    g_argument_error = ct ? PyObject_GetAttrString(ct, "ArgumentError") : NULL;
    Py_XDECREF(np); Py_XDECREF(ct);
    if (!g_ndarray || !g_void_p || !g_argument_error) return NULL;
    g_error = Py_NewRef(PyExc_RuntimeError);           /* until init() */
    return PyModule_Create(&kModule);
}
