// The calls of a denoising pass without ctypes: a CPython module that takes the arguments of the binding's functions, turns them
// into those of the C ABI and returns the status code.  Marshalling only, as in binding.py, whose ctypes functions it stands in for:
// what is not of the plain kind (an integer where the ABI has a float, a numpy scalar) is left to them, at their price.
//   Of an append's 5.2 us of host time 2.1 were the launch and 2.0 the Python functions and ctypes' conversions (0.8 now), where the kernel of
// a small one runs for 2.1 us: 360 tokens, 2 heads of 128: 5.2 -> 3.65 us a call in a row; append and attention of 16 tokens
// 10.0 -> 7.5 us; six streams of 115 tokens, 16 heads of 64: 41.4 -> 27.5 us a step.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "llattn.h"

static PyObject *get_device, *get_stream;          // torch._C._cuda_getDevice, _cuda_getCurrentRawStream
static PyObject *s_data_ptr, *s_value, *s_cuda_stream;
static PyTypeObject *handle_type;                  // ctypes.c_void_p
static PyObject *not_here;                         // returned for arguments that only ctypes takes (or refuses)

// One argument list being converted: `bad` once something is not of the plain kind.
typedef struct {
    PyObject *const *a;
    int bad;
} Args;

static uint64_t as_u64(Args *x, PyObject *o)
{
    if (!PyLong_Check(o)) { x->bad = 1; return 0; }
    return PyLong_AsUnsignedLongLongMask(o);
}
static int as_int(Args *x, int i) { return (int)as_u64(x, x->a[i]); }
static int64_t as_i64(Args *x, int i) { return (int64_t)as_u64(x, x->a[i]); }

static float as_float(Args *x, int i)
{
    if (PyFloat_CheckExact(x->a[i])) return (float)PyFloat_AS_DOUBLE(x->a[i]);
    x->bad = 1;
    return 0.f;
}

// A tensor's address; None: NULL.
static void *as_ptr(Args *x, int i)
{
    PyObject *o = x->a[i], *r;
    void *p;
    if (o == Py_None || x->bad) return NULL;
    r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!r) { x->bad = 1; return NULL; }
    p = (void *)(uintptr_t)as_u64(x, r);
    Py_DECREF(r);
    return p;
}

// A handle: an integer or a c_void_p.  (Whatever else has a `value` is not one: ctypes says what becomes of it.)
static ll_cache *as_handle(Args *x, int i)
{
    PyObject *o = x->a[i], *r;
    void *p;
    if (PyLong_Check(o)) return (ll_cache *)(uintptr_t)as_u64(x, o);
    r = Py_TYPE(o) == handle_type ? PyObject_GetAttr(o, s_value) : NULL;
    if (!r) { x->bad = 1; return NULL; }
    p = r == Py_None ? NULL : (void *)(uintptr_t)as_u64(x, r);
    Py_DECREF(r);
    return (ll_cache *)p;
}

// The stream argument: None is torch's current stream of the current device.
static void *as_stream(Args *x, int i)
{
    PyObject *o = x->a[i], *dev, *r;
    void *p;
    if (x->bad) return NULL;
    if (PyLong_Check(o)) return (void *)(uintptr_t)as_u64(x, o);
    if (o == Py_None) {
        if (!get_stream) { x->bad = 1; return NULL; }
        dev = PyObject_CallNoArgs(get_device);
        if (!dev) { x->bad = 1; return NULL; }
        r = PyObject_CallOneArg(get_stream, dev);
        Py_DECREF(dev);
    } else {
        r = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!r) { x->bad = 1; return NULL; }
    p = (void *)(uintptr_t)as_u64(x, r);
    Py_DECREF(r);
    return p;
}

// What ctypes makes of the rest: the caller goes there, errors and all.
static PyObject *elsewhere(void)
{
    PyErr_Clear();
    Py_INCREF(not_here);
    return not_here;
}

// The library's functions, as binding.py found them.
static struct {
    __typeof__(&ll_rope_append_kv) rope_append_kv;
    __typeof__(&ll_norm_rope_append_kv) norm_rope_append_kv;
    __typeof__(&ll_sink_window_attn) sink_window_attn;
    __typeof__(&ll_cross_attn) cross_attn;
    __typeof__(&ll_qkv_proj_append) qkv_proj_append;
    __typeof__(&ll_sink_window_attn_batched) sink_window_attn_batched;
} L;

// The call itself runs without the interpreter lock, as under ctypes.
#define CALL(expr)                                   \
    do {                                             \
        int code_;                                   \
        if (x.bad) return elsewhere();               \
        Py_BEGIN_ALLOW_THREADS                       \
        code_ = (expr);                              \
        Py_END_ALLOW_THREADS                         \
        return PyLong_FromLong(code_);               \
    } while (0)

// (h, layer, q, k, v, frame_start, n_frames, grid_h, grid_w, rope_theta, q_out, stream)
static PyObject *rope_append_kv(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    Args x = {a, n != 12 || !L.rope_append_kv};
    if (x.bad) return elsewhere();
    ll_cache *h = as_handle(&x, 0);
    void *q = as_ptr(&x, 2), *k = as_ptr(&x, 3), *v = as_ptr(&x, 4), *q_out = as_ptr(&x, 10), *stream = as_stream(&x, 11);
    const int layer = as_int(&x, 1), frames = as_int(&x, 6), gh = as_int(&x, 7), gw = as_int(&x, 8);
    const int64_t start = as_i64(&x, 5);
    const float theta = as_float(&x, 9);
    CALL(L.rope_append_kv(h, layer, q, k, v, start, frames, gh, gw, theta, q_out, stream));
}

// (h, layer, q, k, v, gain_q, gain_k, eps, frame_start, n_frames, grid_h, grid_w, rope_theta, q_out, stream)
static PyObject *norm_rope_append_kv(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    Args x = {a, n != 15 || !L.norm_rope_append_kv};
    if (x.bad) return elsewhere();
    ll_cache *h = as_handle(&x, 0);
    void *q = as_ptr(&x, 2), *k = as_ptr(&x, 3), *v = as_ptr(&x, 4), *gq = as_ptr(&x, 5), *gk = as_ptr(&x, 6), *q_out = as_ptr(&x, 13),
         *stream = as_stream(&x, 14);
    const int layer = as_int(&x, 1), frames = as_int(&x, 9), gh = as_int(&x, 10), gw = as_int(&x, 11);
    const int64_t start = as_i64(&x, 8);
    const float eps = as_float(&x, 7), theta = as_float(&x, 12);
    CALL(L.norm_rope_append_kv(h, layer, q, k, v, gq, gk, eps, start, frames, gh, gw, theta, q_out, stream));
}

// (h, layer, q_roped, q_frame_start, n_q_frames, out, lse_out, stream)
static PyObject *sink_window_attn(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    Args x = {a, n != 8 || !L.sink_window_attn};
    if (x.bad) return elsewhere();
    ll_cache *h = as_handle(&x, 0);
    void *q = as_ptr(&x, 2), *out = as_ptr(&x, 5), *lse = as_ptr(&x, 6), *stream = as_stream(&x, 7);
    const int layer = as_int(&x, 1), frames = as_int(&x, 4);
    const int64_t start = as_i64(&x, 3);
    CALL(L.sink_window_attn(h, layer, q, start, frames, out, lse, stream));
}

// (h, q, n_q, k, v, n_k, out, lse_out, stream)
static PyObject *cross_attn(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    Args x = {a, n != 9 || !L.cross_attn};
    if (x.bad) return elsewhere();
    ll_cache *h = as_handle(&x, 0);
    void *q = as_ptr(&x, 1), *k = as_ptr(&x, 3), *v = as_ptr(&x, 4), *out = as_ptr(&x, 6), *lse = as_ptr(&x, 7), *stream = as_stream(&x, 8);
    const int64_t n_q = as_i64(&x, 2), n_k = as_i64(&x, 5);
    CALL(L.cross_attn(h, q, n_q, k, v, n_k, out, lse, stream));
}

// (h, layer, x, d_model, w_qkv, bias, gain_q, gain_k, eps, frame_start, n_frames, grid_h, grid_w, rope_theta, q_out, q_row_scale, workspace,
//  workspace_bytes, stream)
static PyObject *qkv_proj_append(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    Args x = {a, n != 19 || !L.qkv_proj_append};
    if (x.bad) return elsewhere();
    ll_cache *h = as_handle(&x, 0);
    void *in = as_ptr(&x, 2), *w = as_ptr(&x, 4), *bias = as_ptr(&x, 5), *gq = as_ptr(&x, 6), *gk = as_ptr(&x, 7), *q_out = as_ptr(&x, 14),
         *scale = as_ptr(&x, 15), *ws = as_ptr(&x, 16), *stream = as_stream(&x, 18);
    const int layer = as_int(&x, 1), d_model = as_int(&x, 3), frames = as_int(&x, 10), gh = as_int(&x, 11), gw = as_int(&x, 12);
    const int64_t start = as_i64(&x, 9);
    const size_t bytes = (size_t)as_i64(&x, 17);
    const float eps = as_float(&x, 8), theta = as_float(&x, 13);
    CALL(L.qkv_proj_append(h, layer, in, d_model, w, bias, gq, gk, eps, start, frames, gh, gw, theta, q_out, scale, ws, bytes, stream));
}

// (items, stream); an item is (handle, layer, q_roped, q_frame_start, n_q_frames, out, lse_out)
static PyObject *sink_window_attn_batched(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    ll_attn_item items[LL_MAX_BATCH];
    Args x = {a, n != 2 || !L.sink_window_attn_batched || !PyList_CheckExact(a[0]) || PyList_GET_SIZE(a[0]) > LL_MAX_BATCH};
    if (x.bad) return elsewhere();
    const int count = (int)PyList_GET_SIZE(a[0]);
    for (int i = 0; i < count; ++i) {
        PyObject *t = PyList_GET_ITEM(a[0], i);
        if (!PyTuple_CheckExact(t) || PyTuple_GET_SIZE(t) != 7) return elsewhere();
        PyObject *parts[7];
        for (int j = 0; j < 7; ++j) parts[j] = PyTuple_GET_ITEM(t, j);
        Args y = {parts, 0};
        items[i].cache = as_handle(&y, 0);
        items[i].layer = as_int(&y, 1);
        items[i].n_q_frames = as_int(&y, 4);
        items[i].q_roped = as_ptr(&y, 2);
        items[i].q_frame_start = as_i64(&y, 3);
        items[i].out = as_ptr(&y, 5);
        items[i].lse_out = as_ptr(&y, 6);
        if (y.bad) return elsewhere();
    }
    void *stream = as_stream(&x, 1);
    CALL(L.sink_window_attn_batched(items, count, stream));
}

// bind({name: address}, c_void_p): the library's functions, and the type of a handle.
static PyObject *bind(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    PyObject *o;
    if (n != 2 || !PyDict_Check(a[0]) || !PyType_Check(a[1])) {
        PyErr_SetString(PyExc_TypeError, "bind({name: address}, c_void_p)");
        return NULL;
    }
    PyObject *const d = a[0];
#define TAKE(name)                                              \
    o = PyDict_GetItemString(d, "ll_" #name);                   \
    if (!o) return PyErr_Format(PyExc_KeyError, "ll_" #name);   \
    L.name = (__typeof__(L.name))PyLong_AsVoidPtr(o);           \
    if (PyErr_Occurred()) return NULL;
    TAKE(rope_append_kv)
    TAKE(norm_rope_append_kv)
    TAKE(sink_window_attn)
    TAKE(cross_attn)
    TAKE(qkv_proj_append)
    TAKE(sink_window_attn_batched)
    Py_INCREF(a[1]);
    Py_XSETREF(handle_type, (PyTypeObject *)a[1]);
    Py_RETURN_NONE;
}

// streams(get_device, get_stream): where the current stream's raw handle comes from, once CUDA is initialised.
static PyObject *streams(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    if (n != 2) { PyErr_SetString(PyExc_TypeError, "streams(get_device, get_stream)"); return NULL; }
    Py_INCREF(a[0]);
    Py_INCREF(a[1]);
    Py_XSETREF(get_device, a[0]);
    Py_XSETREF(get_stream, a[1]);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {
    FAST(rope_append_kv), FAST(norm_rope_append_kv), FAST(sink_window_attn), FAST(cross_attn), FAST(qkv_proj_append),
    FAST(sink_window_attn_batched), FAST(streams), FAST(bind), {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", "Argument marshalling of the hot calls.", -1, methods};

PyMODINIT_FUNC PyInit__marshal(void)
{
    PyObject *m = PyModule_Create(&module);
    if (!m) return NULL;
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_value = PyUnicode_InternFromString("value");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    not_here = PyObject_CallNoArgs((PyObject *)&PyBaseObject_Type);
    if (!s_data_ptr || !s_value || !s_cuda_stream || !not_here || PyModule_AddObjectRef(m, "ELSEWHERE", not_here) < 0) return NULL;
    return m;
}
