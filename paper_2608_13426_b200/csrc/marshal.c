/* Argument marshalling of the two calls whose launches are short enough for the host to bound them, rmm_product and
 * rmm_reduced_attn, as one native call each: reading three or four tensors, asking for the workspace size and calling the library
 * through ctypes took about as long as the GPU needs for a small product twice over.
 *
 * Only the plain form is taken (torch.Tensor or Parameter, no buffer passed in).  Whatever else it meets, and every
 * argument that would be refused, is answered with None: the caller's Python code then does the whole call, and raises what
 * it always raised.  Outputs and workspaces come from the same torch calls as there. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include "rmm.h"

static PyTypeObject *type_tensor, *type_parameter;
static PyObject *dt_bf16, *dt_f32, *dt_i32;
static PyObject *fn_stream, *fn_device, *names;   /* names: the Python module's, looked up at every call */
static PyObject *s_is_cuda, *s_dtype, *s_shape, *s_stride, *s_data_ptr, *s_new_empty, *s_get_device, *s_numel, *s_device, *s_cuda, *s_ws_cache, *s_workspace, *s_check, *s_out, *kw_dtype;
static int poison;

static int (*p_keep_count)(double, int64_t, int64_t *);
static size_t (*p_product_ws)(const rmm_mat_t *, const rmm_mat_t *, const rmm_mat_t *);
static size_t (*p_score_ws)(const rmm_mat_t *, int);
static size_t (*p_gemm_ws)(const rmm_mat_t *, const rmm_mat_t *, int64_t, const rmm_mat_t *);
static int (*p_product)(const rmm_mat_t *, const rmm_mat_t *, double, int64_t, float, const rmm_mat_t *, int32_t *, float *, void *, size_t, void *);
static size_t (*p_attn_ws)(const rmm_attn_desc_t *);
static int (*p_attn)(const rmm_attn_desc_t *, const void *, const void *, const void *, void *, int32_t *, int32_t *, void *, size_t, void *);

/* 1: read; 0: not a plain CUDA tensor of a known dtype (no exception is left set) */
typedef struct {
    void *ptr;
    PyObject *dtype;   /* borrowed: one of the dtypes above */
    int dims;
    int64_t shape[4], stride[4];
} tensor_t;

static int read_tensor(PyObject *t, tensor_t *o)
{
    PyObject *v, *shape = NULL, *stride = NULL;
    int ok = 0;
    if (Py_TYPE(t) != type_tensor && Py_TYPE(t) != type_parameter) return 0;
    if ((v = PyObject_GetAttr(t, s_is_cuda)) == NULL) goto out;
    ok = v == Py_True;
    Py_DECREF(v);
    if (!ok) return 0;
    ok = 0;
    if ((v = PyObject_GetAttr(t, s_dtype)) == NULL) goto out;
    o->dtype = v == dt_bf16 ? dt_bf16 : v == dt_f32 ? dt_f32 : NULL;
    Py_DECREF(v);
    if (o->dtype == NULL) return 0;
    if ((shape = PyObject_GetAttr(t, s_shape)) == NULL || (stride = PyObject_CallMethodNoArgs(t, s_stride)) == NULL) goto out;
    if (!PyTuple_Check(shape) || !PyTuple_Check(stride) || PyTuple_GET_SIZE(shape) > 4 || PyTuple_GET_SIZE(shape) != PyTuple_GET_SIZE(stride)) goto out;
    o->dims = (int)PyTuple_GET_SIZE(shape);
    for (int i = 0; i < o->dims; ++i) {
        if (!PyLong_CheckExact(PyTuple_GET_ITEM(shape, i)) || !PyLong_CheckExact(PyTuple_GET_ITEM(stride, i))) goto out;
        o->shape[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(shape, i));
        o->stride[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(stride, i));
    }
    if ((v = PyObject_CallMethodNoArgs(t, s_data_ptr)) == NULL) goto out;
    o->ptr = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    ok = !PyErr_Occurred();
out:
    Py_XDECREF(shape);
    Py_XDECREF(stride);
    PyErr_Clear();
    return ok;
}

static int read_mat(PyObject *t, rmm_mat_t *m, int *dims)
{
    tensor_t r;
    if (!read_tensor(t, &r) || (r.dims != 2 && r.dims != 3)) return 0;
    const int b = r.dims - 2;
    m->ptr = r.ptr;
    m->dtype = r.dtype == dt_bf16 ? RMM_BF16 : RMM_F32;
    m->batch = b ? r.shape[0] : 1;
    m->rows = r.shape[b]; m->cols = r.shape[b + 1];
    m->stride_batch = b ? r.stride[0] : 0;
    m->stride_row = r.stride[b]; m->stride_col = r.stride[b + 1];
    *dims = r.dims;
    return 1;
}

static PyObject *named(PyObject *name)   /* borrowed */
{
    PyObject *v = PyDict_GetItemWithError(names, name);
    if (v == NULL && !PyErr_Occurred()) PyErr_SetObject(PyExc_NameError, name);
    return v;
}

static int number(PyObject *o, double *v)
{
    if (!PyFloat_CheckExact(o) && !PyLong_CheckExact(o)) return 0;
    *v = PyFloat_AsDouble(o);
    if (PyErr_Occurred()) { PyErr_Clear(); return 0; }
    return 1;
}

/* A new tensor on `like`'s device, of the given sizes; its address through *ptr.  NULL with an exception on failure. */
static PyObject *new_out(PyObject *like, int dims, const int64_t *size, PyObject *dtype, void **ptr)
{
    PyObject *shape = PyTuple_New(dims), *t = NULL, *v;
    if (shape == NULL) return NULL;
    for (int i = 0; i < dims; ++i) {
        if ((v = PyLong_FromLongLong(size[i])) == NULL) { Py_DECREF(shape); return NULL; }
        PyTuple_SET_ITEM(shape, i, v);
    }
    if (poison) {
        PyObject *args[3] = {shape, dtype, like}, *out = named(s_out);
        t = out != NULL ? PyObject_Vectorcall(out, args, 3, NULL) : NULL;
    } else {
        PyObject *args[3] = {like, shape, dtype};
        t = PyObject_VectorcallMethod(s_new_empty, args, 2, kw_dtype);
    }
    Py_DECREF(shape);
    if (t == NULL) return NULL;
    if ((v = PyObject_CallMethodNoArgs(t, s_data_ptr)) == NULL) { Py_DECREF(t); return NULL; }
    *ptr = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return t;
}

/* The cached workspace of `like`'s device, at least `need` bytes: a new reference, its 256-byte aligned part through *ptr, *bytes */
static PyObject *workspace_of(PyObject *like, size_t need, void **ptr, size_t *bytes)
{
    PyObject *ws = NULL, *v, *key, *cache, *make;
    if (need < RMM_WS_HEADER_BYTES) need = RMM_WS_HEADER_BYTES;
    if ((v = PyObject_CallMethodNoArgs(like, s_get_device)) == NULL) return NULL;
    key = PyTuple_Pack(2, s_cuda, v);
    Py_DECREF(v);
    if (key == NULL) return NULL;
    /* (borrowed names are used at once: a tensor's methods may run Python code, which may bind them anew) */
    if ((cache = named(s_ws_cache)) != NULL && !PyDict_Check(cache)) PyErr_SetString(PyExc_TypeError, "_ws_cache must be a dict");
    ws = cache != NULL && PyDict_Check(cache) ? PyDict_GetItemWithError(cache, key) : NULL;
    Py_DECREF(key);
    if (ws == NULL && PyErr_Occurred()) return NULL;
    Py_XINCREF(ws);
    size_t have = 0;
    for (int pass = 0; pass < 2; ++pass) {
        if (ws != NULL) {
            if ((v = PyObject_CallMethodNoArgs(ws, s_numel)) == NULL) goto fail;
            have = PyLong_AsSize_t(v);
            Py_DECREF(v);
        }
        if (ws != NULL && have >= need) break;
        Py_XDECREF(ws);
        PyObject *dev = PyObject_GetAttr(like, s_device), *n = PyLong_FromSize_t(need);
        PyObject *args[2] = {n, dev};
        make = dev != NULL && n != NULL ? named(s_workspace) : NULL;
        ws = make != NULL ? PyObject_Vectorcall(make, args, 2, NULL) : NULL;
        Py_XDECREF(dev);
        Py_XDECREF(n);
        if (ws == NULL) return NULL;
    }
    if ((v = PyObject_CallMethodNoArgs(ws, s_data_ptr)) == NULL) goto fail;
    {
        const uintptr_t p = (uintptr_t)PyLong_AsVoidPtr(v), a = (p + 255) / 256 * 256;
        Py_DECREF(v);
        *ptr = (void *)a;
        *bytes = have - (size_t)(a - p);
    }
    if (PyErr_Occurred()) goto fail;
    return ws;
fail:
    Py_XDECREF(ws);
    return NULL;
}

static int stream_of(void **stream)
{
    PyObject *dev = PyObject_CallNoArgs(fn_device), *v;
    if (dev == NULL) return 0;
    v = PyObject_CallOneArg(fn_stream, dev);
    Py_DECREF(dev);
    if (v == NULL) return 0;
    *stream = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}

static int raise_status(int rc)   /* the library's text belongs to this thread, as in the Python code */
{
    PyObject *n = PyLong_FromLong(rc), *check = named(s_check), *v = n != NULL && check != NULL ? PyObject_CallOneArg(check, n) : NULL;
    Py_XDECREF(n);
    Py_XDECREF(v);
    return v != NULL;
}

/* product(A, B, rho, k, scale) -> (Y, idx) or None */
static PyObject *product(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    rmm_mat_t a, b, y;
    int da, db;
    double rho, scale;
    int64_t k;
    (void)self;
    if (n != 5 || !read_mat(args[0], &a, &da) || !read_mat(args[1], &b, &db) || !number(args[2], &rho) || !PyLong_CheckExact(args[3]) ||
        !number(args[4], &scale))
        Py_RETURN_NONE;
    k = PyLong_AsLongLong(args[3]);
    if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }
    int64_t kk = k;
    if (k <= 0 && p_keep_count(rho, a.cols, &kk) != RMM_OK) Py_RETURN_NONE;

    PyObject *Y = NULL, *idx = NULL, *ws = NULL, *ret = NULL;
    const int64_t ys[3] = {a.batch, a.rows, b.cols}, is[2] = {a.batch, kk};
    void *ip, *wp, *stream;
    size_t bytes, need;
    PyObject *dtype = a.dtype == RMM_BF16 ? dt_bf16 : dt_f32;
    if ((Y = new_out(args[0], da, ys + (da == 3 ? 0 : 1), dtype, &y.ptr)) == NULL) goto out;
    if ((idx = new_out(args[0], da - 1, is + (da == 3 ? 0 : 1), dt_i32, &ip)) == NULL) goto out;
    y.dtype = a.dtype; y.batch = a.batch; y.rows = a.rows; y.cols = b.cols;
    y.stride_col = 1;
    y.stride_row = b.cols > 0 ? b.cols : 1;   /* as torch describes a new tensor */
    y.stride_batch = da == 3 ? (a.rows > 0 ? a.rows : 1) * y.stride_row : 0;
    if (a.dtype == RMM_F32) {
        const size_t s = p_score_ws(&a, 1), g = p_gemm_ws(&a, &b, kk, &y);
        need = s == 0 || g == 0 ? 0 : s > g ? s : g;
    } else {
        need = p_product_ws(&a, &b, &y);
    }
    if (need == 0) { ret = Py_None; Py_INCREF(ret); goto out; }
    if ((ws = workspace_of(args[0], need, &wp, &bytes)) == NULL || !stream_of(&stream)) goto out;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = p_product(&a, &b, rho, k, (float)scale, &y, (int32_t *)ip, NULL, wp, bytes, stream);
    if (rc != RMM_OK) { Py_BLOCK_THREADS raise_status(rc); Py_UNBLOCK_THREADS }
    Py_END_ALLOW_THREADS
    if (rc == RMM_OK) ret = PyTuple_Pack(2, Y, idx);
out:
    Py_XDECREF(Y);
    Py_XDECREF(idx);
    Py_XDECREF(ws);
    return ret;
}

/* attn(Q, K, V, causal, rho_d, rho_t) -> O or None */
static PyObject *attn(PyObject *self, PyObject *const *args, Py_ssize_t n)
{
    tensor_t t[3];
    rmm_attn_desc_t d = {0};
    (void)self;
    if (n != 6) Py_RETURN_NONE;
    for (int i = 0; i < 3; ++i)
        if (!read_tensor(args[i], &t[i]) || t[i].dims != 4 || t[i].dtype != dt_bf16 || t[i].stride[3] != 1) Py_RETURN_NONE;
    if ((args[3] != Py_True && args[3] != Py_False) || !number(args[4], &d.rho_d) || !number(args[5], &d.rho_t)) Py_RETURN_NONE;
    d.B = t[0].shape[0]; d.Hq = t[0].shape[1]; d.Lq = t[0].shape[2]; d.Dh = t[0].shape[3];
    d.Hkv = t[1].shape[1]; d.Lk = t[1].shape[2];
    if (d.B < 1 || d.Hq < 1 || d.Lq < 1 || d.Dh < 1) Py_RETURN_NONE;
    if (t[1].shape[0] < d.B || t[1].shape[3] < d.Dh || t[2].shape[0] < d.B || t[2].shape[1] < d.Hkv || t[2].shape[2] < d.Lk ||
        t[2].shape[3] < d.Dh)
        Py_RETURN_NONE;   /* refused there: the library sees strides only */
    d.causal = args[3] == Py_True;
    for (int i = 0; i < 3; ++i) {
        d.q_stride[i] = t[0].stride[i];
        d.k_stride[i] = t[1].stride[i];
        d.v_stride[i] = t[2].stride[i];
    }
    d.o_stride[2] = d.Dh; d.o_stride[1] = d.Lq * d.Dh; d.o_stride[0] = d.Hq * d.o_stride[1];
    const size_t need = p_attn_ws(&d);
    if (need == 0) Py_RETURN_NONE;
    PyObject *O = NULL, *ws = NULL, *ret = NULL;
    const int64_t os[4] = {d.B, d.Hq, d.Lq, d.Dh};
    void *op, *wp, *stream;
    size_t bytes;
    int rc;
    if ((O = new_out(args[0], 4, os, dt_bf16, &op)) == NULL) goto out;
    if ((ws = workspace_of(args[0], need, &wp, &bytes)) == NULL || !stream_of(&stream)) goto out;
    Py_BEGIN_ALLOW_THREADS
    rc = p_attn(&d, t[0].ptr, t[1].ptr, t[2].ptr, op, NULL, NULL, wp, bytes, stream);
    if (rc != RMM_OK) { Py_BLOCK_THREADS raise_status(rc); Py_UNBLOCK_THREADS }
    Py_END_ALLOW_THREADS
    if (rc == RMM_OK) { ret = O; Py_INCREF(ret); }
out:
    Py_XDECREF(O);
    Py_XDECREF(ws);
    return ret;
}

static PyObject *set_poison(PyObject *self, PyObject *on)
{
    (void)self;
    poison = PyObject_IsTrue(on);
    Py_RETURN_NONE;
}

/* init(library path, (Tensor, Parameter), (bfloat16, float32, int32), (raw stream, current device), the module's names) */
static PyObject *init(PyObject *self, PyObject *args)
{
    const char *path;
    PyObject *tt, *tp;
    (void)self;
    if (!PyArg_ParseTuple(args, "s(OO)(OOO)(OO)O!", &path, &tt, &tp, &dt_bf16, &dt_f32, &dt_i32, &fn_stream, &fn_device, &PyDict_Type,
                          &names))
        return NULL;
    void *h = dlopen(path, RTLD_NOW);
    if (h == NULL) { PyErr_SetString(PyExc_RuntimeError, dlerror()); return NULL; }
    *(void **)&p_keep_count = dlsym(h, "rmm_keep_count");
    *(void **)&p_product_ws = dlsym(h, "rmm_product_workspace_bytes");
    *(void **)&p_score_ws = dlsym(h, "rmm_score_select_workspace_bytes");
    *(void **)&p_gemm_ws = dlsym(h, "rmm_reduced_gemm_workspace_bytes");
    *(void **)&p_product = dlsym(h, "rmm_product");
    *(void **)&p_attn_ws = dlsym(h, "rmm_reduced_attn_workspace_bytes");
    *(void **)&p_attn = dlsym(h, "rmm_reduced_attn");
    if (!p_keep_count || !p_product_ws || !p_score_ws || !p_gemm_ws || !p_product || !p_attn_ws || !p_attn) {
        PyErr_SetString(PyExc_RuntimeError, "librmm_b200.so lacks an entry point");
        return NULL;
    }
    type_tensor = (PyTypeObject *)tt;
    type_parameter = (PyTypeObject *)tp;
    PyObject *keep[] = {tt, tp, dt_bf16, dt_f32, dt_i32, fn_stream, fn_device, names};
    for (size_t i = 0; i < sizeof keep / sizeof *keep; ++i) Py_INCREF(keep[i]);   /* for the life of the process */
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"init", init, METH_VARARGS, NULL},
    {"set_poison", set_poison, METH_O, NULL},
    {"product", (PyCFunction)(void (*)(void))product, METH_FASTCALL, NULL},
    {"attn", (PyCFunction)(void (*)(void))attn, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "rmm_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit_rmm_marshal(void)
{
    struct { PyObject **p; const char *s; } texts[] = {
        {&s_is_cuda, "is_cuda"}, {&s_dtype, "dtype"}, {&s_shape, "shape"}, {&s_stride, "stride"}, {&s_data_ptr, "data_ptr"},
        {&s_new_empty, "new_empty"}, {&s_get_device, "get_device"}, {&s_numel, "numel"}, {&s_device, "device"}, {&s_cuda, "cuda"},
        {&s_ws_cache, "_ws_cache"}, {&s_workspace, "workspace"}, {&s_check, "_check"}, {&s_out, "_out"}};
    for (size_t i = 0; i < sizeof texts / sizeof *texts; ++i)
        if ((*texts[i].p = PyUnicode_InternFromString(texts[i].s)) == NULL) return NULL;
    if ((kw_dtype = PyTuple_Pack(1, s_dtype)) == NULL) return NULL;
    return PyModule_Create(&module);
}
