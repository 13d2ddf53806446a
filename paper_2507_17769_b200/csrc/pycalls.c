/* The calls of every iteration (append, gather, plan, run) as a CPython extension: argument marshalling only.
 *
 * Through ctypes each of them spends 3 to 4 us on marshalling, more than its kernel launch takes; a small batch, whose
 * kernels take 15 us, was bound by that.  Pointers travel as Python integers, length arrays through the buffer protocol.
 * The addresses of the C ABI's functions are handed in by binding.py, so that this module uses the library that it loaded.
 * Every call gives the interpreter lock back while the library runs and returns the library's status. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

typedef int (*kv_write_fn)(void *, const void *, const void *, const int32_t *, int32_t, const int32_t *, const int32_t *, int32_t, void *);
typedef int (*kv_gather_fn)(const void *, const int32_t *, int32_t, void *, void *, void *);
typedef int (*attn_plan_fn)(const void *, const int32_t *, const int32_t *, int32_t, int32_t, const void *, void **, size_t *);
typedef int (*attn_run_fn)(void *, const void *, const void *, const int32_t *, void *, float *, void *, size_t, void *);

static kv_write_fn f_write;
static kv_gather_fn f_gather;
static attn_plan_fn f_plan;
static attn_run_fn f_run;

/* an address or None */
static int as_ptr(PyObject *o, void **p) {
    if (o == Py_None) {
        *p = NULL;
        return 1;
    }
    *p = PyLong_AsVoidPtr(o);
    return !(*p == NULL && PyErr_Occurred());
}
static int as_i32(PyObject *o, int32_t *v) {
    const long x = PyLong_AsLong(o);
    if (x == -1 && PyErr_Occurred()) return 0;
    if (x > INT32_MAX || x < INT32_MIN) {
        PyErr_SetString(PyExc_OverflowError, "argument does not fit 32 bits");
        return 0;
    }
    *v = (int32_t)x;
    return 1;
}
/* a contiguous int32 array of one entry per request */
static int as_lengths(PyObject *o, Py_buffer *b) {
    if (PyObject_GetBuffer(o, b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) return 0;
    if (b->ndim >= 1 && b->itemsize == 4 && b->format && strcmp(b->format, "i") == 0) return 1;
    PyBuffer_Release(b);
    PyErr_SetString(PyExc_TypeError, "lengths must be an int32 array");
    return 0;
}
/* the two length arrays of a batch and its number of requests, which is prior's */
static int as_batch(PyObject *prior, PyObject *q_len, Py_buffer *a, Py_buffer *b, int32_t *n) {
    if (!as_lengths(prior, a)) return 0;
    if (!as_lengths(q_len, b)) {
        PyBuffer_Release(a);
        return 0;
    }
    *n = (int32_t)a->shape[0];
    if (a->shape[0] <= b->shape[0] && a->shape[0] <= INT32_MAX) return 1;
    PyBuffer_Release(a);
    PyBuffer_Release(b);
    PyErr_SetString(PyExc_ValueError, "q_len is shorter than prior");
    return 0;
}
static int count_is(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return 1;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
    return 0;
}

static PyObject *py_bind(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *p[4];
    if (!count_is(n, 4)) return NULL;
    for (int k = 0; k < 4; ++k)
        if (!as_ptr(a[k], &p[k])) return NULL;
    f_write = (kv_write_fn)p[0];
    f_gather = (kv_gather_fn)p[1];
    f_plan = (attn_plan_fn)p[2];
    f_run = (attn_run_fn)p[3];
    Py_RETURN_NONE;
}

/* (kv, k, v, block_table, max_pages, prior, q_len, stream) -> status */
static PyObject *py_kv_write(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *kv, *k, *v, *bt, *stream;
    int32_t max_pages, n_req;
    Py_buffer pr, ql;
    int st;
    if (!count_is(n, 8) || !as_ptr(a[0], &kv) || !as_ptr(a[1], &k) || !as_ptr(a[2], &v) || !as_ptr(a[3], &bt) || !as_i32(a[4], &max_pages) ||
        !as_ptr(a[7], &stream) || !as_batch(a[5], a[6], &pr, &ql, &n_req))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = f_write(kv, k, v, (const int32_t *)bt, max_pages, (const int32_t *)pr.buf, (const int32_t *)ql.buf, n_req, stream);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&pr);
    PyBuffer_Release(&ql);
    return PyLong_FromLong(st);
}

/* (kv, block_table_row, length, k_out, v_out, stream) -> status */
static PyObject *py_kv_gather(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *kv, *bt, *k, *v, *stream;
    int32_t len;
    int st;
    if (!count_is(n, 6) || !as_ptr(a[0], &kv) || !as_ptr(a[1], &bt) || !as_i32(a[2], &len) || !as_ptr(a[3], &k) || !as_ptr(a[4], &v) ||
        !as_ptr(a[5], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = f_gather(kv, (const int32_t *)bt, len, k, v, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

/* (address of the shape, prior, q_len, max_pages, plan or None) -> (status, plan, workspace bytes) */
static PyObject *py_attn_plan(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *shape, *plan;
    int32_t max_pages, n_req;
    size_t ws = 0;
    Py_buffer pr, ql;
    int st;
    if (!count_is(n, 5) || !as_ptr(a[0], &shape) || !as_i32(a[3], &max_pages) || !as_ptr(a[4], &plan) || !as_batch(a[1], a[2], &pr, &ql, &n_req))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = f_plan(shape, (const int32_t *)pr.buf, (const int32_t *)ql.buf, n_req, max_pages, NULL, &plan, &ws);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&pr);
    PyBuffer_Release(&ql);
    return Py_BuildValue("iNn", st, PyLong_FromVoidPtr(plan), (Py_ssize_t)ws);
}

/* (plan, kv, q, block_table, out, lse or None, workspace, workspace bytes, stream) -> status */
static PyObject *py_attn_run(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *plan, *kv, *q, *bt, *out, *lse, *ws, *stream;
    size_t bytes;
    int st;
    if (!count_is(n, 9) || !as_ptr(a[0], &plan) || !as_ptr(a[1], &kv) || !as_ptr(a[2], &q) || !as_ptr(a[3], &bt) || !as_ptr(a[4], &out) ||
        !as_ptr(a[5], &lse) || !as_ptr(a[6], &ws) || !as_ptr(a[8], &stream))
        return NULL;
    bytes = PyLong_AsSize_t(a[7]);
    if (bytes == (size_t)-1 && PyErr_Occurred()) return NULL;
    Py_BEGIN_ALLOW_THREADS
    st = f_run(plan, kv, q, (const int32_t *)bt, out, (float *)lse, ws, bytes, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

static PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, "addresses of ps_kv_write, ps_kv_gather, ps_attn_plan, ps_attn_run"},
    {"kv_write", (PyCFunction)(void (*)(void))py_kv_write, METH_FASTCALL, "ps_kv_write"},
    {"kv_gather", (PyCFunction)(void (*)(void))py_kv_gather, METH_FASTCALL, "ps_kv_gather"},
    {"attn_plan", (PyCFunction)(void (*)(void))py_attn_plan, METH_FASTCALL, "ps_attn_plan without options"},
    {"attn_run", (PyCFunction)(void (*)(void))py_attn_run, METH_FASTCALL, "ps_attn_run"},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycalls", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__pycalls(void) { return PyModule_Create(&module); }
