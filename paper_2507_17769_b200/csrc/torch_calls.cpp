// Append, gather and run of PagedAttention as a CPython extension that takes torch tensors: the checks, the allocation of the
// results and the call into the library in one step.
//
// Iterations of small batches are bound by the host: 15 us of calls beside kernels of 8 to 12.  Of that the allocation of two results
// from Python took 4 us, and the tensors' addresses and checks 1 a call.  Measured (8 decode rows of 512 tokens): run 7.9 -> 5.5 us,
// append 4.1 -> 3.2, the iteration 14.7 -> 11.7; a gather 8.7 -> 6.6.  Tensors of subclasses do not come here (session.py).
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>
#include <ATen/ATen.h>

#include <cstdint>
#include <cstring>

namespace {

typedef int (*kv_write_fn)(void*, const void*, const void*, const int32_t*, int32_t, const int32_t*, const int32_t*, int32_t, void*);
typedef int (*kv_gather_fn)(const void*, const int32_t*, int32_t, void*, void*, void*);
typedef int (*attn_run_fn)(void*, const void*, const void*, const int32_t*, void*, float*, void*, size_t, void*);
kv_write_fn f_write;
kv_gather_fn f_gather;
attn_run_fn f_run;

bool count_is(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
    return false;
}
// an address, or None, which the library refuses: a closed session's handles are None
bool as_ptr(PyObject* o, void** p) {
    if (o == Py_None) {
        *p = nullptr;
        return true;
    }
    *p = PyLong_AsVoidPtr(o);
    return !(*p == nullptr && PyErr_Occurred());
}
bool as_i64(PyObject* o, int64_t* v) {  // (what has __index__; a truth value is no size to torch either)
    if (PyBool_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "an integer expected, got bool");
        return false;
    }
    *v = PyLong_AsLongLong(o);
    return !(*v == -1 && PyErr_Occurred());
}
bool as_tensor(PyObject* o, const at::Tensor** t) {
    if (THPVariable_Check(o)) {
        *t = &THPVariable_Unpack(o);
        return true;
    }
    PyErr_SetString(PyExc_TypeError, "a tensor expected");
    return false;
}
bool holds(bool what, const char* message) {
    if (!what) PyErr_SetString(PyExc_AssertionError, message);
    return what;
}

// a contiguous int32 array of one entry per request
struct Lengths {
    Py_buffer b;
    bool held = false;
    bool get(PyObject* o) {
        if (PyObject_GetBuffer(o, &b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) return false;
        held = true;
        if (b.ndim >= 1 && b.itemsize == 4 && b.format && strcmp(b.format, "i") == 0) return true;
        PyErr_SetString(PyExc_TypeError, "lengths must be an int32 array");
        return false;
    }
    ~Lengths() {
        if (held) PyBuffer_Release(&b);
    }
};

// The interpreter lock is given back while the library runs and while results are allocated: an allocation may wait for the device, and
// what that waits for may need the interpreter.
struct Unlocked {
    PyThreadState* s = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(s); }
};

PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void* p[3];
    if (!count_is(n, 3)) return nullptr;
    for (int k = 0; k < 3; ++k)
        if (!as_ptr(a[k], &p[k])) return nullptr;
    f_write = (kv_write_fn)p[0];
    f_gather = (kv_gather_fn)p[1];
    f_run = (attn_run_fn)p[2];
    Py_RETURN_NONE;
}

// (kv, k, v, block table, max_pages or None, prior, q_len, stream) -> status
PyObject* py_write(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    void *kv, *stream;
    const at::Tensor *k, *v, *bt;
    int64_t max_pages;
    Lengths prior, q_len;
    if (!count_is(n, 8) || !as_ptr(a[0], &kv) || !as_tensor(a[1], &k) || !as_tensor(a[2], &v) || !as_tensor(a[3], &bt) || !as_ptr(a[7], &stream)) return nullptr;
    if (a[4] == Py_None) max_pages = bt->size(-1);
    else if (!as_i64(a[4], &max_pages)) return nullptr;
    if (!holds(k->is_contiguous() && v->is_contiguous() && bt->is_contiguous(), "k_new, v_new and the block table must be contiguous")) return nullptr;
    if (max_pages > INT32_MAX || max_pages < INT32_MIN) {
        PyErr_SetString(PyExc_OverflowError, "argument does not fit 32 bits");
        return nullptr;
    }
    if (!prior.get(a[5]) || !q_len.get(a[6])) return nullptr;
    if (prior.b.shape[0] > q_len.b.shape[0] || prior.b.shape[0] > INT32_MAX) {
        PyErr_SetString(PyExc_ValueError, "q_len is shorter than prior");
        return nullptr;
    }
    int st;
    {
        Unlocked u;
        st = f_write(kv, k->data_ptr(), v->data_ptr(), (const int32_t*)bt->data_ptr(), (int32_t)max_pages, (const int32_t*)prior.b.buf, (const int32_t*)q_len.b.buf,
                     (int32_t)prior.b.shape[0], stream);
    }
    return PyLong_FromLong(st);
    END_HANDLE_TH_ERRORS
}

PyObject* three(int st, PyObject* x, PyObject* y) {  // (takes both references)
    THPObjectPtr ox(x), oy(y), os(PyLong_FromLong(st));
    if (!ox || !oy || !os) return nullptr;
    PyObject* t = PyTuple_New(3);
    if (!t) return nullptr;
    PyTuple_SET_ITEM(t, 0, os.release());
    PyTuple_SET_ITEM(t, 1, ox.release());
    PyTuple_SET_ITEM(t, 2, oy.release());
    return t;
}
PyObject* again(PyObject* o) {
    Py_INCREF(o);
    return o;
}

// (kv, block table row, length, kv heads, head dim, a tensor of the pool's device, stream) -> (status, K, V)
PyObject* py_gather(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    void *kv, *stream;
    const at::Tensor *bt, *pool;
    int64_t len, hkv, d;
    if (!count_is(n, 7) || !as_ptr(a[0], &kv) || !as_tensor(a[1], &bt) || !as_i64(a[2], &len) || !as_i64(a[3], &hkv) || !as_i64(a[4], &d) || !as_tensor(a[5], &pool) ||
        !as_ptr(a[6], &stream))
        return nullptr;
    if (len > INT32_MAX || len < INT32_MIN) {
        PyErr_SetString(PyExc_OverflowError, "argument does not fit 32 bits");
        return nullptr;
    }
    at::Tensor k, v;
    int st;
    {
        Unlocked u;
        const auto opts = pool->options().dtype(at::kBFloat16);
        k = at::empty({len, hkv, d}, opts), v = at::empty({len, hkv, d}, opts);
        st = f_gather(kv, (const int32_t*)bt->data_ptr(), (int32_t)len, k.data_ptr(), v.data_ptr(), stream);
    }
    return three(st, THPVariable_Wrap(std::move(k)), THPVariable_Wrap(std::move(v)));
    END_HANDLE_TH_ERRORS
}

// (plan, kv, q, block table, out or None, lse or None, want lse, q tokens, q heads, a tensor of the pool's device, workspace, its
// bytes, stream) -> (status, out, lse or None)
PyObject* py_run(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    void *plan, *kv, *ws, *stream;
    const at::Tensor *q, *bt, *pool;
    int64_t total_q, hq, bytes;
    if (!count_is(n, 13) || !as_ptr(a[0], &plan) || !as_ptr(a[1], &kv) || !as_tensor(a[2], &q) || !as_tensor(a[3], &bt) || !as_i64(a[7], &total_q) ||
        !as_i64(a[8], &hq) || !as_tensor(a[9], &pool) || !as_ptr(a[10], &ws) || !as_i64(a[11], &bytes) || !as_ptr(a[12], &stream))
        return nullptr;
    if (!holds(q->is_contiguous() && q->size(0) == total_q && bt->is_contiguous(), "q must be contiguous with a row per planned token, and the block table contiguous"))
        return nullptr;
    const at::Tensor *given_out = nullptr, *given_lse = nullptr;
    if ((a[4] != Py_None && !as_tensor(a[4], &given_out)) || (a[5] != Py_None && !as_tensor(a[5], &given_lse))) return nullptr;
    at::Tensor out, lse;
    int st;
    {
        Unlocked u;
        if (!given_out) out = at::empty(q->sizes(), q->options());
        if (!given_lse && a[6] == Py_True) lse = at::empty({total_q, hq}, pool->options().dtype(at::kFloat));
        void* const lse_ptr = given_lse ? given_lse->data_ptr() : lse.defined() ? lse.data_ptr() : nullptr;
        st = f_run(plan, kv, q->data_ptr(), (const int32_t*)bt->data_ptr(), given_out ? given_out->data_ptr() : out.data_ptr(), (float*)lse_ptr, ws, (size_t)bytes,
                   stream);
    }
    return three(st, out.defined() ? THPVariable_Wrap(std::move(out)) : again(a[4]), lse.defined() ? THPVariable_Wrap(std::move(lse)) : again(a[5]));
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, "addresses of ps_kv_write, ps_kv_gather, ps_attn_run"},
    {"write", (PyCFunction)(void (*)(void))py_write, METH_FASTCALL, "ps_kv_write"},
    {"gather", (PyCFunction)(void (*)(void))py_gather, METH_FASTCALL, "ps_kv_gather into new tensors"},
    {"run", (PyCFunction)(void (*)(void))py_run, METH_FASTCALL, "ps_attn_run"},
    {nullptr, nullptr, 0, nullptr},
};
struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_calls(void) { return PyModule_Create(&module); }
