// Native half of the Python binding: checks the tensors of a call and passes their device pointers on to
// the C ABI.
//
// A decode step of a small model is a handful of launches of a few microseconds each, so what the host
// spends on a call decides its rate.  Through ctypes a call took 8.6 us (one launch) to 14.7 us (three):
// mostly Python-level attribute look-ups of the tensors (device, type, contiguity, shape), the current
// stream and the conversion of nine arguments.  Here the same checks read the tensor objects directly.
// The arithmetic, and every check of values, stays in the library.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <new>

#include "../../include/esa.h"

namespace {

PyObject* g_error = nullptr;      // binding.EsaError(status, where)

struct CtxObject {
    PyObject_HEAD
    esa_ctx* h;
    esa_config cfg;
};

struct FitObject {
    PyObject_HEAD
    esa_fit* h;
    esa_config cfg;
};

bool raise_status(esa_status st, const char* where) {
    PyObject* e = PyObject_CallFunction(g_error, "is", (int)st, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    return false;
}

// ------------------------------------------------------------------ tensors
const at::Tensor* as_tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a torch tensor", name);
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

bool has_shape(const at::Tensor& t, const int64_t* want, int n) {
    const auto s = t.sizes();
    if ((int)s.size() != n) return false;
    for (int i = 0; i < n; ++i)
        if (s[i] != want[i]) return false;
    return true;
}

void shape_error(const at::Tensor& t, const char* name, const int64_t* want, int n) {
    PyObject* w = PyTuple_New(n);
    PyObject* g = PyTuple_New((Py_ssize_t)t.dim());
    if (w && g) {
        for (int i = 0; i < n; ++i) PyTuple_SET_ITEM(w, i, PyLong_FromLongLong(want[i]));
        for (int i = 0; i < (int)t.dim(); ++i) PyTuple_SET_ITEM(g, i, PyLong_FromLongLong(t.size(i)));
        PyErr_Format(PyExc_ValueError, "%s must have shape %R, got %R", name, w, g);
    }
    Py_XDECREF(w);
    Py_XDECREF(g);
}

// Device pointer of a contiguous CUDA tensor of the given type and shape, or a Python error.
bool device_ptr(PyObject* o, const char* name, at::ScalarType dtype, std::initializer_list<int64_t> shape, void** out) {
    const at::Tensor* t = as_tensor(o, name);
    if (!t) return false;
    if (!t->is_cuda()) {
        PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor", name);
        return false;
    }
    if (t->scalar_type() != dtype) {
        PyObject* got = PyObject_GetAttrString(o, "dtype");
        PyErr_Format(PyExc_TypeError, "%s must have dtype %s, got %S", name,
                     dtype == at::ScalarType::BFloat16 ? "torch.bfloat16" : dtype == at::ScalarType::Int ? "torch.int32" : "torch.float32",
                     got ? got : Py_None);
        Py_XDECREF(got);
        return false;
    }
    if (!t->is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
        return false;
    }
    if (!has_shape(*t, shape.begin(), (int)shape.size())) {
        shape_error(*t, name, shape.begin(), (int)shape.size());
        return false;
    }
    *out = t->data_ptr();
    return true;
}

bool leading_sizes(PyObject* o, const char* name, int n, int64_t* out) {
    const at::Tensor* t = as_tensor(o, name);
    if (!t) return false;
    if ((int)t->dim() < n) {
        PyErr_Format(PyExc_ValueError, "%s must have at least %d dimensions", name, n);
        return false;
    }
    for (int i = 0; i < n; ++i) out[i] = t->size(i);
    return true;
}

// ------------------------------------------------------------------ scalars
constexpr int kMaxSeq = 64;       // the library refuses larger batches; longer lists are still measured against B first

struct NPrev {
    int64_t v[kMaxSeq];
    int n = 0;
};

bool read_n_prev(PyObject* o, int64_t B, NPrev* out) {
    if (PyObject_Size(o) < 0) return false;         // (something with a length: a call would use an iterator up)
    PyObject* seq = PySequence_Fast(o, "n_prev must be a sequence of integers");
    if (!seq) return false;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    bool ok = n == (Py_ssize_t)B;
    if (!ok) PyErr_SetString(PyExc_ValueError, "n_prev must have one entry per sequence");
    for (Py_ssize_t i = 0; ok && i < n && i < kMaxSeq; ++i) {
        PyObject* it = PySequence_Fast_GET_ITEM(seq, i);
        if (PyLong_Check(it)) {
            out->v[i] = PyLong_AsLongLong(it);
        } else {
            PyObject* as_int = PyNumber_Long(it);
            if (!as_int) { ok = false; break; }
            out->v[i] = PyLong_AsLongLong(as_int);
            Py_DECREF(as_int);
        }
        if (out->v[i] == -1 && PyErr_Occurred()) ok = false;
    }
    out->n = (int)n;
    Py_DECREF(seq);
    return ok;
}

// stream: None (torch's current stream), an integer handle, or an object with a cuda_stream attribute
bool read_stream(PyObject* o, void** out) {
    if (o == Py_None) {
        *out = (void*)c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* v = PyLong_Check(o) ? Py_NewRef(o) : PyObject_GetAttrString(o, "cuda_stream");
    if (!v) return false;
    const unsigned long long x = PyLong_AsUnsignedLongLong(v);
    Py_DECREF(v);
    if (x == (unsigned long long)-1 && PyErr_Occurred()) return false;
    *out = (void*)(uintptr_t)x;
    return true;
}

// Trailing (stream, sync) pair of every call.
struct Where {
    void* stream = nullptr;
    bool sync = false;
};

bool read_where(PyObject* stream, PyObject* sync, Where* w) {
    const int s = PyObject_IsTrue(sync);
    if (s < 0) return false;
    w->sync = s != 0;
    return w->sync || read_stream(stream, &w->stream);
}

bool want_args(Py_ssize_t got, Py_ssize_t want, const char* name) {
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", name, want, got);
    return false;
}

// Runs a library call without the interpreter lock (it may wait for the device, or for room in the launch queue).
template <typename F>
PyObject* finish(const char* name, F call) {
    esa_status st = ESA_OK;
    bool threw = false;
    Py_BEGIN_ALLOW_THREADS
    try {
        st = call();
    } catch (...) {                 // (the library throws nothing but what its allocations on the host throw)
        threw = true;
    }
    Py_END_ALLOW_THREADS
    if (threw) return PyErr_NoMemory();
    if (st != ESA_OK) {
        raise_status(st, name);
        return nullptr;
    }
    Py_RETURN_NONE;
}

constexpr at::ScalarType kBf16 = at::ScalarType::BFloat16, kI32 = at::ScalarType::Int, kF32 = at::ScalarType::Float;

// ------------------------------------------------------------------ context calls
// (K_new, V_new, K_cache, V_cache, n_prev, stream, sync)
PyObject* ctx_append_kv(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 7, "append_kv")) return nullptr;
    const esa_config& c = self->cfg;
    int64_t d[2];
    void *kn, *vn, *kc, *vc;
    NPrev np;
    Where w;
    if (!leading_sizes(a[0], "K_new", 2, d) ||
        !device_ptr(a[0], "K_new", kBf16, {d[0], d[1], c.n_kv_heads, c.head_dim}, &kn) ||
        !device_ptr(a[1], "V_new", kBf16, {d[0], d[1], c.n_kv_heads, c.head_dim}, &vn) ||
        !device_ptr(a[2], "K_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &kc) ||
        !device_ptr(a[3], "V_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &vc) ||
        !read_n_prev(a[4], d[0], &np) || !read_where(a[5], a[6], &w))
        return nullptr;
    return finish("esa_append_kv", [&] {
        return w.sync ? esa_append_kv(self->h, (int32_t)d[0], kn, vn, (int32_t)d[1], kc, vc, np.v)
                      : esa_append_kv_async(self->h, (int32_t)d[0], kn, vn, (int32_t)d[1], kc, vc, np.v, w.stream);
    });
}

// (K_new, kc_cache, n_prev, stream, sync)
PyObject* ctx_compress_keys(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 5, "compress_keys")) return nullptr;
    const esa_config& c = self->cfg;
    int64_t d[2];
    void *kn, *kc;
    NPrev np;
    Where w;
    if (!leading_sizes(a[0], "K_new", 2, d) ||
        !device_ptr(a[0], "K_new", kBf16, {d[0], d[1], c.n_kv_heads, c.head_dim}, &kn) ||
        !device_ptr(a[1], "kc_cache", kBf16, {d[0], c.max_tokens, c.d_c}, &kc) || !read_n_prev(a[2], d[0], &np) ||
        !read_where(a[3], a[4], &w))
        return nullptr;
    return finish("esa_compress_keys", [&] {
        return w.sync ? esa_compress_keys(self->h, (int32_t)d[0], kn, (int32_t)d[1], kc, np.v)
                      : esa_compress_keys_async(self->h, (int32_t)d[0], kn, (int32_t)d[1], kc, np.v, w.stream);
    });
}

// (Q_cur, kc_cache, n_prev, idx_out, n_sel_out, stream, sync)
PyObject* ctx_select(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 7, "select")) return nullptr;
    const esa_config& c = self->cfg;
    int64_t d[2];
    void *q, *kc, *idx, *n_sel;
    NPrev np;
    Where w;
    if (!leading_sizes(a[0], "Q_cur", 2, d) || !device_ptr(a[0], "Q_cur", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &q) ||
        !device_ptr(a[1], "kc_cache", kBf16, {d[0], c.max_tokens, c.d_c}, &kc) ||
        !device_ptr(a[3], "idx_out", kI32, {d[0], c.top_k}, &idx) || !device_ptr(a[4], "n_sel_out", kI32, {d[0]}, &n_sel) ||
        !read_n_prev(a[2], d[0], &np) || !read_where(a[5], a[6], &w))
        return nullptr;
    return finish("esa_select", [&] {
        return w.sync ? esa_select(self->h, (int32_t)d[0], q, (int32_t)d[1], kc, np.v, (int32_t*)idx, (int32_t*)n_sel)
                      : esa_select_async(self->h, (int32_t)d[0], q, (int32_t)d[1], kc, np.v, (int32_t*)idx, (int32_t*)n_sel,
                                         w.stream);
    });
}

// (Q_cur, K_cache, n_prev, mode, idx_out, n_sel_out, stream, sync)
PyObject* ctx_select_full(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 8, "select_full")) return nullptr;
    const esa_config& c = self->cfg;
    int64_t d[2];
    void *q, *kc, *idx, *n_sel;
    NPrev np;
    Where w;
    if (!leading_sizes(a[0], "Q_cur", 2, d) || !device_ptr(a[0], "Q_cur", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &q) ||
        !device_ptr(a[1], "K_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &kc) ||
        !device_ptr(a[4], "idx_out", kI32, {d[0], c.top_k}, &idx) || !device_ptr(a[5], "n_sel_out", kI32, {d[0]}, &n_sel) ||
        !read_n_prev(a[2], d[0], &np) || !read_where(a[6], a[7], &w))
        return nullptr;
    const int mode = PyObject_IsTrue(a[3]);
    if (mode < 0) return nullptr;
    return finish("esa_select_full", [&] {
        return w.sync ? esa_select_full(self->h, (int32_t)d[0], q, (int32_t)d[1], kc, np.v, mode, (int32_t*)idx, (int32_t*)n_sel)
                      : esa_select_full_async(self->h, (int32_t)d[0], q, (int32_t)d[1], kc, np.v, mode, (int32_t*)idx,
                                              (int32_t*)n_sel, w.stream);
    });
}

// (Q_cur, Q_far | None, K_cache, K_far_cache | None, V_cache, n_prev, idx, n_sel, O, stream, sync); `two`: named in errors
PyObject* attend_common(CtxObject* self, PyObject* q_o, PyObject* qf_o, PyObject* k_o, PyObject* kf_o, PyObject* v_o, PyObject* np_o,
                        PyObject* idx_o, PyObject* ns_o, PyObject* o_o, PyObject* stream, PyObject* sync, bool two) {
    const esa_config& c = self->cfg;
    int64_t d[2];
    void *q, *qf = nullptr, *k, *kf = nullptr, *v, *idx, *n_sel, *o;
    NPrev np;
    Where w;
    if (!leading_sizes(q_o, "Q_cur", 2, d) || !device_ptr(q_o, "Q_cur", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &q)) return nullptr;
    if (qf_o != Py_None && !device_ptr(qf_o, "Q_far", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &qf)) return nullptr;
    if (!device_ptr(k_o, "K_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &k)) return nullptr;
    if (kf_o != Py_None && !device_ptr(kf_o, "K_far_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &kf)) return nullptr;
    if (!device_ptr(v_o, "V_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &v) ||
        !device_ptr(idx_o, "idx", kI32, {d[0], c.top_k}, &idx) || !device_ptr(ns_o, "n_sel", kI32, {d[0]}, &n_sel) ||
        !device_ptr(o_o, "O", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &o) || !read_n_prev(np_o, d[0], &np) ||
        !read_where(stream, sync, &w))
        return nullptr;
    return finish(two ? "esa_attend_two_position" : "esa_attend", [&] {
        return w.sync ? esa_attend_two_position(self->h, (int32_t)d[0], q, qf, (int32_t)d[1], k, kf, v, np.v, (const int32_t*)idx,
                                                (const int32_t*)n_sel, o)
                      : esa_attend_two_position_async(self->h, (int32_t)d[0], q, qf, (int32_t)d[1], k, kf, v, np.v,
                                                      (const int32_t*)idx, (const int32_t*)n_sel, o, w.stream);
    });
}

// (Q_cur, K_cache, V_cache, n_prev, idx, n_sel, O, stream, sync)
PyObject* ctx_attend(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 9, "attend")) return nullptr;
    return attend_common(self, a[0], Py_None, a[1], Py_None, a[2], a[3], a[4], a[5], a[6], a[7], a[8], false);
}

PyObject* ctx_attend_two_position(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 11, "attend_two_position")) return nullptr;
    return attend_common(self, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], true);
}

bool pinned_ptr(PyObject* o, const char* name, std::initializer_list<int64_t> shape, void** out) {
    const at::Tensor* t = as_tensor(o, name);
    if (!t) return false;
    if (t->is_cuda() || !t->is_pinned()) {
        PyErr_Format(PyExc_TypeError, "%s must be a pinned host tensor", name);
        return false;
    }
    if (t->scalar_type() != kBf16 || !t->is_contiguous() || !has_shape(*t, shape.begin(), (int)shape.size())) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous bf16 [B, max_tokens, H_G, d]", name);
        return false;
    }
    *out = t->data_ptr();
    return true;
}

// (Q_cur, K_host, V_host, n_prev, idx, n_sel, K_stage, V_stage, O, stream, sync)
PyObject* ctx_attend_host_kv(CtxObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 11, "attend_host_kv")) return nullptr;
    const esa_config& c = self->cfg;
    int64_t d[2], sd[2];
    void *q, *k, *v, *idx, *n_sel, *ks, *vs, *o;
    NPrev np;
    Where w;
    if (!leading_sizes(a[0], "Q_cur", 2, d) || !device_ptr(a[0], "Q_cur", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &q) ||
        !pinned_ptr(a[1], "K_host", {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &k) ||
        !pinned_ptr(a[2], "V_host", {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &v) || !leading_sizes(a[6], "K_stage", 2, sd) ||
        !device_ptr(a[6], "K_stage", kBf16, {d[0], sd[1], c.n_kv_heads, c.head_dim}, &ks) ||
        !device_ptr(a[7], "V_stage", kBf16, {d[0], sd[1], c.n_kv_heads, c.head_dim}, &vs) ||
        !device_ptr(a[4], "idx", kI32, {d[0], c.top_k}, &idx) || !device_ptr(a[5], "n_sel", kI32, {d[0]}, &n_sel) ||
        !device_ptr(a[8], "O", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &o) || !read_n_prev(a[3], d[0], &np) ||
        !read_where(a[9], a[10], &w))
        return nullptr;
    return finish("esa_attend_host_kv", [&] {
        return w.sync ? esa_attend_host_kv(self->h, (int32_t)d[0], q, (int32_t)d[1], k, v, np.v, (const int32_t*)idx,
                                           (const int32_t*)n_sel, ks, vs, sd[1], o)
                      : esa_attend_host_kv_async(self->h, (int32_t)d[0], q, (int32_t)d[1], k, v, np.v, (const int32_t*)idx,
                                                 (const int32_t*)n_sel, ks, vs, sd[1], o, w.stream);
    });
}

// ------------------------------------------------------------------ calls without a context
// Fields of a binding.EsaConfig object, in the order of esa_config.
bool read_config(PyObject* o, esa_config* c) {
    auto get = [&](const char* name, long long* out) {
        PyObject* v = PyObject_GetAttrString(o, name);
        if (!v) return false;
        PyObject* i = PyNumber_Index(v);
        Py_DECREF(v);
        if (!i) return false;
        *out = PyLong_AsLongLong(i);
        Py_DECREF(i);
        return !(*out == -1 && PyErr_Occurred());
    };
    long long v[11];
    static const char* names[11] = {"n_q_heads", "n_kv_heads", "head_dim", "d_c", "l_init", "l_local", "top_k", "eps", "max_chunk",
                                    "max_batch", "max_tokens"};
    for (int i = 0; i < 11; ++i)
        if (!get(names[i], &v[i])) return false;
    c->n_q_heads = (int32_t)v[0]; c->n_kv_heads = (int32_t)v[1]; c->head_dim = (int32_t)v[2]; c->d_c = (int32_t)v[3];
    c->l_init = (int32_t)v[4]; c->l_local = (int32_t)v[5]; c->top_k = (int32_t)v[6]; c->eps = (int32_t)v[7];
    c->max_chunk = (int32_t)v[8]; c->max_batch = (int32_t)v[9]; c->max_tokens = v[10];
    PyObject* s = PyObject_GetAttrString(o, "softmax_scale");
    if (!s) return false;
    const double x = PyFloat_AsDouble(s);
    Py_DECREF(s);
    if (x == -1.0 && PyErr_Occurred()) return false;
    c->softmax_scale = (float)x;
    return true;
}

// (cfg, Q_cur, K_cache, V_cache, n_prev, idx, n_sel, O, stream)
PyObject* mod_attend_noalloc(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 9, "attend_noalloc")) return nullptr;
    esa_config c;
    int64_t d[2];
    void *q, *k, *v, *idx, *n_sel, *o, *stream;
    NPrev np;
    if (!read_config(a[0], &c) || !leading_sizes(a[1], "Q_cur", 2, d) ||
        !device_ptr(a[1], "Q_cur", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &q) ||
        !device_ptr(a[2], "K_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &k) ||
        !device_ptr(a[3], "V_cache", kBf16, {d[0], c.max_tokens, c.n_kv_heads, c.head_dim}, &v) ||
        !device_ptr(a[5], "idx", kI32, {d[0], c.top_k}, &idx) || !device_ptr(a[6], "n_sel", kI32, {d[0]}, &n_sel) ||
        !device_ptr(a[7], "O", kBf16, {d[0], d[1], c.n_q_heads, c.head_dim}, &o) || !read_n_prev(a[4], d[0], &np) ||
        !read_stream(a[8], &stream))
        return nullptr;
    return finish("esa_attend_noalloc", [&] {
        return esa_attend_noalloc(&c, (int32_t)d[0], q, (int32_t)d[1], k, v, np.v, (const int32_t*)idx, (const int32_t*)n_sel, o, stream);
    });
}

// (Q_batch, K_batch, loss_out | None, stream)
PyObject* fit_step(FitObject* self, PyObject* const* a, Py_ssize_t n) {
    if (!want_args(n, 4, "step")) return nullptr;
    const esa_config& c = self->cfg;
    int64_t d[1];
    void *q, *k, *loss = nullptr, *stream;
    if (!leading_sizes(a[0], "Q_batch", 1, d) || !device_ptr(a[0], "Q_batch", kBf16, {d[0], c.n_q_heads, c.head_dim}, &q) ||
        !device_ptr(a[1], "K_batch", kBf16, {d[0], c.n_kv_heads, c.head_dim}, &k) ||
        (a[2] != Py_None && !device_ptr(a[2], "loss_out", kF32, {1}, &loss)) || !read_stream(a[3], &stream))
        return nullptr;
    return finish("esa_fit_step_async", [&] { return esa_fit_step_async(self->h, q, k, (int32_t)d[0], (float*)loss, stream); });
}

// ------------------------------------------------------------------ types
// Ctx(handle, config) / Fit(handle, config): the handle stays owned by the Python object; drop() forgets it.
template <typename T>
int obj_init(PyObject* self, PyObject* args, PyObject*) {
    unsigned long long h = 0;
    PyObject* cfg = nullptr;
    if (!PyArg_ParseTuple(args, "KO", &h, &cfg)) return -1;
    T* t = reinterpret_cast<T*>(self);
    if (!read_config(cfg, &t->cfg)) return -1;
    t->h = reinterpret_cast<decltype(t->h)>((uintptr_t)h);
    return 0;
}

template <typename T>
PyObject* obj_drop(PyObject* self, PyObject*) {
    reinterpret_cast<T*>(self)->h = nullptr;
    Py_RETURN_NONE;
}

// A C++ exception must not leave a function that the interpreter has called (it would end the process).  torch throws where
// a tensor has no plain storage, sizes or layout to ask for -- sparse, fake, or wrapped by a transformation: these become the
// errors that its own Python methods raise.
template <typename Self, PyObject* (*F)(Self*, PyObject* const*, Py_ssize_t)>
PyObject* entry(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    try {
        return F(reinterpret_cast<Self*>(self), a, n);
    } catch (python_error& e) {
        e.restore();
    } catch (const c10::NotImplementedError& e) {
        PyErr_SetString(PyExc_NotImplementedError, e.what_without_backtrace());
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::bad_alloc&) {
        PyErr_NoMemory();
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

#define ESA_FAST(...) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(entry<__VA_ARGS__>))

PyMethodDef ctx_methods[] = {
    {"append_kv", ESA_FAST(CtxObject, ctx_append_kv), METH_FASTCALL, nullptr},
    {"compress_keys", ESA_FAST(CtxObject, ctx_compress_keys), METH_FASTCALL, nullptr},
    {"select", ESA_FAST(CtxObject, ctx_select), METH_FASTCALL, nullptr},
    {"select_full", ESA_FAST(CtxObject, ctx_select_full), METH_FASTCALL, nullptr},
    {"attend", ESA_FAST(CtxObject, ctx_attend), METH_FASTCALL, nullptr},
    {"attend_two_position", ESA_FAST(CtxObject, ctx_attend_two_position), METH_FASTCALL, nullptr},
    {"attend_host_kv", ESA_FAST(CtxObject, ctx_attend_host_kv), METH_FASTCALL, nullptr},
    {"drop", obj_drop<CtxObject>, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyMethodDef fit_methods[] = {
    {"step", ESA_FAST(FitObject, fit_step), METH_FASTCALL, nullptr},
    {"drop", obj_drop<FitObject>, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyType_Slot ctx_slots[] = {{Py_tp_init, reinterpret_cast<void*>(obj_init<CtxObject>)}, {Py_tp_methods, ctx_methods},
                           {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)}, {0, nullptr}};
PyType_Slot fit_slots[] = {{Py_tp_init, reinterpret_cast<void*>(obj_init<FitObject>)}, {Py_tp_methods, fit_methods},
                           {Py_tp_new, reinterpret_cast<void*>(PyType_GenericNew)}, {0, nullptr}};
PyType_Spec ctx_spec = {"_esa_native.Ctx", sizeof(CtxObject), 0, Py_TPFLAGS_DEFAULT, ctx_slots};
PyType_Spec fit_spec = {"_esa_native.Fit", sizeof(FitObject), 0, Py_TPFLAGS_DEFAULT, fit_slots};

PyObject* mod_set_error(PyObject*, PyObject* cls) {
    Py_XSETREF(g_error, Py_NewRef(cls));
    Py_RETURN_NONE;
}

PyMethodDef mod_methods[] = {
    {"attend_noalloc", ESA_FAST(PyObject, mod_attend_noalloc), METH_FASTCALL, nullptr},
    {"set_error", mod_set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef mod_def = {PyModuleDef_HEAD_INIT, "_esa_native", nullptr, -1, mod_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__esa_native(void) {
    PyObject* m = PyModule_Create(&mod_def);
    if (!m) return nullptr;
    PyObject* ctx_type = PyType_FromSpec(&ctx_spec);
    PyObject* fit_type = PyType_FromSpec(&fit_spec);
    if (!ctx_type || !fit_type || PyModule_AddObject(m, "Ctx", ctx_type) < 0 || PyModule_AddObject(m, "Fit", fit_type) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
