// Native half of binding.py: turns torch tensors and a cache description into the arguments of the C ABI and
// makes the call, without a Python-level loop over tensors and fields.
//
// Why it exists: a speculation round called straight from Python is bound by the host.  Marshalling through
// ctypes (a structure of twenty fields, a dtype / device / contiguity check and a pointer per tensor) took
// 15-20 us per call, several times the device time of the small calls (a draft call is 3-5 us, the
// controller's kernels 2 us); here the same checks are a few field reads on the tensor objects.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "spec_attn.h"

namespace {

// Attribute names of the cache description, interned once.
enum Name { K, V, LAYER_STRIDE, PAGE_STRIDE, HEAD_STRIDE, SLOT_STRIDE, N_LAYERS, PAGE_SIZE, PAGE_TABLE, MAX_PAGES, BATCH,
            N_Q_HEADS, N_KV_HEADS, HEAD_DIM, SM_SCALE, N_PAGES, FP8, K_SCALE, V_SCALE, N_NAMES };
const char* const kNames[N_NAMES] = {"k", "v", "layer_stride", "page_stride", "head_stride", "slot_stride", "n_layers",
                                     "page_size", "page_table", "max_pages", "batch", "n_q_heads", "n_kv_heads", "head_dim",
                                     "sm_scale", "n_pages", "fp8", "k_scale", "v_scale"};
PyObject* g_names[N_NAMES];

struct Ref {  // an owned reference
    PyObject* p;
    explicit Ref(PyObject* o) : p(o) {}
    ~Ref() { Py_XDECREF(p); }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
};

// The tensor behind a Python object, or null with TypeError set.
const at::Tensor* tensor_of(PyObject* o, const char* name)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s: expected a torch tensor", name);
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

// Device pointer of a contiguous CUDA tensor of the given type; false with an exception set otherwise.
bool dev_ptr(PyObject* o, at::ScalarType type, const char* name, void** out)
{
    const at::Tensor* t = tensor_of(o, name);
    if (!t) return false;
    if (!t->is_cuda()) {
        PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor (no CPU path exists)", name);
        return false;
    }
    if (t->scalar_type() != type || !t->is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s: expected contiguous %s, got %s%s", name, c10::toString(type),
                     c10::toString(t->scalar_type()), t->is_contiguous() ? "" : " (not contiguous)");
        return false;
    }
    *out = t->data_ptr();
    return true;
}
bool dev_ptr_or_none(PyObject* o, at::ScalarType type, const char* name, void** out)
{
    *out = nullptr;
    return o == Py_None || dev_ptr(o, type, name, out);
}

bool to_i64(PyObject* o, int64_t* out)
{
    *out = PyLong_AsLongLong(o);
    return *out != -1 || !PyErr_Occurred();
}
bool to_i32(PyObject* o, int32_t* out)
{
    int64_t x = 0;
    if (!to_i64(o, &x)) return false;
    if (x < INT32_MIN || x > INT32_MAX) {
        PyErr_SetString(PyExc_OverflowError, "value does not fit 32 bits");
        return false;
    }
    *out = (int32_t)x;
    return true;
}
bool to_f32(PyObject* o, float* out)
{
    const double x = PyFloat_AsDouble(o);
    *out = (float)x;
    return x != -1.0 || !PyErr_Occurred();
}

bool attr_i64(PyObject* kv, Name n, int64_t* out)
{
    Ref a(PyObject_GetAttr(kv, g_names[n]));
    return a.p && to_i64(a.p, out);
}
bool attr_i32(PyObject* kv, Name n, int32_t* out)
{
    Ref a(PyObject_GetAttr(kv, g_names[n]));
    return a.p && to_i32(a.p, out);
}
// an attribute that a description may lack: a new reference, or null (no exception) where it is missing
PyObject* optional_attr(PyObject* kv, Name n)
{
    PyObject* a = PyObject_GetAttr(kv, g_names[n]);
    if (!a && PyErr_ExceptionMatches(PyExc_AttributeError)) PyErr_Clear();
    return a;
}

// spec_kv_t of a KVCache-like object (same fields and checks as binding._kv_struct)
bool kv_of(PyObject* kv, spec_kv_t* s)
{
    bool fp8 = false;
    {
        Ref a(optional_attr(kv, FP8));
        if (!a.p && PyErr_Occurred()) return false;
        const int truth = a.p ? PyObject_IsTrue(a.p) : 0;
        if (truth < 0) return false;
        fp8 = truth != 0;
    }
    const at::ScalarType type = fp8 ? at::kByte : at::kBFloat16;
    void* p = nullptr;
    {
        Ref a(PyObject_GetAttr(kv, g_names[K]));
        if (!a.p || !dev_ptr(a.p, type, "kv.k", &p)) return false;
        s->k = p;
    }
    {
        Ref a(PyObject_GetAttr(kv, g_names[V]));
        if (!a.p || !dev_ptr(a.p, type, "kv.v", &p)) return false;
        s->v = p;
    }
    {
        Ref a(PyObject_GetAttr(kv, g_names[PAGE_TABLE]));
        if (!a.p || !dev_ptr_or_none(a.p, at::kInt, "kv.page_table", &p)) return false;
        s->page_table = static_cast<const int32_t*>(p);
    }
    if (!attr_i64(kv, LAYER_STRIDE, &s->layer_stride) || !attr_i64(kv, PAGE_STRIDE, &s->page_stride) ||
        !attr_i64(kv, HEAD_STRIDE, &s->head_stride) || !attr_i64(kv, SLOT_STRIDE, &s->slot_stride) ||
        !attr_i32(kv, N_LAYERS, &s->n_layers) || !attr_i32(kv, PAGE_SIZE, &s->page_size) ||
        !attr_i32(kv, MAX_PAGES, &s->max_pages) || !attr_i32(kv, BATCH, &s->batch) ||
        !attr_i32(kv, N_Q_HEADS, &s->n_q_heads) || !attr_i32(kv, N_KV_HEADS, &s->n_kv_heads) ||
        !attr_i32(kv, HEAD_DIM, &s->head_dim))
        return false;
    {
        Ref a(PyObject_GetAttr(kv, g_names[SM_SCALE]));
        if (!a.p) return false;
        s->sm_scale = 0.f;
        if (a.p != Py_None && !to_f32(a.p, &s->sm_scale)) return false;
    }
    {
        Ref a(optional_attr(kv, N_PAGES));
        if (!a.p && PyErr_Occurred()) return false;
        s->n_pages = 0;
        if (a.p && a.p != Py_None && !to_i32(a.p, &s->n_pages)) return false;
    }
    s->kv_dtype = fp8 ? SPEC_KV_FP8_E4M3 : SPEC_KV_BF16;
    s->k_scale = s->v_scale = nullptr;
    if (fp8) {
        Ref a(optional_attr(kv, K_SCALE));
        if (!a.p && PyErr_Occurred()) return false;
        if (a.p && a.p != Py_None) {
            if (!dev_ptr(a.p, at::kFloat, "kv.k_scale", &p)) return false;
            s->k_scale = static_cast<const float*>(p);
            Ref b(PyObject_GetAttr(kv, g_names[V_SCALE]));
            if (!b.p || !dev_ptr(b.p, at::kFloat, "kv.v_scale", &p)) return false;
            s->v_scale = static_cast<const float*>(p);
        }
    }
    return true;
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

bool want_args(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

// The call itself, without the interpreter lock: a launch that waits for room in a full queue must not stop the other
// Python threads.  What needs the lock happens before; the caller's arguments keep the tensors alive meanwhile.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    Unlocked() = default;
    ~Unlocked() { PyEval_RestoreThread(state); }
    Unlocked(const Unlocked&) = delete;
    Unlocked& operator=(const Unlocked&) = delete;
};
template <typename F>
PyObject* unlocked(F f)
{
    int rc = 0;
    {
        Unlocked u;
        rc = f();
    }
    return PyLong_FromLong(rc);
}

// A C++ exception (a stream query on a machine without a driver) becomes a Python one.
template <typename F>
PyObject* guarded(F f)
{
    try {
        return f();
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// verify(kv, q, ctx_len, max_ctx_len, stat_window, out, lse, stats, stat_stride, workspace, flags, score_hist)
PyObject* verify(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 12)) return nullptr;
    return guarded([&]() -> PyObject* {
        spec_kv_t s;
        void *q, *ctx, *out, *lse, *stats, *hist;
        int32_t max_ctx, window;
        int64_t flags, stride;
        if (!kv_of(a[0], &s) || !to_i64(a[10], &flags) || !to_i64(a[8], &stride) || !dev_ptr(a[1], at::kBFloat16, "q", &q) ||
            !dev_ptr(a[2], at::kInt, "ctx_len", &ctx) || !to_i32(a[3], &max_ctx) || !to_i32(a[4], &window) ||
            !dev_ptr(a[5], (flags & SPEC_VERIFY_OUT_BF16) ? at::kBFloat16 : at::kFloat, "out", &out) ||
            !dev_ptr_or_none(a[6], at::kFloat, "lse", &lse) || !dev_ptr(a[7], at::kFloat, "stats", &stats))
            return nullptr;
        const at::Tensor& tq = THPVariable_Unpack(a[1]);
        const at::Tensor& ts = THPVariable_Unpack(a[7]);
        if (tq.dim() != 5) {
            PyErr_SetString(PyExc_ValueError, "q: expected [layers, batch, n_q, n_q_heads, head_dim]");
            return nullptr;
        }
        const int64_t heads = (flags & SPEC_VERIFY_STATS_PER_QUERY_HEAD) ? s.n_q_heads : s.n_kv_heads;
        if (ts.dim() != 4 || ts.size(2) != heads) {
            PyErr_SetString(PyExc_ValueError, "stats: wrong head count for this mode");
            return nullptr;
        }
        if (!dev_ptr_or_none(a[11], at::kInt, "score_hist", &hist)) return nullptr;
        if (hist) {
            const at::Tensor& th = THPVariable_Unpack(a[11]);
            if (th.dim() != 4 || th.size(0) != ts.size(0) || th.size(1) != ts.size(1) || th.size(2) != ts.size(2) ||
                th.size(3) != 2048) {
                PyErr_SetString(PyExc_ValueError, "score_hist: expected [L, B, heads, 2048]");
                return nullptr;
            }
        }
        const at::Tensor* ws = tensor_of(a[9], "workspace");
        if (!ws) return nullptr;
        void* const st = stream();
        return unlocked([&] {
            return spec_verify_attn_hist(
                &s, q, (int32_t)tq.size(2), static_cast<const int32_t*>(ctx), max_ctx, window, static_cast<float*>(out),
                static_cast<float*>(lse), static_cast<float*>(stats), stride, ws->data_ptr(), (size_t)ws->numel(),
                (uint32_t)flags, static_cast<uint32_t*>(hist), st);
        });
    });
}

// select(stats, sel_len, k_sink, k_recent, k_total, indices, n_indices, score_hist, hist_len)
PyObject* select(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 9)) return nullptr;
    return guarded([&]() -> PyObject* {
        void *stats, *len, *idx, *cnt, *hist, *hlen;
        int32_t sink, recent, total;
        if (!dev_ptr(a[0], at::kFloat, "stats", &stats) || !dev_ptr(a[1], at::kInt, "sel_len", &len) ||
            !to_i32(a[2], &sink) || !to_i32(a[3], &recent) || !to_i32(a[4], &total) ||
            !dev_ptr(a[5], at::kInt, "indices", &idx) || !dev_ptr(a[6], at::kInt, "n_indices", &cnt) ||
            !dev_ptr_or_none(a[7], at::kInt, "score_hist", &hist))
            return nullptr;
        if (hist ? !dev_ptr(a[8], at::kInt, "hist_len", &hlen) : (hlen = nullptr, false)) return nullptr;
        const at::Tensor& t = THPVariable_Unpack(a[0]);
        if (t.dim() != 4) {
            PyErr_SetString(PyExc_ValueError, "stats: expected [layers, batch, heads, stride]");
            return nullptr;
        }
        void* const st = stream();
        return unlocked([&] {
            return spec_select_recall_hist(
                static_cast<const float*>(stats), t.size(3), (int32_t)t.size(0), (int32_t)t.size(1), (int32_t)t.size(2),
                static_cast<const int32_t*>(len), sink, recent, total, static_cast<int32_t*>(idx), static_cast<int32_t*>(cnt),
                static_cast<uint32_t*>(hist), static_cast<const int32_t*>(hlen), nullptr, 0, st);
        });
    });
}

// draft(kv, q, indices, n_indices, tail_start, cur_len, max_tail, out, lse, workspace, flags)
PyObject* draft(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 11)) return nullptr;
    return guarded([&]() -> PyObject* {
        spec_kv_t s;
        void *q, *idx, *cnt, *ts, *cl, *out, *lse;
        int32_t max_tail;
        int64_t flags;
        if (!kv_of(a[0], &s) || !to_i64(a[10], &flags) || !dev_ptr(a[1], at::kBFloat16, "q", &q) ||
            !dev_ptr(a[2], at::kInt, "indices", &idx) || !dev_ptr(a[3], at::kInt, "n_indices", &cnt) ||
            !dev_ptr(a[4], at::kInt, "tail_start", &ts) || !dev_ptr(a[5], at::kInt, "cur_len", &cl) ||
            !to_i32(a[6], &max_tail) ||
            !dev_ptr(a[7], (flags & SPEC_DRAFT_OUT_BF16) ? at::kBFloat16 : at::kFloat, "out", &out) ||
            !dev_ptr_or_none(a[8], at::kFloat, "lse", &lse))
            return nullptr;
        const at::Tensor& ti = THPVariable_Unpack(a[2]);
        const int64_t heads = (flags & SPEC_DRAFT_INDICES_PER_QUERY_HEAD) ? s.n_q_heads : s.n_kv_heads;
        if (ti.dim() != 4 || ti.size(2) != heads) {
            PyErr_SetString(PyExc_ValueError, "indices: wrong head count for this mode");
            return nullptr;
        }
        const at::Tensor* ws = tensor_of(a[9], "workspace");
        if (!ws) return nullptr;
        void* const st = stream();
        return unlocked([&] {
            return spec_sparse_draft_attn_ex(
                &s, q, static_cast<const int32_t*>(idx), static_cast<const int32_t*>(cnt), (int32_t)ti.size(3),
                static_cast<const int32_t*>(ts), static_cast<const int32_t*>(cl), max_tail, static_cast<float*>(out),
                static_cast<float*>(lse), ws->data_ptr(), (size_t)ws->numel(), (uint32_t)flags, st);
        });
    });
}

// Logits of `dim` dimensions on the device, fp32 or bf16; false with ValueError set otherwise.
const at::Tensor* logits_of(PyObject* o, int64_t dim, bool contiguous, const char* what)
{
    const at::Tensor* t = tensor_of(o, "logits");
    if (!t) return nullptr;
    if (!t->is_cuda() || t->dim() != dim || (contiguous ? !t->is_contiguous() : t->stride(dim - 1) != 1)) {
        PyErr_Format(PyExc_ValueError, "logits: expected a %s", what);
        return nullptr;
    }
    if (t->scalar_type() != at::kFloat && t->scalar_type() != at::kBFloat16) {
        PyErr_Format(PyExc_ValueError, "logits: expected fp32 or bf16, got %s", c10::toString(t->scalar_type()));
        return nullptr;
    }
    return t;
}

// rows(logits, token, entropy): token None = entropy only
PyObject* rows(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 3)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor* t = logits_of(a[0], 2, false, "CUDA [rows, vocab] tensor with unit inner stride");
        void *token, *entropy;
        if (!t || !dev_ptr_or_none(a[1], at::kInt, "token", &token) ||
            !dev_ptr_or_none(a[2], at::kFloat, "entropy", &entropy))
            return nullptr;
        const int32_t dt = t->scalar_type() == at::kBFloat16 ? 1 : 0, r = (int32_t)t->size(0), v = (int32_t)t->size(1);
        // a single row's stride says nothing
        const int64_t stride = (a[1] != Py_None || r <= 1) ? std::max(t->stride(0), t->size(1)) : t->stride(0);
        void* const st = stream();
        return unlocked([&] {
            return a[1] == Py_None
                       ? spec_token_entropy(t->data_ptr(), dt, r, v, stride, static_cast<float*>(entropy), st)
                       : spec_token_argmax(t->data_ptr(), dt, r, v, stride, static_cast<int32_t*>(token),
                                           static_cast<float*>(entropy), st);
        });
    });
}

// accept(logits, draft, n_draft, target, n_accepted, next_token)
PyObject* accept(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 6)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor* t = logits_of(a[0], 3, true, "contiguous CUDA [batch, k + 1, vocab] tensor");
        void *draft_p = nullptr, *nd, *target, *acc, *next;
        if (!t || (t->size(1) > 1 && !dev_ptr(a[1], at::kInt, "draft", &draft_p)) ||
            !dev_ptr_or_none(a[2], at::kInt, "n_draft", &nd) || !dev_ptr(a[3], at::kInt, "target", &target) ||
            !dev_ptr(a[4], at::kInt, "n_accepted", &acc) || !dev_ptr(a[5], at::kInt, "next_token", &next))
            return nullptr;
        const int32_t vocab = (int32_t)t->size(2);
        void* const st = stream();
        return unlocked([&] {
            return spec_accept_greedy(
                t->data_ptr(), t->scalar_type() == at::kBFloat16 ? 1 : 0, (int32_t)t->size(0), (int32_t)t->size(1), vocab, vocab,
                static_cast<const int32_t*>(draft_p), static_cast<const int32_t*>(nd), static_cast<int32_t*>(target),
                static_cast<int32_t*>(acc), static_cast<int32_t*>(next), st);
        });
    });
}

// advance(committed, n_accepted, k, ctx_verify, cur_len, max_len, workspace)
PyObject* advance(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 7)) return nullptr;
    return guarded([&]() -> PyObject* {
        void *committed, *acc, *ctx, *cur, *ws = nullptr;
        int32_t k, max_len;
        if (!dev_ptr(a[0], at::kInt, "committed", &committed) || !dev_ptr_or_none(a[1], at::kInt, "n_accepted", &acc) ||
            !to_i32(a[2], &k) || !to_i32(a[5], &max_len))
            return nullptr;
        if (a[6] != Py_None) {
            const at::Tensor* t = tensor_of(a[6], "workspace");
            if (!t) return nullptr;
            ws = t->data_ptr();
        }
        if (!dev_ptr_or_none(a[3], at::kInt, "ctx_verify", &ctx) || !dev_ptr_or_none(a[4], at::kInt, "cur_len", &cur))
            return nullptr;
        void* const st = stream();
        return unlocked([&] {
            return spec_advance_lengths(
                static_cast<int32_t*>(committed), static_cast<const int32_t*>(acc), (int32_t)THPVariable_Unpack(a[0]).numel(), k,
                max_len, ws, static_cast<int32_t*>(ctx), static_cast<int32_t*>(cur), st);
        });
    });
}

// controller_update(state, entropy, n_accepted, beta)
PyObject* controller_update(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 4)) return nullptr;
    return guarded([&]() -> PyObject* {
        void *state, *entropy, *acc;
        float beta;
        if (!dev_ptr(a[0], at::kFloat, "state", &state) || !dev_ptr(a[1], at::kFloat, "entropy", &entropy) ||
            !dev_ptr(a[2], at::kInt, "n_accepted", &acc) || !to_f32(a[3], &beta))
            return nullptr;
        void* const st = stream();
        return unlocked([&] {
            return spec_controller_update(static_cast<float*>(state), static_cast<const float*>(entropy),
                                                          (int32_t)THPVariable_Unpack(a[1]).numel(),
                                                          static_cast<const int32_t*>(acc), beta, st);
        });
    });
}

// controller_select(state, entropy, cand, c_d, c_v, k_star, p, score)
PyObject* controller_select(PyObject*, PyObject* const* a, Py_ssize_t n)
{
    if (!want_args(n, 8)) return nullptr;
    return guarded([&]() -> PyObject* {
        void *state, *entropy, *cand, *k_star, *p, *score;
        float c_d, c_v;
        if (!dev_ptr(a[0], at::kFloat, "state", &state) || !dev_ptr(a[1], at::kFloat, "entropy", &entropy) ||
            !dev_ptr(a[2], at::kInt, "cand", &cand) || !to_f32(a[3], &c_d) || !to_f32(a[4], &c_v) ||
            !dev_ptr(a[5], at::kInt, "k_star", &k_star) || !dev_ptr(a[6], at::kFloat, "p", &p) ||
            !dev_ptr(a[7], at::kFloat, "score", &score))
            return nullptr;
        void* const st = stream();
        return unlocked([&] {
            return spec_controller_select(
                static_cast<const float*>(state), static_cast<const float*>(entropy), (int32_t)THPVariable_Unpack(a[1]).numel(),
                static_cast<const int32_t*>(cand), (int32_t)THPVariable_Unpack(a[2]).numel(), c_d, c_v,
                static_cast<int32_t*>(k_star), static_cast<float*>(p), static_cast<float*>(score), st);
        });
    });
}

#define SPEC_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {SPEC_METHOD(verify), SPEC_METHOD(select), SPEC_METHOD(draft), SPEC_METHOD(rows), SPEC_METHOD(accept),
                          SPEC_METHOD(advance), SPEC_METHOD(controller_update), SPEC_METHOD(controller_select),
                          {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_spec_native", "Argument marshalling of the spec_attn C ABI.", -1, kMethods,
                       nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__spec_native(void)
{
    for (int i = 0; i < N_NAMES; ++i)
        if (!(g_names[i] = PyUnicode_InternFromString(kNames[i]))) return nullptr;
    PyObject* m = PyModule_Create(&kModule);
    if (m && PyModule_AddStringConstant(m, "abi", SPEC_NATIVE_ABI) != 0) {  // see build.py
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
