// The calls of paper_2604_08971_b200.Sentry that a serving loop makes, from Python objects to the C ABI of libsentry
// (include/sentry.h) in native code: tensor checks, pointers, descriptors, workspace size and the current stream.  What is
// left in Python is the signature and the allocation of outputs that the caller did not bring.
//
// A small call is bound by this path: a launch takes about 2.2 us of host time, and marshalling through ctypes took 12 us
// per call (the current stream's Python object alone 3 us, 0.2 us per tensor).  Host time of a step of three calls and four
// launches: 49 us through ctypes, 19 here; of the deployment pass of five calls: 68 us and 35.
//
// Every function takes (owner, context handle, workspace bytes, ...): owner.ensure_workspace(n) is called when the call
// needs more than the given size.  The GIL is released around the library call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <string>
#include <type_traits>

#include "../../include/sentry.h"

namespace {

PyObject* g_error = nullptr;   // SentryError(code, what)

struct Raised {};              // a Python exception is set
[[noreturn]] void raise(PyObject* type, const std::string& text) {
    PyErr_SetString(type, text.c_str());
    throw Raised{};
}
[[noreturn]] void raise_status(int rc, const char* what) {
    PyObject* e = g_error ? PyObject_CallFunction(g_error, "is", rc, what) : nullptr;
    if (e != nullptr) {
        PyErr_SetObject((PyObject*)Py_TYPE(e), e);
        Py_DECREF(e);
    } else if (!PyErr_Occurred()) {
        PyErr_Format(PyExc_RuntimeError, "%s failed (%d)", what, rc);
    }
    throw Raised{};
}
void require(bool ok, const char* what) {
    if (!ok) raise(PyExc_AssertionError, what);
}

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string("expected a tensor, got ") + Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}
const at::Tensor& tensor(PyObject* o, int dims) {
    const at::Tensor& t = tensor(o);
    if (t.dim() != dims) raise(PyExc_ValueError, "expected a tensor of " + std::to_string(dims) + " dimensions, got " + std::to_string(t.dim()));
    return t;
}
// Device address of a contiguous device tensor; None is a null pointer.
template <typename T = void>
T* ptr(const at::Tensor& t) {
    if (!t.is_cuda()) raise(PyExc_ValueError, "libsentry takes device tensors (got a " + t.device().str() + " tensor)");
    if (!t.is_contiguous()) raise(PyExc_ValueError, "libsentry takes contiguous tensors");
    return (T*)t.data_ptr();
}
template <typename T = void>
T* ptr(PyObject* o) {
    return o == Py_None ? nullptr : ptr<T>(tensor(o));
}
// The caller's output, or a fresh one beside `like` (from native code: half the time of torch.empty).
at::Tensor output(PyObject* o, at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) {
    return o != Py_None ? tensor(o) : at::empty(shape, like.options().dtype(type));
}
int dtype_code(const at::Tensor& t) {
    switch (t.scalar_type()) {
        case at::kFloat: return SENTRY_F32;
        case at::kBFloat16: return SENTRY_BF16;
        case at::kHalf: return SENTRY_F16;
        default: raise(PyExc_ValueError, std::string("unsupported dtype ") + c10::toString(t.scalar_type()));
    }
}
long long integer(PyObject* o) {
    if (!PyLong_Check(o)) {
        PyObject* n = PyNumber_Long(o);
        if (n == nullptr) throw Raised{};
        const long long v = PyLong_AsLongLong(n);
        Py_DECREF(n);
        if (v == -1 && PyErr_Occurred()) throw Raised{};
        return v;
    }
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return v;
}
int small(PyObject* o) { return (int)integer(o); }
float real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised{};
    return (float)v;
}
void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }

struct Call {
    PyObject* const* a;   // arguments after the three common ones
    PyObject* owner;
    sentry_ctx* ctx;
    long long ws;
    Call(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : a(args + 3), owner(args[0]) {
        if (n != want + 3) raise(PyExc_TypeError, "wrong number of arguments");
        ctx = (sentry_ctx*)(uintptr_t)(args[1] == Py_None ? 0 : integer(args[1]));
        ws = integer(args[2]);
    }
    void workspace(size_t bytes) {
        if ((long long)bytes <= ws) return;
        PyObject* r = PyObject_CallMethod(owner, "ensure_workspace", "n", (Py_ssize_t)bytes);
        if (r == nullptr) throw Raised{};
        Py_DECREF(r);
    }
};

// Runs body(call) and turns what it throws into a Python exception.
template <typename F>
PyObject* guarded(PyObject* const* args, Py_ssize_t n, Py_ssize_t want, F body) {
    try {
        Call c(args, n, want);
        if constexpr (std::is_void_v<decltype(body(c))>) {
            body(c);
            Py_RETURN_NONE;
        } else {
            return THPVariable_Wrap(body(c));   // the output
        }
    } catch (const Raised&) {
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}
// The library call itself, without the GIL.
template <typename F>
void invoke(const char* what, F f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    if (rc != SENTRY_OK) raise_status(rc, what);
}
#define METHOD(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t n)

// ------------------------------------------------------------------------------------------ gate
METHOD(gate_select) {   // scores, masks, k, kept, groups, heads_per_group
    return guarded(args, n, 6, [](Call& c) -> at::Tensor {
        const at::Tensor& scores = tensor(c.a[0], 2);
        const at::Tensor& masks = tensor(c.a[1]);
        require(scores.scalar_type() == at::kFloat && (masks.scalar_type() == at::kInt || masks.scalar_type() == at::kUInt32),
                "gate_select: fp32 scores and 32-bit masks");
        const int S = (int)scores.size(0), units = (int)scores.size(1), k = small(c.a[2]), n_masks = (int)masks.size(0);
        c.workspace(std::max<size_t>(1u << 20, (size_t)S * std::max(k, 0) * 4 + (size_t)S * 4 + 1024));
        const float* sc = ptr<float>(c.a[0]);
        const uint32_t* m = ptr<uint32_t>(c.a[1]);
        at::Tensor out = output(c.a[3], {n_masks, k}, at::kInt, scores);
        int32_t* kept = ptr<int32_t>(out);
        uint32_t* groups = ptr<uint32_t>(c.a[4]);
        const int hpg = small(c.a[5]);
        void* st = stream();
        invoke("sentry_gate_select", [&] { return sentry_gate_select(c.ctx, sc, S, units, m, n_masks, k, kept, groups, hpg, st); });
        return out;
    });
}
METHOD(gate_select_multi) {   // list of (scores, masks, k, heads_per_group, kept, groups)
    return guarded(args, n, 1, [](Call& c) {
        const Py_ssize_t sets = PyList_Check(c.a[0]) ? PyList_GET_SIZE(c.a[0]) : -1;
        if (sets < 1) raise(PyExc_TypeError, "gate_select_multi: a list of sets");
        if (sets > SENTRY_GATE_MAX_SETS) raise_status(SENTRY_ERR_BAD_SHAPE, "sentry_gate_select_multi");
        sentry_gate_set g[SENTRY_GATE_MAX_SETS];
        int S = 0;
        size_t need = 1024;
        for (Py_ssize_t i = 0; i < sets; ++i) {
            PyObject* item = PyList_GET_ITEM(c.a[0], i);
            if (!PyTuple_Check(item) || PyTuple_GET_SIZE(item) != 6) raise(PyExc_TypeError, "gate_select_multi: a set is a 6-tuple");
            PyObject** s = &PyTuple_GET_ITEM(item, 0);
            const at::Tensor& scores = tensor(s[0], 2);
            if (i == 0) S = (int)scores.size(0);
            require((int)scores.size(0) == S && scores.scalar_type() == at::kFloat, "gate_select_multi: fp32 scores of one S");
            g[i].scores = ptr<float>(s[0]);
            g[i].n_units = (int)scores.size(1);
            g[i].k = small(s[2]);
            g[i].masks = ptr<uint32_t>(s[1]);
            g[i].n_masks = (int)tensor(s[1]).size(0);
            g[i].kept = ptr<int32_t>(s[4]);
            g[i].kv_groups = ptr<uint32_t>(s[5]);
            g[i].heads_per_group = small(s[3]);
            need += (size_t)S * std::max(g[i].k, 0) * 4 + (size_t)S * 4 + 512;
        }
        c.workspace(std::max<size_t>(1u << 20, need));
        void* st = stream();
        invoke("sentry_gate_select_multi", [&] { return sentry_gate_select_multi(c.ctx, S, g, (int)sets, st); });
    });
}
METHOD(gate_eval) {   // layer_offsets, zeta, gamma, W1, b1, w2, b2, logits, gates
    return guarded(args, n, 9, [](Call& c) -> at::Tensor {
        const at::Tensor& W1 = tensor(c.a[3], 3);
        const int units = (int)W1.size(0), hidden = (int)W1.size(1), M = (int)W1.size(2), layers = (int)tensor(c.a[2]).size(0);
        const int32_t* off = ptr<int32_t>(c.a[0]);
        const float *zeta = ptr<float>(c.a[1]), *gamma = ptr<float>(c.a[2]), *w1 = ptr<float>(c.a[3]), *b1 = ptr<float>(c.a[4]),
                    *w2 = ptr<float>(c.a[5]), *b2 = ptr<float>(c.a[6]);
        at::Tensor out = output(c.a[7], {(int64_t)1 << std::min(M, 30), units}, at::kFloat, W1);
        float *logits = ptr<float>(out), *gates = ptr<float>(c.a[8]);
        void* st = stream();
        invoke("sentry_gate_eval", [&] {
            return sentry_gate_eval(c.ctx, M, hidden, layers, off, units, zeta, gamma, w1, b1, w2, b2, logits, gates, st);
        });
        return out;
    });
}
METHOD(gate_layer_counts) {   // kept, layer_offsets, counts
    return guarded(args, n, 3, [](Call& c) -> at::Tensor {
        const at::Tensor& kept = tensor(c.a[0], 2);
        const int n_masks = (int)kept.size(0), k = (int)kept.size(1), layers = (int)tensor(c.a[1]).size(0) - 1;
        const int32_t *kp = ptr<int32_t>(c.a[0]), *off = ptr<int32_t>(c.a[1]);
        at::Tensor out = output(c.a[2], {n_masks, layers}, at::kInt, kept);
        int32_t* counts = ptr<int32_t>(out);
        void* st = stream();
        invoke("sentry_gate_layer_counts", [&] { return sentry_gate_layer_counts(c.ctx, kp, n_masks, k, off, layers, counts, st); });
        return out;
    });
}

// ------------------------------------------------------------------------------------- attention
sentry_attend_desc attend_desc(PyObject* Q, PyObject* K, int k_h, int c, int score_mode) {
    const at::Tensor& q = tensor(Q, 4);
    sentry_attend_desc d;
    d.B = (int)q.size(0); d.Hq = (int)q.size(1); d.T = (int)q.size(2); d.d = (int)q.size(3);
    d.Hk = (int)tensor(K, 4).size(1);
    d.k_h = k_h; d.dtype = dtype_code(q); d.c = c; d.score_mode = score_mode;
    return d;
}
METHOD(gate_attend_fwd) {   // head_scores, k_h, Q, K, V, ids, masks, table, offsets, c, score_mode, O, kept_heads, active_out
    return guarded(args, n, 14, [](Call& c) {
        const sentry_attend_desc d = attend_desc(c.a[2], c.a[3], small(c.a[1]), small(c.a[9]), small(c.a[10]));
        const int S = (int)tensor(c.a[0]).size(0);
        c.workspace(std::max(sentry_workspace_bytes(&d, nullptr), (size_t)S * std::max(d.k_h, 0) * 4 + (size_t)S * 4 + 1024));
        const int subsets = c.a[8] == Py_None ? 0 : (int)tensor(c.a[8]).size(0);
        const float* sc = ptr<float>(c.a[0]);
        void *Q = ptr(c.a[2]), *K = ptr(c.a[3]), *V = ptr(c.a[4]), *O = ptr(c.a[11]);
        const int32_t *ids = ptr<int32_t>(c.a[5]), *tbl = ptr<int32_t>(c.a[7]);
        const uint32_t* masks = ptr<uint32_t>(c.a[6]);
        const int64_t* off = ptr<int64_t>(c.a[8]);
        int32_t *kept = ptr<int32_t>(c.a[12]), *act = ptr<int32_t>(c.a[13]);
        void* st = stream();
        invoke("sentry_gate_attend_fwd", [&] {
            return sentry_gate_attend_fwd(c.ctx, &d, sc, S, Q, K, V, ids, masks, tbl, off, subsets, O, kept, act, st);
        });
    });
}
METHOD(attend_fwd) {   // Q, K, V, kept_heads, ids, masks, table, offsets, c, score_mode, O, active_out, active_in
    return guarded(args, n, 13, [](Call& c) {
        const sentry_attend_desc d = attend_desc(c.a[0], c.a[1], (int)tensor(c.a[3], 2).size(1), small(c.a[8]), small(c.a[9]));
        const at::Tensor &K_ = tensor(c.a[1]), &V_ = tensor(c.a[2]);
        require(K_.sizes() == V_.sizes() && K_.scalar_type() == tensor(c.a[0]).scalar_type() && V_.scalar_type() == K_.scalar_type(),
                "attend_fwd: K and V of one shape, Q, K and V of one type");
        c.workspace(sentry_workspace_bytes(&d, nullptr));
        const int subsets = c.a[7] == Py_None ? 0 : (int)tensor(c.a[7]).size(0);
        void *Q = ptr(c.a[0]), *K = ptr(c.a[1]), *V = ptr(c.a[2]), *O = ptr(c.a[10]);
        const int32_t *kept = ptr<int32_t>(c.a[3]), *ids = ptr<int32_t>(c.a[4]), *tbl = ptr<int32_t>(c.a[6]);
        const uint32_t* masks = ptr<uint32_t>(c.a[5]);
        const int64_t* off = ptr<int64_t>(c.a[7]);
        int32_t *out = ptr<int32_t>(c.a[11]), *in = ptr<int32_t>(c.a[12]);
        void* st = stream();
        invoke("sentry_attend_fwd",
               [&] { return sentry_attend_fwd(c.ctx, &d, Q, K, V, kept, ids, masks, tbl, off, subsets, O, out, in, st); });
    });
}
METHOD(project_qkv) {   // X, WQ, WK, WV, kept_heads, ids, masks, Hq, Hk, d, Q, K, V
    return guarded(args, n, 13, [](Call& c) {
        const at::Tensor& X = tensor(c.a[0], 3);
        sentry_proj_desc d;
        d.B = (int)X.size(0); d.T = (int)X.size(1); d.D = (int)X.size(2);
        d.Hq = small(c.a[7]); d.Hk = small(c.a[8]); d.d = small(c.a[9]);
        d.k_h = (int)tensor(c.a[4], 2).size(1); d.dtype = dtype_code(X);
        void *x = ptr(c.a[0]), *wq = ptr(c.a[1]), *wk = ptr(c.a[2]), *wv = ptr(c.a[3]), *q = ptr(c.a[10]), *k = ptr(c.a[11]), *v = ptr(c.a[12]);
        const int32_t *kept = ptr<int32_t>(c.a[4]), *ids = ptr<int32_t>(c.a[5]);
        const uint32_t* masks = ptr<uint32_t>(c.a[6]);
        void* st = stream();
        invoke("sentry_project_qkv", [&] { return sentry_project_qkv(c.ctx, &d, x, wq, wk, wv, kept, ids, masks, q, k, v, st); });
    });
}
METHOD(project_out) {   // A, WO, kept_heads, ids, masks, Hq, out
    return guarded(args, n, 7, [](Call& c) {
        const at::Tensor& A = tensor(c.a[0], 4);
        sentry_proj_desc d;
        d.B = (int)A.size(0); d.k_h = (int)A.size(1); d.T = (int)A.size(2); d.d = (int)A.size(3);
        d.D = (int)tensor(c.a[1], 2).size(1); d.Hq = small(c.a[5]); d.Hk = 1; d.dtype = dtype_code(A);
        void *a = ptr(c.a[0]), *w = ptr(c.a[1]), *out = ptr(c.a[6]);
        const int32_t *kept = ptr<int32_t>(c.a[2]), *ids = ptr<int32_t>(c.a[3]);
        const uint32_t* masks = ptr<uint32_t>(c.a[4]);
        void* st = stream();
        invoke("sentry_project_out", [&] { return sentry_project_out(c.ctx, &d, a, w, kept, ids, masks, out, st); });
    });
}

// ------------------------------------------------------------------------------------------- FFN
sentry_ffn_desc ffn_desc(const at::Tensor& X, int F, int k_c, int lists, int dtype) {
    sentry_ffn_desc d;
    d.B = (int)X.size(0); d.T = (int)X.size(1); d.D = (int)X.size(2);
    d.F = F; d.k_c = k_c; d.n_lists = lists; d.dtype = dtype;
    return d;
}
// kept lists [n_lists, k_c] or one list [k_c]
void list_shape(const at::Tensor& kept, int& lists, int& k_c) {
    if (kept.dim() != 1 && kept.dim() != 2) raise(PyExc_ValueError, "kept channels: one list or [n_lists, k_c]");
    lists = kept.dim() == 1 ? 1 : (int)kept.size(0);
    k_c = (int)kept.size(-1);
}
METHOD(ffn_fwd) {   // X, W1, W2, kept_channels, list_of_sample, ids, masks, Y
    return guarded(args, n, 8, [](Call& c) {
        const at::Tensor &X = tensor(c.a[0], 3), &W1 = tensor(c.a[1], 2);
        int lists, k_c;
        list_shape(tensor(c.a[3]), lists, k_c);
        const sentry_ffn_desc d = ffn_desc(X, (int)W1.size(1), k_c, lists, dtype_code(X));
        require(W1.scalar_type() == X.scalar_type() && tensor(c.a[2]).scalar_type() == X.scalar_type(), "ffn_fwd: X, W1 and W2 of one type");
        c.workspace(sentry_workspace_bytes(nullptr, &d));
        void *x = ptr(c.a[0]), *w1 = ptr(c.a[1]), *w2 = ptr(c.a[2]), *y = ptr(c.a[7]);
        const int32_t *kept = ptr<int32_t>(c.a[3]), *los = ptr<int32_t>(c.a[4]), *ids = ptr<int32_t>(c.a[5]);
        const uint32_t* masks = ptr<uint32_t>(c.a[6]);
        void* st = stream();
        invoke("sentry_ffn_fwd", [&] { return sentry_ffn_fwd(c.ctx, &d, x, w1, w2, kept, los, ids, masks, y, st); });
    });
}
METHOD(ffn_fwd_packed) {   // X, packed, F, k_c, n_lists, list_of_sample, ids, masks, Y
    return guarded(args, n, 9, [](Call& c) {
        const at::Tensor& X = tensor(c.a[0], 3);
        const sentry_ffn_desc d = ffn_desc(X, small(c.a[2]), small(c.a[3]), small(c.a[4]), dtype_code(X));
        c.workspace(sentry_workspace_bytes(nullptr, &d));
        void *x = ptr(c.a[0]), *packed = ptr(c.a[1]), *y = ptr(c.a[8]);
        const int32_t *los = ptr<int32_t>(c.a[5]), *ids = ptr<int32_t>(c.a[6]);
        const uint32_t* masks = ptr<uint32_t>(c.a[7]);
        void* st = stream();
        invoke("sentry_ffn_fwd_packed", [&] { return sentry_ffn_fwd_packed(c.ctx, &d, x, packed, los, ids, masks, y, st); });
    });
}
METHOD(ffn_fwd_fp8) {   // Xq, packed, F, k_c, n_lists, scale_x, scale_w1, scale_w2, scale_h, list_of_sample, ids, masks, Y
    return guarded(args, n, 13, [](Call& c) {
        const at::Tensor& X = tensor(c.a[0], 3);
        const sentry_ffn_desc d = ffn_desc(X, small(c.a[2]), small(c.a[3]), small(c.a[4]), SENTRY_FP8_E4M3);
        sentry_ffn_desc d16 = d;
        d16.dtype = SENTRY_BF16;
        c.workspace(sentry_workspace_bytes(nullptr, &d16));
        void *x = ptr(c.a[0]), *packed = ptr(c.a[1]), *y = ptr(c.a[12]);
        const float sx = real(c.a[5]), s1 = real(c.a[6]), s2 = real(c.a[7]), sh = real(c.a[8]);
        const int32_t *los = ptr<int32_t>(c.a[9]), *ids = ptr<int32_t>(c.a[10]);
        const uint32_t* masks = ptr<uint32_t>(c.a[11]);
        void* st = stream();
        invoke("sentry_ffn_fwd_fp8", [&] { return sentry_ffn_fwd_fp8(c.ctx, &d, x, packed, los, ids, masks, sx, s1, s2, sh, y, st); });
    });
}
METHOD(ffn_prepack) {   // W1, W2, kept_channels, packed
    return guarded(args, n, 4, [](Call& c) -> at::Tensor {
        const at::Tensor& W1 = tensor(c.a[0], 2);
        sentry_ffn_desc d;
        d.B = d.T = 1; d.D = (int)W1.size(0); d.F = (int)W1.size(1); d.dtype = dtype_code(W1);
        list_shape(tensor(c.a[2]), d.n_lists, d.k_c);
        at::Tensor out = c.a[3] != Py_None ? tensor(c.a[3]) : output(c.a[3], {(int64_t)sentry_ffn_packed_bytes(&d)}, at::kByte, W1);
        void *w1 = ptr(c.a[0]), *w2 = ptr(c.a[1]), *packed = ptr(out);
        const int32_t* kept = ptr<int32_t>(c.a[2]);
        const size_t bytes = (size_t)out.numel();
        void* st = stream();
        invoke("sentry_ffn_prepack", [&] { return sentry_ffn_prepack(c.ctx, &d, w1, w2, kept, packed, bytes, st); });
        return out;
    });
}
METHOD(moe_ffn_fwd) {   // X, expert_ids, expert_weights, W1, W2, kept_channels, packed, F, E, k_c, Y
    return guarded(args, n, 11, [](Call& c) {
        const at::Tensor& X = tensor(c.a[0], 2);
        sentry_moe_desc d;
        d.N = (int)X.size(0); d.D = (int)X.size(1); d.F = small(c.a[7]); d.E = small(c.a[8]);
        d.top_k = (int)tensor(c.a[1], 2).size(1); d.k_c = small(c.a[9]); d.dtype = dtype_code(X);
        c.workspace(sentry_moe_workspace_bytes(&d));
        void *x = ptr(c.a[0]), *w1 = ptr(c.a[3]), *w2 = ptr(c.a[4]), *packed = ptr(c.a[6]), *y = ptr(c.a[10]);
        const int32_t *ids = ptr<int32_t>(c.a[1]), *kept = ptr<int32_t>(c.a[5]);
        const float* w = ptr<float>(c.a[2]);
        void* st = stream();
        invoke("sentry_moe_ffn_fwd", [&] { return sentry_moe_ffn_fwd(c.ctx, &d, x, w1, w2, kept, packed, ids, w, y, st); });
    });
}

PyObject* set_error(PyObject*, PyObject* cls) {
    Py_INCREF(cls);
    Py_XSETREF(g_error, cls);
    Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {ENTRY(gate_select), ENTRY(gate_select_multi), ENTRY(gate_eval), ENTRY(gate_layer_counts),
                           ENTRY(gate_attend_fwd), ENTRY(attend_fwd), ENTRY(project_qkv), ENTRY(project_out), ENTRY(ffn_fwd),
                           ENTRY(ffn_fwd_packed), ENTRY(ffn_fwd_fp8), ENTRY(ffn_prepack), ENTRY(moe_ffn_fwd),
                           {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&g_module); }
