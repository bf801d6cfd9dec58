// The Python binding's checks and argument marshalling, natively.
//
// Every function here takes the arguments of the binding's call of the same name (see
// __init__.py), makes the checks that call makes and, when they all pass, calls the
// library and returns its status.  When any check does not pass, or an argument is of a
// kind this file does not handle (a tensor subclass, pinned host memory), it returns None
// and enqueues nothing: the binding then does the same in Python, which words the error.
//
// Why: a call's checks and ctypes conversions took 10-14 us of Python for 2-5 us of
// launches, so a step of a small batch was bound by the host: batch 8 x 4k tokens through
// the separate calls took 74-78 us a step for 19 us of GPU time, 20 us now; batch 1 x 512
// 53 -> 19 us; batch 32 x 8k with attention ranking 70 -> 33 us.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <climits>
#include <cmath>
#include <cstring>

#include "pldp.h"

namespace {

// The library's calls, bound by address (bind()), so that this extension and ctypes use
// the one loaded library.
struct Library {
    decltype(&pldp_find_candidates) find_candidates;
    decltype(&pldp_rank_hidden) rank_hidden;
    decltype(&pldp_rank_attention) rank_attention;
    decltype(&pldp_extract_draft) extract_draft;
    decltype(&pldp_draft_step) draft_step;
    decltype(&pldp_index_build) index_build;
    decltype(&pldp_verify_greedy) verify_greedy;
    decltype(&pldp_verify_greedy_draft) verify_greedy_draft;
    decltype(&pldp_verify_sample) verify_sample;
    decltype(&pldp_verify_sample_draft) verify_sample_draft;
    decltype(&pldp_identify_heads) identify_heads;
    decltype(&pldp_top_heads) top_heads;
} lib;

#ifdef PLDP_TEST_ANY_DEVICE
constexpr bool kAnyDevice = true;    // test build: host tensors pass, so that the checks run without a GPU
#else
constexpr bool kAnyDevice = false;
#endif

// Reads arguments; `ok` goes false at the first one that is not what the call wants.
struct Args {
    bool ok = true;

    // A plain tensor (not a subclass), or null for None where that is allowed.
    const at::Tensor* tensor(PyObject* o, bool optional = false) {
        if (o == nullptr || o == Py_None) {
            if (!optional) ok = false;
            return nullptr;
        }
        if (!THPVariable_CheckExact(o)) {
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.defined() || !(kAnyDevice || t.is_cuda())) {
            ok = false;
            return nullptr;
        }
        return &t;
    }
    // The data of a contiguous tensor of at least n elements (n < 0: any count); null
    // for None where that is allowed.
    void* dense(PyObject* o, int64_t n, bool optional = false, c10::ScalarType type = at::kInt, bool any_type = false) {
        const at::Tensor* t = tensor(o, optional);
        if (!t) return nullptr;
        if (!t->is_contiguous() || (n >= 0 && t->numel() < n) || (!any_type && t->scalar_type() != type)) {
            ok = false;
            return nullptr;
        }
        return t->data_ptr();
    }
    int32_t* ints(PyObject* o, int64_t n, bool optional = false) { return static_cast<int32_t*>(dense(o, n, optional)); }
    float* floats(PyObject* o, int64_t n, bool optional = false) {
        return static_cast<float*>(dense(o, n, optional, at::kFloat));
    }
    uint32_t* words(PyObject* o, int64_t n, bool optional = true) {   // int32 or uint32
        const at::Tensor* t = tensor(o, optional);
        if (!t) return nullptr;
        if (!t->is_contiguous() || t->numel() < n || (t->scalar_type() != at::kInt && t->scalar_type() != at::kUInt32)) {
            ok = false;
            return nullptr;
        }
        return static_cast<uint32_t*>(t->data_ptr());
    }
    void* bytes(PyObject* o, size_t* size, bool optional = false) {
        const at::Tensor* t = tensor(o, optional);
        *size = 0;
        if (!t) return nullptr;
        if (!t->is_contiguous()) {
            ok = false;
            return nullptr;
        }
        *size = static_cast<size_t>(t->numel()) * t->element_size();
        return t->data_ptr();
    }
    int64_t integer(PyObject* o, int64_t lo = INT32_MIN, int64_t hi = INT32_MAX) {
        if (o == nullptr || !PyLong_CheckExact(o)) {
            ok = false;
            return 0;
        }
        int overflow = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &overflow);
        if (overflow || v < lo || v > hi) ok = false;
        return v;
    }
    float real(PyObject* o) {
        if (o == nullptr || !(PyFloat_CheckExact(o) || PyLong_CheckExact(o))) {
            ok = false;
            return 0.f;
        }
        const double v = PyFloat_AsDouble(o);
        if (v == -1.0 && PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return static_cast<float>(v);
    }
    pldp_dtype code(const at::Tensor* t) {
        if (t && t->scalar_type() == at::kFloat) return PLDP_F32;
        if (t && t->scalar_type() == at::kBFloat16) return PLDP_BF16;
        ok = false;
        return PLDP_F32;
    }
    // A [B, T] int32 tensor whose rows may be strided, with at least B rows (B < 0: its own
    // count); T_cap None or within its columns.
    struct Rows {
        int32_t* p = nullptr;
        int64_t stride = 0, T_cap = 0, B = 0;
    };
    Rows rows(PyObject* o, int64_t B, PyObject* T_cap) {
        Rows r;
        const at::Tensor* t = tensor(o);
        if (!t) return r;
        if (t->dim() != 2 || t->stride(1) != 1 || t->scalar_type() != at::kInt || (B >= 0 && t->size(0) < B)) {
            ok = false;
            return r;
        }
        r.p = static_cast<int32_t*>(t->data_ptr());
        r.stride = t->stride(0);
        r.B = t->size(0);
        r.T_cap = t->size(1);
        if (T_cap != nullptr && T_cap != Py_None) r.T_cap = integer(T_cap, 0, t->size(1));
        if (r.B > INT32_MAX) ok = false;
        return r;
    }
    // H [B, T_cap, d] with contiguous rows.
    const at::Tensor* hidden(PyObject* o) {
        const at::Tensor* t = tensor(o);
        if (t && (t->dim() != 3 || t->stride(2) != 1 || t->stride(1) != t->size(2))) ok = false;
        return ok ? t : nullptr;
    }
    const at::Tensor* dims3(PyObject* o) {
        const at::Tensor* t = tensor(o);
        if (t && t->dim() != 3) ok = false;
        return ok ? t : nullptr;
    }
    void* stream(PyObject* o) {
        if (o == nullptr || o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        if (PyLong_CheckExact(o)) {
            void* s = PyLong_AsVoidPtr(o);
            if (s != nullptr || !PyErr_Occurred()) return s;
            PyErr_Clear();                                     // out of range: Python's to take or to refuse
        }
        ok = false;                                            // a stream object, which Python unwraps
        return nullptr;
    }
    int cols(PyObject* o) {                                    // C_cap of a [B, C_cap] tensor
        const at::Tensor* t = tensor(o);
        if (!t || t->dim() != 2 || t->size(1) > INT32_MAX) {
            ok = false;
            return 0;
        }
        return static_cast<int>(t->size(1));
    }
};

// The interpreter's lock given up, and taken back however the scope is left.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};

// Makes the library's call without the interpreter's lock.  `call` holds values only:
// asking a tensor anything may raise (data_ptr() does for one without storage), and
// belongs to the checks before it.
template <typename F>
PyObject* finish(const Args& a, F call) {
    if (!a.ok) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
    pldp_status rc;
    {
        const Unlocked unlocked;
        rc = call();
    }
    return PyLong_FromLong(rc);
}

#define PLDP_CALL(name) PyObject* name(PyObject*, PyObject* const* v, Py_ssize_t n) noexcept
// An exception of the tensor library counts as a check that did not pass; the
// interpreter's lock is held wherever one can arise (see finish).
#define PLDP_BEGIN(count)              \
    if (n != (count)) Py_RETURN_NONE;  \
    try {                              \
        Args a;
#define PLDP_END                       \
    }                                  \
    catch (...) {                      \
        PyErr_Clear();                 \
        Py_RETURN_NONE;                \
    }

// ids, seq_len, ngram_min, ngram_max, cand_pos, cand_count, match_len, status, T_cap, stream
PLDP_CALL(find_candidates) {
    PLDP_BEGIN(10)
    const Args::Rows r = a.rows(v[0], -1, v[8]);
    const int C = a.cols(v[4]);
    const int32_t* L = a.ints(v[1], r.B);
    const int lo = static_cast<int>(a.integer(v[2])), hi = static_cast<int>(a.integer(v[3]));
    int32_t* cand = a.ints(v[4], r.B * C);
    int32_t* cnt = a.ints(v[5], r.B);
    int32_t* ml = a.ints(v[6], r.B);
    uint32_t* st = a.words(v[7], r.B);
    void* s = a.stream(v[9]);
    return finish(a, [&] {
        return lib.find_candidates(r.p, r.stride, L, static_cast<int>(r.B), r.T_cap, lo, hi, cand, C, cnt, ml, st, s);
    });
    PLDP_END
}

// H, seq_len, cand_pos, cand_count, best_pos, scores, best_score, threshold, status, stream
PLDP_CALL(rank_hidden) {
    PLDP_BEGIN(10)
    const at::Tensor* H = a.hidden(v[0]);
    if (!H) Py_RETURN_NONE;
    const void* h = H->data_ptr();
    const int64_t B = H->size(0), T_cap = H->size(1), d = H->size(2), stride = H->stride(0);
    const pldp_dtype code = a.code(H);
    const int C = a.cols(v[2]);
    const int32_t* L = a.ints(v[1], B);
    const int32_t* cand = a.ints(v[2], B * C);
    const int32_t* cnt = a.ints(v[3], B);
    int32_t* best = a.ints(v[4], B);
    float* sc = a.floats(v[5], B * C, true);
    float* bs = a.floats(v[6], B, true);
    const float thr = a.real(v[7]);
    uint32_t* st = a.words(v[8], B);
    void* s = a.stream(v[9]);
    if (B > INT32_MAX) a.ok = false;
    return finish(a, [&] {
        return lib.rank_hidden(h, code, d, stride, L, static_cast<int>(B), T_cap, cand, cnt, C, thr, sc, best, bs, st, s);
    });
    PLDP_END
}

// A, seq_len, cand_pos, cand_count, best_pos, row_idx, agg, scores, best_score, status, stream
PLDP_CALL(rank_attention) {
    PLDP_BEGIN(11)
    const at::Tensor* A = a.dims3(v[0]);
    if (!A) Py_RETURN_NONE;
    const void* rows = A->data_ptr();
    const int64_t B = A->size(0), R = A->size(1), T_cap = A->size(2);
    const int64_t row_stride = A->stride(1), key_stride = A->stride(2), seq_stride = A->stride(0);
    const pldp_dtype code = a.code(A);
    const int C = a.cols(v[2]);
    const int32_t* L = a.ints(v[1], B);
    const int32_t* cand = a.ints(v[2], B * C);
    const int32_t* cnt = a.ints(v[3], B);
    int32_t* best = a.ints(v[4], B);
    const int32_t* ri = a.ints(v[5], -1, true);
    const int64_t n_sel = ri ? THPVariable_Unpack(v[5]).numel() : R;
    const int agg = static_cast<int>(a.integer(v[6]));
    float* sc = a.floats(v[7], B * C, true);
    float* bs = a.floats(v[8], B, true);
    uint32_t* st = a.words(v[9], B);
    void* s = a.stream(v[10]);
    if (B > INT32_MAX || R > INT32_MAX || n_sel > INT32_MAX || (v[5] != Py_None && !ri)) a.ok = false;
    return finish(a, [&] {
        return lib.rank_attention(rows, code, static_cast<int>(R), row_stride, key_stride, seq_stride, ri,
                                  static_cast<int>(n_sel), static_cast<pldp_agg>(agg), L, static_cast<int>(B), T_cap, cand,
                                  cnt, C, sc, best, bs, st, s);
    });
    PLDP_END
}

// ids, seq_len, best_pos, draft, draft_len, T_cap, stream
PLDP_CALL(extract_draft) {
    PLDP_BEGIN(7)
    const at::Tensor* d = a.tensor(v[3]);
    if (!d || d->dim() != 2 || d->size(0) > INT32_MAX || d->size(1) > INT32_MAX) Py_RETURN_NONE;
    const int64_t B = d->size(0), K = d->size(1);
    const Args::Rows r = a.rows(v[0], B, v[5]);
    const int32_t* L = a.ints(v[1], B);
    const int32_t* best = a.ints(v[2], B);
    int32_t* draft = a.ints(v[3], B * K);
    int32_t* dl = a.ints(v[4], B);
    void* s = a.stream(v[6]);
    return finish(a, [&] {
        return lib.extract_draft(r.p, r.stride, L, r.T_cap, best, static_cast<int>(B), static_cast<int>(K), draft, dl, s);
    });
    PLDP_END
}

// The keyword arguments of the drafting calls, interned.
enum { kH, kBestH, kHScores, kBestHScore, kThreshold, kA, kBestA, kRowIdx, kAgg, kAScores, kBestAScore, kDraftFrom, kStatus,
       kTcap, kIndex, kV, kKeys };
const char* const kNames[kKeys] = {"H", "best_h", "h_scores", "best_h_score", "threshold", "A", "best_a", "row_idx", "agg",
                                   "a_scores", "best_a_score", "draft_from", "status", "T_cap", "index", "V"};
PyObject* names[kKeys];
PyObject *s_hidden, *s_attention;

// The argument block of pldp_draft_step from its positional arguments p[0 .. 10) = ids,
// seq_len, ngram_min, ngram_max, cand_pos, cand_count, match_len, K, draft, draft_len, the
// workspace (or null) and the keywords `kw`; index and V as given when not in `kw`.
void draft_args(Args& a, PyObject* const* p, PyObject* workspace, PyObject* kw, PyObject* index, int64_t V,
                pldp_draft_step_args& d) {
    PyObject* k[kKeys] = {};
    if (!PyDict_CheckExact(kw)) {
        a.ok = false;
        return;
    }
    Py_ssize_t found = 0;
    for (int i = 0; i < kKeys; ++i) {
        k[i] = PyDict_GetItemWithError(kw, names[i]);
        found += k[i] != nullptr;
    }
    if (found != PyDict_GET_SIZE(kw) || (index && (k[kIndex] || k[kV]))) {
        a.ok = false;                                          // a keyword the call does not have
        return;
    }
    auto given = [&](int i) { return k[i] != nullptr && k[i] != Py_None; };
    const Args::Rows r = a.rows(p[0], -1, k[kTcap]);
    const int64_t B = r.B;
    d.ids = r.p;
    d.ids_stride = r.stride;
    d.T_cap = r.T_cap;
    d.B = static_cast<int>(B);
    d.seq_len = a.ints(p[1], B);
    d.ngram_min = static_cast<int>(a.integer(p[2]));
    d.ngram_max = static_cast<int>(a.integer(p[3]));
    d.C_cap = a.cols(p[4]);
    d.cand_pos = a.ints(p[4], B * d.C_cap);
    d.cand_count = a.ints(p[5], B);
    d.match_len = a.ints(p[6], B);
    const int64_t K = a.integer(p[7]);
    d.K = static_cast<int>(K);
    d.draft = a.ints(p[8], B * K);
    d.draft_len = a.ints(p[9], B);
    if (K < 0) a.ok = false;
    if (given(kH)) {
        const at::Tensor* H = a.hidden(k[kH]);
        if (!H) return;
        if (H->size(0) < B || H->size(1) < r.T_cap) a.ok = false;
        d.H = H->data_ptr();
        d.h_dtype = a.code(H);
        d.d = H->size(2);
        d.h_seq_stride = H->stride(0);
        d.threshold = k[kThreshold] ? a.real(k[kThreshold]) : -INFINITY;
        d.h_scores = a.floats(k[kHScores], B * d.C_cap, true);
        d.best_h = a.ints(k[kBestH], B);
        d.best_h_score = a.floats(k[kBestHScore], B, true);
    }
    if (given(kA)) {
        const at::Tensor* A = a.dims3(k[kA]);
        if (!A) return;
        if (A->size(0) < B || A->size(2) < r.T_cap || A->size(1) > INT32_MAX) a.ok = false;
        d.A = A->data_ptr();
        d.a_dtype = a.code(A);
        d.R = static_cast<int>(A->size(1));
        d.a_row_stride = A->stride(1);
        d.a_key_stride = A->stride(2);
        d.a_seq_stride = A->stride(0);
        d.n_sel = d.R;
        if (given(kRowIdx)) {
            d.row_idx = a.ints(k[kRowIdx], -1);
            if (!d.row_idx) a.ok = false;
            if (!a.ok) return;
            const int64_t n_sel = THPVariable_Unpack(k[kRowIdx]).numel();
            if (n_sel > INT32_MAX) a.ok = false;
            d.n_sel = static_cast<int>(n_sel);
        }
        d.agg = static_cast<pldp_agg>(k[kAgg] ? a.integer(k[kAgg]) : static_cast<int64_t>(PLDP_AGG_MAX));
        d.a_scores = a.floats(k[kAScores], B * d.C_cap, true);
        d.best_a = a.ints(k[kBestA], B);
        d.best_a_score = a.floats(k[kBestAScore], B, true);
    }
    if (PyObject* f = k[kDraftFrom]) {
        if (PyUnicode_CheckExact(f)) {
            if (PyUnicode_Compare(f, s_attention) == 0) d.draft_from = 1;
            else if (PyUnicode_Compare(f, s_hidden) != 0) a.ok = false;
        } else {
            d.draft_from = static_cast<int>(a.integer(f, 0, 1));
        }
    }
    d.status = a.words(k[kStatus], B);
    if (workspace && workspace != Py_None) d.workspace = a.bytes(workspace, &d.workspace_bytes);
    if (!index && given(kIndex)) {
        index = k[kIndex];
        V = a.integer(k[kV]);
    }
    if (index) {
        d.index = a.bytes(index, &d.index_bytes);
        d.V = static_cast<int>(V);
        if (V < INT32_MIN || V > INT32_MAX) a.ok = false;
    }
}

// ids, seq_len, ngram_min, ngram_max, cand_pos, cand_count, match_len, K, draft, draft_len,
// workspace, stream, keywords
PLDP_CALL(draft_step) {
    PLDP_BEGIN(13)
    pldp_draft_step_args d = {};
    draft_args(a, v, v[10], v[12], nullptr, 0, d);
    void* s = a.stream(v[11]);
    return finish(a, [&] { return lib.draft_step(&d, s); });
    PLDP_END
}

// ids, seq_len, V, index, status, T_cap, stream
PLDP_CALL(index_build) {
    PLDP_BEGIN(7)
    const Args::Rows r = a.rows(v[0], -1, v[5]);
    const int32_t* L = a.ints(v[1], r.B);
    const int V = static_cast<int>(a.integer(v[2]));
    size_t size;
    void* ix = a.bytes(v[3], &size);
    uint32_t* st = a.words(v[4], r.B);
    void* s = a.stream(v[6]);
    return finish(a, [&] {
        return lib.index_build(r.p, r.stride, L, static_cast<int>(r.B), r.T_cap, V, ix, size, st, s);
    });
    PLDP_END
}

// The logits of a verification [B, K + 1, V] and what every form of it shares.
struct Logits {
    void* p = nullptr;
    pldp_dtype code = PLDP_F32;
    int64_t B = 0, K = 0, V = 0;
};
Logits logits(Args& a, PyObject* o, PyObject* draft) {
    Logits l;
    const at::Tensor* t = a.tensor(o);
    const at::Tensor* d = a.tensor(draft);
    if (!t || !d) return l;
    if (t->dim() != 3 || !t->is_contiguous() || t->size(0) > INT32_MAX || t->size(1) > INT32_MAX || t->size(2) > INT32_MAX) {
        a.ok = false;
        return l;
    }
    l.p = t->data_ptr();
    l.code = a.code(t);
    l.B = t->size(0);
    l.K = t->size(1) - 1;
    l.V = t->size(2);
    if (d->dim() != 2 || d->size(0) != l.B || d->size(1) != l.K) a.ok = false;
    return l;
}
void shape2(Args& a, PyObject* o, int64_t x, int64_t y) {
    const at::Tensor* t = a.tensor(o);
    if (!t || t->dim() != 2 || t->size(0) != x || t->size(1) != y) a.ok = false;
}
// ids, T_cap of a verification: the rows to append to, or none (T_cap given or 0).
Args::Rows context(Args& a, PyObject* ids, PyObject* T_cap, int64_t B) {
    if (ids != Py_None) return a.rows(ids, B, T_cap);
    Args::Rows r;
    if (T_cap != Py_None) r.T_cap = a.integer(T_cap, INT64_MIN, INT64_MAX);
    return r;
}

// logits, draft, draft_len, accept_len, next_token, workspace, argmax, ids, seq_len,
// kv_keep_len, status, T_cap, stream
PLDP_CALL(verify_greedy) {
    PLDP_BEGIN(13)
    const Logits l = logits(a, v[0], v[1]);
    const int32_t* draft = a.ints(v[1], l.B * l.K);
    const int32_t* dl = a.ints(v[2], l.B);
    int32_t* acc = a.ints(v[3], l.B);
    int32_t* nxt = a.ints(v[4], l.B);
    size_t size;
    void* ws = a.bytes(v[5], &size);
    int32_t* am = a.ints(v[6], l.B * (l.K + 1), true);
    const Args::Rows r = context(a, v[7], v[11], l.B);
    int32_t* L = a.ints(v[8], l.B, true);
    int32_t* kv = a.ints(v[9], l.B, true);
    uint32_t* st = a.words(v[10], l.B);
    void* s = a.stream(v[12]);
    return finish(a, [&] {
        return lib.verify_greedy(l.p, l.code, static_cast<int>(l.B), static_cast<int>(l.K), static_cast<int>(l.V), draft, dl,
                                 am, acc, nxt, r.p, r.stride, L, r.T_cap, kv, st, ws, size, s);
    });
    PLDP_END
}

// logits, uniforms, draft, draft_len, accept_len, next_token, workspace, temperature,
// sampled, ids, seq_len, kv_keep_len, status, T_cap, stream
PLDP_CALL(verify_sample) {
    PLDP_BEGIN(15)
    const Logits l = logits(a, v[0], v[2]);
    shape2(a, v[1], l.B, l.K + 1);
    const float* u = a.floats(v[1], -1);
    const int32_t* draft = a.ints(v[2], l.B * l.K);
    const int32_t* dl = a.ints(v[3], l.B);
    int32_t* acc = a.ints(v[4], l.B);
    int32_t* nxt = a.ints(v[5], l.B);
    size_t size;
    void* ws = a.bytes(v[6], &size);
    const float T = a.real(v[7]);
    int32_t* am = a.ints(v[8], l.B * (l.K + 1), true);
    const Args::Rows r = context(a, v[9], v[13], l.B);
    int32_t* L = a.ints(v[10], l.B, true);
    int32_t* kv = a.ints(v[11], l.B, true);
    uint32_t* st = a.words(v[12], l.B);
    void* s = a.stream(v[14]);
    return finish(a, [&] {
        return lib.verify_sample(l.p, l.code, static_cast<int>(l.B), static_cast<int>(l.K), static_cast<int>(l.V), T, u, draft,
                                 dl, am, acc, nxt, r.p, r.stride, L, r.T_cap, kv, st, ws, size, s);
    });
    PLDP_END
}

// The fused calls' shared arguments from v: draft, draft_len, accept_len, next_token,
// workspace, ids, seq_len, ngram_min, ngram_max, cand_pos, cand_count, match_len,
// next_draft, next_draft_len, index; then the tokens out, kv_keep_len and the keywords.
template <typename Block>
void fused(Args& a, const Logits& l, PyObject* const* v, PyObject* tokens, PyObject* kv, PyObject* kw, Block& b,
           int32_t** tokens_out) {
    shape2(a, v[12], l.B, l.K);
    const at::Tensor* ids = a.tensor(v[5]);
    if (!ids || ids->dim() != 2 || ids->size(0) != l.B) a.ok = false;
    if (!a.ok) return;
    PyObject* K = PyLong_FromLongLong(l.K);
    if (!K) {
        PyErr_Clear();
        a.ok = false;
        return;
    }
    PyObject* const p[10] = {v[5], v[6], v[7], v[8], v[9], v[10], v[11], K, v[12], v[13]};
    draft_args(a, p, nullptr, kw, v[14], l.V, b.next);
    Py_DECREF(K);
    if (v[14] == Py_None) a.ok = false;
    b.logits = l.p;
    b.dtype = l.code;
    b.V = static_cast<int>(l.V);
    b.draft = a.ints(v[0], l.B * l.K);
    b.draft_len = a.ints(v[1], l.B);
    b.accept_len = a.ints(v[2], l.B);
    b.next_token = a.ints(v[3], l.B);
    b.workspace = a.bytes(v[4], &b.workspace_bytes);
    *tokens_out = a.ints(tokens, l.B * (l.K + 1), true);
    b.kv_keep_len = a.ints(kv, l.B, true);
}

// logits, (the shared arguments), argmax, kv_keep_len, stream, keywords
PLDP_CALL(verify_greedy_draft) {
    PLDP_BEGIN(20)
    pldp_verify_draft_args b = {};
    const Logits l = logits(a, v[0], v[1]);
    fused(a, l, v + 1, v[16], v[17], v[19], b, &b.argmax);
    void* s = a.stream(v[18]);
    return finish(a, [&] { return lib.verify_greedy_draft(&b, s); });
    PLDP_END
}

// logits, uniforms, (the shared arguments), temperature, sampled, kv_keep_len, stream, keywords
PLDP_CALL(verify_sample_draft) {
    PLDP_BEGIN(22)
    pldp_verify_sample_draft_args b = {};
    const Logits l = logits(a, v[0], v[2]);
    shape2(a, v[1], l.B, l.K + 1);
    b.uniforms = a.floats(v[1], l.B * (l.K + 1));
    b.temperature = a.real(v[17]);
    fused(a, l, v + 2, v[18], v[19], v[21], b, &b.sampled);
    void* s = a.stream(v[20]);
    return finish(a, [&] { return lib.verify_sample_draft(&b, s); });
    PLDP_END
}

// ids, pos, A, counts, max_suffix, r_star, status, stream
PLDP_CALL(identify_heads) {
    PLDP_BEGIN(8)
    const at::Tensor* A = a.dims3(v[2]);
    if (!A || A->stride(2) != 1) Py_RETURN_NONE;
    const void* rows = A->data_ptr();
    const int64_t B = A->size(0), R = A->size(1), row_stride = A->stride(1), seq_stride = A->stride(0);
    const Args::Rows r = a.rows(v[0], B, nullptr);
    if (A->size(2) < r.T_cap || B > INT32_MAX || R > INT32_MAX) a.ok = false;
    const pldp_dtype code = a.code(A);
    const int32_t* pos = a.ints(v[1], B);
    uint32_t* counts = a.words(v[3], R, false);
    const int ms = static_cast<int>(a.integer(v[4]));
    int32_t* rs = a.ints(v[5], B, true);
    uint32_t* st = a.words(v[6], B);
    void* s = a.stream(v[7]);
    return finish(a, [&] {
        return lib.identify_heads(r.p, r.stride, pos, static_cast<int>(B), r.T_cap, ms, rows, code, static_cast<int>(R),
                                  row_stride, seq_stride, counts, rs, st, s);
    });
    PLDP_END
}

// counts, k, row_idx, stream
PLDP_CALL(top_heads) {
    PLDP_BEGIN(4)
    const uint32_t* c = a.words(v[0], 0, false);
    const int64_t k = a.integer(v[1]);
    int32_t* out = a.ints(v[2], k < 0 ? 0 : k);
    void* s = a.stream(v[3]);
    if (!a.ok) Py_RETURN_NONE;
    const int64_t R = THPVariable_Unpack(v[0]).numel();
    if (R > INT32_MAX) a.ok = false;
    return finish(a, [&] { return lib.top_heads(c, static_cast<int>(R), static_cast<int>(k), out, s); });
    PLDP_END
}

// bind(addresses): the library's entry points, in the order of `Library`.
PyObject* bind(PyObject*, PyObject* addresses) noexcept {
    constexpr Py_ssize_t count = sizeof(Library) / sizeof(void*);
    if (!PyTuple_CheckExact(addresses) || PyTuple_GET_SIZE(addresses) != count) {
        PyErr_SetString(PyExc_ValueError, "bind: a tuple with every entry point's address");
        return nullptr;
    }
    void* p[count];
    for (Py_ssize_t i = 0; i < count; ++i) {
        p[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(addresses, i));
        if (p[i] == nullptr) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: null address");
            return nullptr;
        }
    }
    std::memcpy(&lib, p, sizeof p);
    Py_RETURN_NONE;
}

#define PLDP_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    PLDP_METHOD(find_candidates), PLDP_METHOD(rank_hidden), PLDP_METHOD(rank_attention), PLDP_METHOD(extract_draft),
    PLDP_METHOD(draft_step), PLDP_METHOD(index_build), PLDP_METHOD(verify_greedy), PLDP_METHOD(verify_greedy_draft),
    PLDP_METHOD(verify_sample), PLDP_METHOD(verify_sample_draft), PLDP_METHOD(identify_heads), PLDP_METHOD(top_heads),
    {"bind", bind, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pldp_calls", "Native argument checks of the PLD+ binding.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pldp_calls(void) {
    for (int i = 0; i < kKeys; ++i)
        if (!(names[i] = PyUnicode_InternFromString(kNames[i]))) return nullptr;
    s_hidden = PyUnicode_InternFromString("hidden");
    s_attention = PyUnicode_InternFromString("attention");
    if (!s_hidden || !s_attention) return nullptr;
    return PyModule_Create(&module);
}
