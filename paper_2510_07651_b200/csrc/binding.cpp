// CPython binding of the C ABI for torch tensors: the host path of api.py in native code.
//
// A score call on a short cache is shorter on the GPU than its host path was when Python marshalled every argument
// through ctypes (26 us of host time for a 1k-token score call of three kernels, 80 us for the whole eviction).  Here a
// call unpacks its tensors, allocates what the caller did not pass, and enters the library once.  Nothing is kept from
// one call to the next.  Positional arguments only; api.py supplies names and defaults.  A failing library call returns
// its status as an int, which api.py turns into ObcError.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "obcache.h"

namespace {

using at::Tensor;

// The argument as a tensor, or an undefined tensor for None; false (with a Python error set) for anything else.
bool tensor_arg(PyObject* o, const Tensor** out, bool optional = false) {
    static const Tensor none;
    if (optional && o == Py_None) { *out = &none; return true; }
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a torch.Tensor"); return false; }
    *out = &THPVariable_Unpack(o);
    return true;
}

// View of a 4-D [batch, heads, tokens, head_dim] CUDA tensor with contiguous head_dim.
bool view4(const Tensor& t, obc_tensor* v) {
    if (!t.is_cuda() || t.dim() != 4 || t.stride(3) != 1) {
        PyErr_SetString(PyExc_ValueError, "expected a CUDA tensor [batch, heads, tokens, head_dim] with contiguous head_dim");
        return false;
    }
    const auto st = t.scalar_type();
    if (st != at::kFloat && st != at::kBFloat16) { PyErr_SetString(PyExc_TypeError, "unsupported dtype"); return false; }
    *v = obc_tensor{t.data_ptr(), st == at::kFloat ? OBC_F32 : OBC_BF16, t.stride(0), t.stride(1), t.stride(2)};
    return true;
}
bool view4_arg(PyObject* o, const Tensor** t, obc_tensor* v) { return tensor_arg(o, t) && view4(**t, v); }

template <typename T = void> T* ptr(const Tensor& t) { return t.defined() ? static_cast<T*>(t.data_ptr()) : nullptr; }

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
Tensor bytes_like(size_t n, const Tensor& like) {
    return at::empty({(int64_t)(n < 256 ? 256 : n)}, like.options().dtype(at::kByte));
}
PyObject* wrap(const Tensor& t) { return THPVariable_Wrap(t); }
PyObject* status(obc_status s) { return PyLong_FromLong((long)s); }
PyObject* tuple_of(std::initializer_list<Tensor> ts) {
    PyObject* tup = PyTuple_New((Py_ssize_t)ts.size());
    Py_ssize_t i = 0;
    for (const Tensor& t : ts) PyTuple_SET_ITEM(tup, i++, wrap(t));
    return tup;
}
long as_long(PyObject* o) { return PyLong_AsLong(o); }
bool expect(Py_ssize_t have, Py_ssize_t want) {
    if (have == want) return true;
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return false;
}

// Python's lock is released while the library runs (a launch blocks when the stream's queue is full).
template <typename F> obc_status unlocked(F f) {
    obc_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return st;
}

obc_score_params score_params(const Tensor& q, const Tensor& k, const Tensor& seq_lens, const Tensor& mask_lens, double scale,
                              long causal, long variants, long path) {
    obc_score_params p{};
    p.struct_size = sizeof(p);
    p.batch = (int32_t)q.size(0); p.n_q_heads = (int32_t)q.size(1); p.n_kv_heads = (int32_t)k.size(1); p.head_dim = (int32_t)q.size(3);
    p.window = (int32_t)q.size(2); p.max_len = (int32_t)k.size(2);
    p.seq_lens = ptr<int32_t>(seq_lens); p.mask_lens = ptr<int32_t>(mask_lens);
    p.scale = (float)scale; p.causal = causal ? 1 : 0; p.variants = (uint32_t)variants; p.path = (int32_t)path;
    return p;
}

// workspace of a score call: the caller's, or a new one
obc_status score_workspace(const obc_score_params& p, const Tensor& k, const Tensor& given, Tensor* ws) {
    if (given.defined()) { *ws = given; return OBC_OK; }
    size_t n = 0;
    const obc_status st = obc_score_workspace(&p, &n);
    if (st == OBC_OK) *ws = bytes_like(n, k);
    return st;
}

Tensor new_scores(const obc_score_params& p, const Tensor& k) {
    return at::empty({(int64_t)__builtin_popcount(p.variants), k.size(0), k.size(1), k.size(2)}, k.options().dtype(at::kFloat));
}

// score(q, k, v, o, lse, seq_lens, mask_lens, scale, causal, variants, path, scores, workspace); o is None: obc_score
PyObject* n_score(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!expect(n, 13)) return nullptr;
    const Tensor *q, *k, *v, *o, *lse, *lens, *mlens, *scores_in, *ws_in;
    obc_tensor tq, tk, tv, to{};
    if (!view4_arg(a[0], &q, &tq) || !view4_arg(a[1], &k, &tk) || !view4_arg(a[2], &v, &tv) || !tensor_arg(a[3], &o, true) ||
        !tensor_arg(a[4], &lse, true) || !tensor_arg(a[5], &lens, true) || !tensor_arg(a[6], &mlens, true) ||
        !tensor_arg(a[11], &scores_in, true) || !tensor_arg(a[12], &ws_in, true)) return nullptr;
    if (o->defined()) {
        if (!lse->defined() || o->sizes() != q->sizes() || lse->sizes() != q->sizes().slice(0, 3)) {
            PyErr_SetString(PyExc_ValueError, "o must be shaped like q and lse like q without its last axis");
            return nullptr;
        }
        if (lse->scalar_type() != at::kFloat || !lse->is_contiguous()) {
            PyErr_SetString(PyExc_ValueError, "lse must be a contiguous float32 tensor");
            return nullptr;
        }
        if (!view4(*o, &to)) return nullptr;
    }
    const double scale = PyFloat_AsDouble(a[7]);
    const long causal = as_long(a[8]), variants = as_long(a[9]), path = as_long(a[10]);
    if (PyErr_Occurred()) return nullptr;
    const obc_score_params p = score_params(*q, *k, *lens, *mlens, scale, causal, variants, path);
    Tensor ws;
    obc_status st = score_workspace(p, *k, *ws_in, &ws);
    if (st != OBC_OK) return status(st);
    const Tensor scores = scores_in->defined() ? *scores_in : new_scores(p, *k);
    void* s = stream();
    st = unlocked([&] {
        return o->defined() ? obc_score_given(&p, tq, tk, tv, to, ptr<float>(*lse), ptr<float>(scores), ws.data_ptr(), (size_t)ws.numel(), s)
                            : obc_score(&p, tq, tk, tv, ptr<float>(scores), ws.data_ptr(), (size_t)ws.numel(), s);
    });
    return st == OBC_OK ? wrap(scores) : status(st);
    END_HANDLE_TH_ERRORS
}

obc_select_params select_params(const Tensor& scores, long budget, const Tensor& budgets, long idx_stride, const Tensor& lens,
                                long n_sink, long n_recent, long pool, long pool_kernel) {
    obc_select_params p{};
    p.struct_size = sizeof(p);
    p.batch = (int32_t)scores.size(0); p.n_kv_heads = (int32_t)scores.size(1); p.max_len = (int32_t)scores.size(2);
    p.seq_lens = ptr<int32_t>(lens); p.budget = (int32_t)budget; p.budgets = ptr<int32_t>(budgets); p.idx_stride = (int32_t)idx_stride;
    p.n_sink = (int32_t)n_sink; p.n_recent = (int32_t)n_recent; p.pool_mode = (int32_t)pool; p.pool_kernel = (int32_t)pool_kernel;
    return p;
}
Tensor new_idx(const obc_select_params& p, const Tensor& like) {
    return at::empty({p.batch, p.n_kv_heads, p.idx_stride}, like.options().dtype(at::kInt));
}

// select(scores, budget, budgets, idx_stride, seq_lens, n_sink, n_recent, pool, pool_kernel, idx, workspace,
//        safeguard, counts); safeguard is None: obc_select -> idx, else obc_select_adaptive -> (idx, counts)
PyObject* n_select(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!expect(n, 13)) return nullptr;
    const Tensor *scores, *budgets, *lens, *idx_in, *ws_in, *counts_in;
    if (!tensor_arg(a[0], &scores) || !tensor_arg(a[2], &budgets, true) || !tensor_arg(a[4], &lens, true) ||
        !tensor_arg(a[9], &idx_in, true) || !tensor_arg(a[10], &ws_in, true) || !tensor_arg(a[12], &counts_in, true)) return nullptr;
    if (scores->dim() != 3) { PyErr_SetString(PyExc_ValueError, "expected scores [batch, heads, tokens]"); return nullptr; }
    const bool adaptive = a[11] != Py_None;
    const double safeguard = adaptive ? PyFloat_AsDouble(a[11]) : 0.0;
    const long budget = as_long(a[1]), stride = as_long(a[3]), n_sink = as_long(a[5]), n_recent = as_long(a[6]), pool = as_long(a[7]),
               pool_kernel = as_long(a[8]);
    if (PyErr_Occurred()) return nullptr;
    const obc_select_params p = select_params(*scores, budget, *budgets, stride, *lens, n_sink, n_recent, pool, pool_kernel);
    const Tensor idx = idx_in->defined() ? *idx_in : new_idx(p, *scores);
    Tensor counts;
    if (adaptive) counts = counts_in->defined() ? *counts_in : at::empty({p.batch, p.n_kv_heads}, scores->options().dtype(at::kInt));
    size_t need = 0;
    obc_status st = adaptive ? obc_select_adaptive_workspace(&p, (float)safeguard, &need) : obc_select_workspace(&p, &need);
    if (st != OBC_OK) return status(st);
    const Tensor ws = ws_in->defined() ? *ws_in : bytes_like(need, *scores);
    void* s = stream();
    st = unlocked([&] {
        return adaptive ? obc_select_adaptive(&p, (float)safeguard, ptr<float>(*scores), ptr<int32_t>(idx), ptr<int32_t>(counts), ws.data_ptr(),
                                              (size_t)ws.numel(), s)
                        : obc_select(&p, ptr<float>(*scores), ptr<int32_t>(idx), ws.data_ptr(), (size_t)ws.numel(), s);
    });
    if (st != OBC_OK) return status(st);
    return adaptive ? tuple_of({idx, counts}) : wrap(idx);
    END_HANDLE_TH_ERRORS
}

// Buffers for the gathered rows.  Where the caller brought none, the kernel zeroes the rows of padding indices itself.
obc_status compact(const Tensor& k, const Tensor& v, const Tensor& idx, Tensor& k_out, Tensor& v_out, const Tensor& s_in, Tensor& s_out,
                   const obc_tensor& tk, const obc_tensor& tv, void* s, bool* bad_view) {
    const int64_t B = k.size(0), H = k.size(1), S = idx.size(2), d = k.size(3);
    uint32_t zero = 0;
    if (!k_out.defined()) { k_out = at::empty({B, H, S, d}, k.options()); zero |= OBC_ZERO_K; }
    if (!v_out.defined()) { v_out = at::empty({B, H, S, d}, v.options()); zero |= OBC_ZERO_V; }
    if (s_in.defined() && !s_out.defined()) { s_out = at::empty({B, H, S}, k.options().dtype(at::kFloat)); zero |= OBC_ZERO_SCORES; }
    obc_tensor tko, tvo;
    if (!view4(k_out, &tko) || !view4(v_out, &tvo)) { *bad_view = true; return OBC_OK; }
    return unlocked([&] {
        return obc_compact_padded((int32_t)B, (int32_t)H, (int32_t)d, (int32_t)S, (int32_t)k.size(2), tk, tv, ptr<int32_t>(idx), tko, tvo,
                                  ptr<float>(s_in), ptr<float>(s_out), zero, s);
    });
}

// compact(k, v, idx, k_out, v_out, scores_in, scores_out)
PyObject* n_compact(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!expect(n, 7)) return nullptr;
    const Tensor *k, *v, *idx, *ko, *vo, *si, *so;
    obc_tensor tk, tv;
    if (!view4_arg(a[0], &k, &tk) || !view4_arg(a[1], &v, &tv) || !tensor_arg(a[2], &idx) || !tensor_arg(a[3], &ko, true) ||
        !tensor_arg(a[4], &vo, true) || !tensor_arg(a[5], &si, true) || !tensor_arg(a[6], &so, true)) return nullptr;
    if (idx->dim() != 3) { PyErr_SetString(PyExc_ValueError, "expected idx [batch, heads, kept]"); return nullptr; }
    Tensor k_out = *ko, v_out = *vo, s_out = *so;
    bool bad_view = false;
    const obc_status st = compact(*k, *v, *idx, k_out, v_out, *si, s_out, tk, tv, stream(), &bad_view);
    if (bad_view) return nullptr;
    if (st != OBC_OK) return status(st);
    return si->defined() ? tuple_of({k_out, v_out, s_out}) : tuple_of({k_out, v_out});
    END_HANDLE_TH_ERRORS
}

// evict(q, k, v, budget, seq_lens, variants, n_sink, n_recent, pool, pool_kernel, causal, path): score -> select -> compact
// with one budget; (k_out, v_out, idx, scores), or (status, stage)
PyObject* n_evict(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!expect(n, 12)) return nullptr;
    const Tensor *q, *k, *v, *lens;
    obc_tensor tq, tk, tv;
    if (!view4_arg(a[0], &q, &tq) || !view4_arg(a[1], &k, &tk) || !view4_arg(a[2], &v, &tv) || !tensor_arg(a[4], &lens, true)) return nullptr;
    const long budget = as_long(a[3]), variants = as_long(a[5]), n_sink = as_long(a[6]), n_recent = as_long(a[7]), pool = as_long(a[8]),
               pool_kernel = as_long(a[9]), causal = as_long(a[10]), path = as_long(a[11]);
    if (PyErr_Occurred()) return nullptr;
    auto fail = [](obc_status st, long stage) { return Py_BuildValue("(ll)", (long)st, stage); };
    const obc_score_params p = score_params(*q, *k, *lens, Tensor(), 0.0, causal, variants, path);
    Tensor ws;
    obc_status st = score_workspace(p, *k, Tensor(), &ws);
    if (st != OBC_OK) return fail(st, 0);
    const Tensor scores = new_scores(p, *k);
    void* s = stream();
    st = unlocked([&] { return obc_score(&p, tq, tk, tv, ptr<float>(scores), ws.data_ptr(), (size_t)ws.numel(), s); });
    if (st != OBC_OK) return fail(st, 0);
    const Tensor plane = scores.select(0, 0);
    const obc_select_params sp = select_params(plane, budget, Tensor(), budget, *lens, n_sink, n_recent, pool, pool_kernel);
    size_t need = 0;
    st = obc_select_workspace(&sp, &need);
    if (st != OBC_OK) return fail(st, 1);
    const Tensor idx = new_idx(sp, *k), ws_sel = bytes_like(need, *k);
    st = unlocked([&] { return obc_select(&sp, ptr<float>(plane), ptr<int32_t>(idx), ws_sel.data_ptr(), (size_t)ws_sel.numel(), s); });
    if (st != OBC_OK) return fail(st, 2);
    Tensor k_out, v_out, none;
    bool bad_view = false;
    st = compact(*k, *v, idx, k_out, v_out, none, none, tk, tv, s, &bad_view);
    if (bad_view) return nullptr;
    if (st != OBC_OK) return fail(st, 3);
    return tuple_of({k_out, v_out, idx, scores});
    END_HANDLE_TH_ERRORS
}

// decode_step(q_t, k_t, v_t, k_cache, v_cache, s_acc, pos, state, step_pos, budget, n_sink, n_recent, variant, scale,
//             workspace, acc_window, s_hist) -> workspace
PyObject* n_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!expect(n, 17)) return nullptr;
    const Tensor *t[5], *acc, *pos, *state, *ws_in, *hist;
    obc_tensor tt[5];
    for (int i = 0; i < 5; ++i) if (!view4_arg(a[i], &t[i], &tt[i])) return nullptr;
    if (!tensor_arg(a[5], &acc) || !tensor_arg(a[6], &pos) || !tensor_arg(a[7], &state) || !tensor_arg(a[14], &ws_in, true) ||
        !tensor_arg(a[16], &hist, true)) return nullptr;
    const double scale = PyFloat_AsDouble(a[13]);
    const long step_pos = as_long(a[8]), budget = as_long(a[9]), n_sink = as_long(a[10]), n_recent = as_long(a[11]), variant = as_long(a[12]),
               acc_window = as_long(a[15]);
    if (PyErr_Occurred()) return nullptr;
    const Tensor &q = *t[0], &kc = *t[3];
    if (acc_window > 0 && hist->defined() &&
        (hist->scalar_type() != at::kFloat || !hist->is_contiguous() || hist->sizes() != at::IntArrayRef({q.size(0), kc.size(1), acc_window, kc.size(2)}))) {
        PyErr_SetString(PyExc_AssertionError, "s_hist must be a contiguous float32 tensor [B,Hkv,acc_window,capacity]");
        return nullptr;
    }
    obc_decode_params p{};
    p.struct_size = sizeof(p);
    p.batch = (int32_t)q.size(0); p.n_q_heads = (int32_t)q.size(1); p.n_kv_heads = (int32_t)kc.size(1); p.head_dim = (int32_t)q.size(3);
    p.capacity = (int32_t)kc.size(2); p.budget = (int32_t)budget; p.n_sink = (int32_t)n_sink; p.n_recent = (int32_t)n_recent;
    p.variant = (uint32_t)variant; p.scale = (float)scale; p.acc_window = (int32_t)acc_window; p.s_hist = ptr<float>(*hist);
    Tensor ws = *ws_in;
    if (!ws.defined()) {
        size_t need = 0;
        const obc_status st = obc_decode_workspace(&p, &need);
        if (st != OBC_OK) return status(st);
        ws = bytes_like(need, kc);
    }
    void* s = stream();
    const obc_status st = unlocked([&] {
        return obc_decode_step(&p, tt[0], tt[1], tt[2], tt[3], tt[4], ptr<float>(*acc), ptr<int32_t>(*pos), ptr<int32_t>(*state),
                               (int32_t)step_pos, ws.data_ptr(), (size_t)ws.numel(), s);
    });
    return st == OBC_OK ? wrap(ws) : status(st);
    END_HANDLE_TH_ERRORS
}

#define OBC_METHOD(name, f) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {OBC_METHOD("score", n_score), OBC_METHOD("select", n_select), OBC_METHOD("compact", n_compact),
                         OBC_METHOD("evict", n_evict), OBC_METHOD("decode_step", n_decode), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
