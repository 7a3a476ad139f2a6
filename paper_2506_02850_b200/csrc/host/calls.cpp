// Native half of binding.py: the entry points that a program calls once per video, per pruning layer or
// per cache, from Python arguments to the C ABI and back.
//
// What bounds a small call is host work: a ctypes call converts some twenty arguments, each output is
// a torch.empty from Python, each scalar output a fill kernel, and the workspace and the stream are looked
// up by name -- 35 to 50 us per call before and between the launches (a call's own launches take 2 to 3 us
// each).  Here a call costs a few microseconds: tensors are unpacked in place, outputs come straight from
// the caching allocator, and the library is called through its function pointer.
//
// The functions take positional arguments from the wrappers of the same name in binding.py, which hold the
// documented signatures, and return the result dict, or the library's status as an int if it is not zero.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/core/LegacyTypeDispatch.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <memory>
#include <vector>

#include "../../../include/metok.h"

namespace {

// ---- the library's entry points, set by bind() when binding.py loads a library -------------------
#define METOK_HOST_CALLS(X)                                                                              \
    X(metok_segment_events_workspace_bytes) X(metok_segment_events)                                      \
    X(metok_segment_score_events_workspace_bytes) X(metok_segment_score_events)                          \
    X(metok_compress_vision_bound) X(metok_compress_vision_workspace_bytes) X(metok_compress_vision)     \
    X(metok_prefill_prune_workspace_bytes) X(metok_prefill_prune)                                        \
    X(metok_retention_budgets) X(metok_prune_schedule_sizes) X(metok_prefill_prune_schedule_workspace_bytes)                        \
    X(metok_prefill_prune_schedule) X(metok_kv_compact_workspace_bytes) X(metok_kv_compact)
struct Api {
#define X(name) decltype(&::name) name;
    METOK_HOST_CALLS(X)
#undef X
} api;

PyObject* bind(PyObject*, PyObject* table) {                  // {name: address}
#define X(name)                                                                                          \
    {                                                                                                    \
        PyObject* v = PyDict_GetItemString(table, #name);                                                \
        if (!v) return PyErr_Format(PyExc_KeyError, #name);                                              \
        api.name = reinterpret_cast<decltype(&::name)>(PyLong_AsVoidPtr(v));                             \
        if (PyErr_Occurred()) return nullptr;                                                            \
    }
    METOK_HOST_CALLS(X)
#undef X
    Py_RETURN_NONE;
}

// ---- small helpers ---------------------------------------------------------------------------------
struct Py {                                                   // owned reference
    PyObject* p;
    explicit Py(PyObject* o) : p(o) {}
    ~Py() { Py_XDECREF(p); }
    Py(const Py&) = delete;
    Py& operator=(const Py&) = delete;
};

// dict keys and argument names, interned once
#define METOK_HOST_NAMES(X)                                                                              \
    X(sims) X(boundaries) X(event_offsets) X(frame_event) X(_sims) X(_boundaries) X(_offsets)            \
    X(token_score) X(token_inv_norm) X(out_feats) X(out_src) X(out_event) X(out_members) X(assign)       \
    X(frame_score) X(event_score) X(event_is_key) X(n_out) X(status) X(scores) X(keep_idx) X(S_out)      \
    X(hidden_out) X(token_group) X(origin) X(n_vis) X(S) X(_inputs) X(keep_len) X(new_len)
struct Names {
#define X(name) PyObject* name;
    METOK_HOST_NAMES(X)
#undef X
} names;

// Every failure sets a Python exception and throws this.
struct PyError {};
[[noreturn]] void fail(PyObject* type, const char* fmt, const char* what) {
    PyErr_Format(type, fmt, what);
    throw PyError();
}

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "%s must be a tensor", name);
    return THPVariable_Unpack(o);
}
const at::Tensor& cuda_contig(PyObject* o, const char* name) {
    const at::Tensor& t = tensor(o, name);
    if (!t.is_cuda()) fail(PyExc_ValueError, "%s must be a CUDA tensor", name);
    if (!t.is_contiguous()) fail(PyExc_ValueError, "%s must be contiguous", name);
    return t;
}
const at::Tensor& of_dims(PyObject* o, const char* name, int dims) {
    const at::Tensor& t = cuda_contig(o, name);
    if (t.dim() != dims) fail(PyExc_ValueError, "%s has the wrong number of dimensions", name);
    return t;
}
int dtype_code(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return METOK_F32;
    if (t.scalar_type() == at::kBFloat16) return METOK_BF16;
    fail(PyExc_TypeError, "unsupported dtype %s", c10::toString(t.scalar_type()));
}
long integer(PyObject* o) {
    if (PyLong_Check(o)) {
        const long v = PyLong_AsLong(o);
        if (v == -1 && PyErr_Occurred()) throw PyError();
        return v;
    }
    Py i(PyNumber_Long(o));
    if (!i.p) throw PyError();
    const long v = PyLong_AsLong(i.p);
    if (v == -1 && PyErr_Occurred()) throw PyError();
    return v;
}
double number(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyError();
    return v;
}
struct Seq {                                                  // a sequence's items
    Py list;
    Py_ssize_t n;
    PyObject** items;
    explicit Seq(PyObject* o) : list(PySequence_Fast(o, "a sequence is wanted")), n(0), items(nullptr) {
        if (!list.p) throw PyError();
        n = PySequence_Fast_GET_SIZE(list.p);
        items = PySequence_Fast_ITEMS(list.p);
    }
};

at::Tensor empty(at::IntArrayRef shape, at::ScalarType dt, const at::Device& dev) {
    return at::Tensor(at::detail::empty_cuda(shape, dt, dev, std::nullopt));
}
at::Tensor empty_i32(int64_t n, const at::Device& dev) { return empty({n}, at::kInt, dev); }
at::Tensor empty_f32(int64_t n, const at::Device& dev) { return empty({n}, at::kFloat, dev); }

void put(PyObject* dict, PyObject* key, const at::Tensor& t) {
    Py v(THPVariable_Wrap(t));
    if (!v.p || PyDict_SetItem(dict, key, v.p) != 0) throw PyError();
}
void put_int(PyObject* dict, PyObject* key, long value) {
    Py v(PyLong_FromLong(value));
    if (!v.p || PyDict_SetItem(dict, key, v.p) != 0) throw PyError();
}
PyObject* item(PyObject* dict, PyObject* key) {
    PyObject* v = PyDict_GetItemWithError(dict, key);
    if (!v) {
        if (!PyErr_Occurred()) PyErr_SetObject(PyExc_KeyError, key);
        throw PyError();
    }
    return v;
}
const at::Tensor& get(PyObject* dict, PyObject* key) { return tensor(item(dict, key), "an output"); }

// The first n elements of the one-dimensional `whole` under `key`; an entry that `have` (the caller's
// dict, may be null) already holds is taken over.
void put_first(PyObject* dict, PyObject* key, PyObject* have, const at::Tensor& whole, int64_t n) {
    if (have) {
        PyObject* old = PyDict_GetItemWithError(have, key);
        if (old && THPVariable_Check(old)) {
            const at::Tensor& t = THPVariable_Unpack(old);
            if (t.dim() == 1 && t.numel() == n && t.data_ptr() == whole.data_ptr() && t.scalar_type() == whole.scalar_type()) {
                if (have != dict && PyDict_SetItem(dict, key, old) != 0) throw PyError();
                return;
            }
        }
        if (PyErr_Occurred()) throw PyError();
    }
    if (whole.numel() == n) {
        put(dict, key, whole);
        return;
    }
    at::AutoDispatchBelowADInplaceOrView guard;
    put(dict, key, whole.slice(0, 0, n));
}

// ---- workspaces ------------------------------------------------------------------------------------
// One buffer per device and stream: calls on one stream never overlap, calls on different streams may.
// Guarded by the interpreter lock.  A stream that outgrows its buffer gets a new one; at most kMaxWorkspaces
// are held, the one used longest ago goes first (the allocator keeps its memory from being reused before
// the stream's queued work is done).
struct Workspace {
    c10::DeviceIndex dev;
    cudaStream_t stream;
    at::Tensor buf, status;                                   // status: the first int32, the call's status word
    uint64_t used;
};
constexpr size_t kMaxWorkspaces = 256;                        // beyond the streams torch itself hands out per device
std::vector<Workspace>& workspaces() {
    static auto* v = new std::vector<Workspace>();            // never destroyed: tensors must not outlive the CUDA context's teardown
    return *v;
}
uint64_t ws_clock = 0;

Workspace workspace(size_t need, const at::Device& dev) {
    const auto stream = c10::cuda::getCurrentCUDAStream(dev.index());
    std::vector<Workspace>& all = workspaces();
    Workspace* w = nullptr;
    for (Workspace& x : all)
        if (x.stream == stream.stream() && x.dev == stream.device_index()) { w = &x; break; }
    if (!w) {
        if (all.size() >= kMaxWorkspaces) {
            size_t oldest = 0;
            for (size_t i = 1; i < all.size(); ++i)
                if (all[i].used < all[oldest].used) oldest = i;
            all.erase(all.begin() + oldest);
        }
        all.push_back({stream.device_index(), stream.stream(), at::Tensor(), at::Tensor(), 0});
        w = &all.back();
    }
    if (!w->buf.defined() || (size_t)w->buf.numel() < need) {
        const int64_t bytes = need > ((size_t)1 << 20) ? (int64_t)need : (int64_t)1 << 20;
        w->buf = empty({bytes}, at::kByte, dev);
        at::AutoDispatchBelowADInplaceOrView guard;
        w->status = w->buf.slice(0, 0, 4).view(at::kInt);
    }
    w->used = ++ws_clock;
    return *w;
}

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

void want(Py_ssize_t n, Py_ssize_t expected) {
    if (n != expected) fail(PyExc_TypeError, "%s", "wrong number of arguments");
}

// ---- calls -----------------------------------------------------------------------------------------
PyObject* py_workspace(PyObject* const* a, Py_ssize_t n) {     // nbytes, any tensor's device given as a tensor or index
    want(n, 2);
    return THPVariable_Wrap(workspace((size_t)integer(a[0]), at::Device(at::kCUDA, (c10::DeviceIndex)integer(a[1]))).buf);
}

// The four arrays a segmentation writes: new, or those of an earlier result.
struct SegOut {
    at::Tensor sims, boundaries, offsets, frame_event;
};
SegOut seg_new(int64_t T, int64_t k, const at::Device& dev) {
    return {empty_f32(T > 1 ? T - 1 : 1, dev), empty_i32(k > 1 ? k - 1 : 1, dev), empty_i32(k > 0 ? k + 1 : 2, dev),
            empty_i32(T, dev)};
}
SegOut seg_from(PyObject* d) {
    return {get(d, names._sims), get(d, names._boundaries), get(d, names._offsets), get(d, names.frame_event)};
}
void seg_put(PyObject* dict, PyObject* have, const SegOut& o, int64_t T, int64_t k) {
    put_first(dict, names.sims, have, o.sims, T - 1);
    put_first(dict, names.boundaries, have, o.boundaries, k > 1 ? k - 1 : 0);
    put_first(dict, names.event_offsets, have, o.offsets, k + 1);
}

PyObject* segment_events(PyObject* const* a, Py_ssize_t n) {   // feats, k, sim_mode, out
    want(n, 4);
    const at::Tensor& feats = of_dims(a[0], "feats", 3);
    const int T = (int)feats.size(0), N = (int)feats.size(1), d = (int)feats.size(2);
    const int k = (int)integer(a[1]), sim = (int)integer(a[2]), dt = dtype_code(feats);
    PyObject* have = a[3] == Py_None ? nullptr : a[3];
    const SegOut o = have ? seg_from(have) : seg_new(T, k, feats.device());
    const Workspace ws = workspace(api.metok_segment_events_workspace_bytes(dt, T, N, d, sim), feats.device());
    const int st = api.metok_segment_events(feats.data_ptr(), dt, T, N, d, k, sim, (float*)o.sims.data_ptr(),
                                            (int32_t*)o.boundaries.data_ptr(), (int32_t*)o.offsets.data_ptr(),
                                            (int32_t*)o.frame_event.data_ptr(), ws.buf.data_ptr(), ws.buf.numel(),
                                            current_stream());
    if (st != METOK_OK) return PyLong_FromLong(st);
    Py res(PyDict_New());
    if (!res.p) throw PyError();
    seg_put(res.p, have, o, T, k);
    put(res.p, names.frame_event, o.frame_event);
    put(res.p, names._sims, o.sims);
    put(res.p, names._boundaries, o.boundaries);
    put(res.p, names._offsets, o.offsets);
    Py_INCREF(res.p);
    return res.p;
}

PyObject* segment_score_events(PyObject* const* a, Py_ssize_t n) {   // feats, k, text_emb, out
    want(n, 4);
    const at::Tensor& feats = of_dims(a[0], "feats", 3);
    const at::Tensor& text = cuda_contig(a[2], "text_emb");
    const int T = (int)feats.size(0), N = (int)feats.size(1), d = (int)feats.size(2);
    const int k = (int)integer(a[1]), dt = dtype_code(feats);
    const bool reuse = a[3] != Py_None;
    Py res(reuse ? a[3] : PyDict_New());
    if (!res.p) throw PyError();
    if (reuse) Py_INCREF(res.p);
    SegOut o;
    at::Tensor score, inv_norm;
    if (reuse) {
        o = seg_from(res.p);
        score = get(res.p, names.token_score);
        inv_norm = get(res.p, names.token_inv_norm);
    } else {
        o = seg_new(T, k, feats.device());
        score = empty_f32((int64_t)T * N, feats.device());
        inv_norm = empty_f32((int64_t)T * N, feats.device());
        put(res.p, names._sims, o.sims);
        put(res.p, names._boundaries, o.boundaries);
        put(res.p, names._offsets, o.offsets);
        put(res.p, names.frame_event, o.frame_event);
        put(res.p, names.token_score, score);
        put(res.p, names.token_inv_norm, inv_norm);
    }
    const Workspace ws = workspace(api.metok_segment_score_events_workspace_bytes(dt, T, N, d), feats.device());
    const int st = api.metok_segment_score_events(
        feats.data_ptr(), dt, T, N, d, k, text.data_ptr(), (float*)o.sims.data_ptr(), (int32_t*)o.boundaries.data_ptr(),
        (int32_t*)o.offsets.data_ptr(), (int32_t*)o.frame_event.data_ptr(), (float*)score.data_ptr(),
        (float*)inv_norm.data_ptr(), ws.buf.data_ptr(), ws.buf.numel(), current_stream());
    if (st != METOK_OK) return PyLong_FromLong(st);
    seg_put(res.p, reuse ? res.p : nullptr, o, T, k);
    Py_INCREF(res.p);
    return res.p;
}

// feats, event_offsets, text_emb, params, cap, out, scored, key_events, key_frames
PyObject* compress_vision(PyObject* const* a, Py_ssize_t n) {
    want(n, 9);
    const at::Tensor& feats = of_dims(a[0], "feats", 3);
    const at::Tensor& offsets = cuda_contig(a[1], "event_offsets");
    const at::Tensor& text = cuda_contig(a[2], "text_emb");
    const int T = (int)feats.size(0), N = (int)feats.size(1), d = (int)feats.size(2);
    const int k = (int)offsets.numel() - 1, dt = dtype_code(feats);
    const at::Device dev = feats.device();
    metok_vision_params p;
    {
        Py_buffer view;
        if (PyObject_GetBuffer(a[3], &view, PyBUF_SIMPLE) != 0) throw PyError();
        const bool fits = view.len == (Py_ssize_t)sizeof(p);
        if (fits) memcpy(&p, view.buf, sizeof(p));
        PyBuffer_Release(&view);
        if (!fits) fail(PyExc_TypeError, "%s must be a VisionParams", "p");
    }
    const bool reuse = a[5] != Py_None;
    int cap;
    if (reuse) {
        cap = (int)get(a[5], names.out_src).numel();
    } else if (a[4] == Py_None) {
        cap = api.metok_compress_vision_bound(T, N, k, &p);
        if (cap < 0) return PyLong_FromLong(cap);
    } else {
        cap = (int)integer(a[4]);
    }
    Py res(reuse ? a[5] : PyDict_New());
    if (!res.p) throw PyError();
    if (reuse) {
        Py_INCREF(res.p);
    } else {
        const int64_t tokens = (int64_t)T * N;
        put(res.p, names.out_feats, empty({cap, d}, feats.scalar_type(), dev));
        put(res.p, names.out_src, empty_i32(cap, dev));
        put(res.p, names.out_event, empty_i32(cap, dev));
        put(res.p, names.out_members, empty_i32(cap, dev));
        put(res.p, names.assign, empty_i32(tokens, dev));
        if (a[6] == Py_None) put(res.p, names.token_score, empty_f32(tokens, dev));
        put(res.p, names.frame_score, empty_f32(T, dev));
        put(res.p, names.event_score, empty_f32(k, dev));
        put(res.p, names.event_is_key, empty({k}, at::kByte, dev));
        put(res.p, names.n_out, empty_i32(1, dev));
    }
    if (a[6] != Py_None) {
        if (PyDict_SetItem(res.p, names.token_score, item(a[6], names.token_score)) != 0) throw PyError();
        p.token_inv_norm = (const float*)get(a[6], names.token_inv_norm).data_ptr();
    }
    if (a[7] != Py_None) {
        const at::Tensor& t = cuda_contig(a[7], "key_events");
        if (t.scalar_type() != at::kByte || t.numel() != k) fail(PyExc_ValueError, "%s must be uint8 [k]", "key_events");
        p.key_events_given = (const uint8_t*)t.data_ptr();
    }
    if (a[8] != Py_None) {
        const at::Tensor& t = cuda_contig(a[8], "key_frames");
        if (t.scalar_type() != at::kByte || t.numel() != T) fail(PyExc_ValueError, "%s must be uint8 [T]", "key_frames");
        p.key_frames_given = (const uint8_t*)t.data_ptr();
    }
    const Workspace ws = workspace(api.metok_compress_vision_workspace_bytes(dt, T, N, d, k, cap, &p), dev);
    auto ptr = [&](PyObject* key) { return get(res.p, key).data_ptr(); };
    const int st = api.metok_compress_vision(
        feats.data_ptr(), dt, T, N, d, (const int32_t*)offsets.data_ptr(), k, text.data_ptr(), &p, ptr(names.out_feats),
        (int32_t*)ptr(names.out_src), (int32_t*)ptr(names.out_event), (int32_t*)ptr(names.out_members),
        (int32_t*)ptr(names.assign), (float*)ptr(names.token_score), (float*)ptr(names.frame_score),
        (float*)ptr(names.event_score), (uint8_t*)ptr(names.event_is_key), (int32_t*)ptr(names.n_out), cap,
        ws.buf.data_ptr(), ws.buf.numel(), current_stream());
    if (st != METOK_OK) return PyLong_FromLong(st);
    put(res.p, names.status, ws.status);
    Py_INCREF(res.p);
    return res.p;
}

// q_text, k_all, hidden, vis_start, n_vis, token_group, group_budget, softmax_scale, out
PyObject* prefill_prune(PyObject* const* a, Py_ssize_t n) {
    want(n, 9);
    const at::Tensor& q = of_dims(a[0], "q_text", 3);
    const at::Tensor& kk = of_dims(a[1], "k_all", 3);
    const at::Tensor& group = cuda_contig(a[5], "token_group");
    const int Hq = (int)q.size(0), Lt = (int)q.size(1), dh = (int)q.size(2), Hkv = (int)kk.size(0), S = (int)kk.size(1);
    const int vis_start = (int)integer(a[3]), n_vis = (int)integer(a[4]), dt = dtype_code(q);
    const float scale = (float)number(a[7]);
    const at::Device dev = q.device();
    at::Tensor hidden;
    int D = 0;
    if (a[2] != Py_None) {
        hidden = cuda_contig(a[2], "hidden");
        D = (int)hidden.size(1);
    }
    int32_t few[METOK_MAX_GROUPS];
    std::vector<int32_t> many;
    int32_t* budgets = few;
    int G;
    {
        Seq b(a[6]);
        G = (int)b.n;
        if (G > METOK_MAX_GROUPS) { many.resize(G); budgets = many.data(); }
        for (int g = 0; g < G; ++g) budgets[g] = (int32_t)integer(b.items[g]);
    }
    const bool reuse = a[8] != Py_None;
    Py res(reuse ? a[8] : PyDict_New());
    if (!res.p) throw PyError();
    at::Tensor scores, keep, s_out, hidden_out;
    if (reuse) {
        Py_INCREF(res.p);
        scores = get(res.p, names.scores);
        keep = get(res.p, names.keep_idx);
        s_out = get(res.p, names.S_out);
        PyObject* h = item(res.p, names.hidden_out);
        if (h != Py_None) hidden_out = tensor(h, "hidden_out");
    } else {
        scores = empty_f32(n_vis, dev);
        keep = empty_i32(S, dev);
        s_out = empty_i32(1, dev);
        put(res.p, names.scores, scores);
        put(res.p, names.keep_idx, keep);
        put(res.p, names.S_out, s_out);
        if (hidden.defined()) {
            hidden_out = empty(hidden.sizes(), hidden.scalar_type(), hidden.device());
            put(res.p, names.hidden_out, hidden_out);
        } else if (PyDict_SetItem(res.p, names.hidden_out, Py_None) != 0) {
            throw PyError();
        }
    }
    const Workspace ws = workspace(api.metok_prefill_prune_workspace_bytes(dt, Hq, Hkv, Lt, S, dh, n_vis), dev);
    const int st = api.metok_prefill_prune(
        q.data_ptr(), kk.data_ptr(), hidden.defined() ? hidden.data_ptr() : nullptr, dt, Hq, Hkv, Lt, S, dh, D, vis_start,
        n_vis, (const int32_t*)group.data_ptr(), G, budgets, scale, (float*)scores.data_ptr(), (int32_t*)keep.data_ptr(),
        (int32_t*)s_out.data_ptr(), hidden_out.defined() ? hidden_out.data_ptr() : nullptr, ws.buf.data_ptr(),
        ws.buf.numel(), current_stream());
    if (st != METOK_OK) return PyLong_FromLong(st);
    put(res.p, names.status, ws.status);
    Py_INCREF(res.p);
    return res.p;
}

PyObject* retention_budgets(PyObject* const* a, Py_ssize_t n) {   // alpha, r, stage, N0
    want(n, 4);
    int32_t n0[2], b[2];
    Seq s(a[3]);
    if (s.n < 2) fail(PyExc_ValueError, "%s must hold two counts", "N0");
    n0[0] = (int32_t)integer(s.items[0]);
    n0[1] = (int32_t)integer(s.items[1]);
    const int st = api.metok_retention_budgets(number(a[0]), number(a[1]), (int)integer(a[2]), n0, b);
    return st == METOK_OK ? Py_BuildValue("[ii]", b[0], b[1]) : PyLong_FromLong(st);
}

// q_texts, k_alls, hiddens, vis_start, token_group, alpha, r, N0, softmax_scale, levels: the last argument is a
// writable buffer of one metok_prune_level per level, filled here (the caller keeps it for the K/V lists)
PyObject* prefill_prune_schedule(PyObject* const* a, Py_ssize_t n) {
    want(n, 10);
    Seq qs(a[0]), ks(a[1]);
    const int n_levels = (int)qs.n;
    std::unique_ptr<Seq> hs;
    if (a[2] != Py_None) hs = std::make_unique<Seq>(a[2]);
    if (n_levels < 1 || n_levels > 3) return PyLong_FromLong(METOK_ERR_INVALID_ARG);
    if (ks.n < n_levels || (hs && hs->n < n_levels)) fail(PyExc_ValueError, "%s: one per level is wanted", "k_alls / hiddens");
    const at::Tensor& group = cuda_contig(a[4], "token_group");
    const int n_vis = (int)group.numel(), vis_start = (int)integer(a[3]);
    const double alpha = number(a[5]), r = number(a[6]);
    int32_t n0[2], sizes[4];
    {
        Seq s(a[7]);
        if (s.n < 2) fail(PyExc_ValueError, "%s must hold two counts", "N0");
        n0[0] = (int32_t)integer(s.items[0]);
        n0[1] = (int32_t)integer(s.items[1]);
    }
    int st = api.metok_prune_schedule_sizes(n_levels, alpha, r, n0, sizes);
    if (st != METOK_OK) return PyLong_FromLong(st);
    const float scale = (float)number(a[8]);
    const at::Tensor& q0 = of_dims(qs.items[0], "q_text", 3);
    const at::Tensor& k0 = of_dims(ks.items[0], "k_all", 3);
    const int Hq = (int)q0.size(0), Lt = (int)q0.size(1), dh = (int)q0.size(2), Hkv = (int)k0.size(0), S = (int)k0.size(1);
    const int dt = dtype_code(q0);
    const int D = hs ? (int)of_dims(hs->items[0], "hidden", 2).size(1) : 0;
    const at::Device dev = group.device();
    Py_buffer view;
    if (PyObject_GetBuffer(a[9], &view, PyBUF_WRITABLE) != 0) throw PyError();
    struct Release { Py_buffer* v; ~Release() { PyBuffer_Release(v); } } release{&view};
    if (view.len < (Py_ssize_t)sizeof(metok_prune_level) * n_levels) fail(PyExc_ValueError, "%s is too small", "levels");
    metok_prune_level* lv = static_cast<metok_prune_level*>(view.buf);
    Py list(PyList_New(n_levels));
    if (!list.p) throw PyError();
    for (int s = 0; s < n_levels; ++s) {
        const at::Tensor& q = cuda_contig(qs.items[s], "q_text");
        const at::Tensor& kk = of_dims(ks.items[s], "k_all", 3);
        const int S_s = S - n_vis + sizes[s];
        if (kk.size(0) != Hkv || kk.size(1) != S_s || kk.size(2) != dh) {
            PyErr_Format(PyExc_ValueError, "level %d: k_all must be (%d, %d, %d), got (%d, %d, %d)", s + 1, Hkv, S_s, dh,
                         (int)kk.size(0), (int)kk.size(1), (int)kk.size(2));
            throw PyError();
        }
        PyObject* d = PyDict_New();
        if (!d) throw PyError();
        PyList_SET_ITEM(list.p, s, d);
        const int64_t nv = sizes[s] > 0 ? sizes[s] : 1;
        const at::Tensor scores = empty_f32(nv, dev), keep = empty_i32(S_s, dev), s_out = empty_i32(1, dev),
                         origin = empty_i32(nv, dev), grp = s == 0 ? group : empty_i32(nv, dev);
        put(d, names.scores, scores);
        put(d, names.keep_idx, keep);
        put(d, names.S_out, s_out);
        lv[s] = {q.data_ptr(), kk.data_ptr(), nullptr, nullptr, (float*)scores.data_ptr(), (int32_t*)keep.data_ptr(),
                 (int32_t*)s_out.data_ptr(), (int32_t*)grp.data_ptr(), (int32_t*)origin.data_ptr()};
        PyObject* hid = hs ? hs->items[s] : Py_None;
        if (hs) {
            const at::Tensor& h = cuda_contig(hid, "hidden");
            const at::Tensor ho = empty(h.sizes(), h.scalar_type(), h.device());
            put(d, names.hidden_out, ho);
            lv[s].hidden = h.data_ptr();
            lv[s].hidden_out = ho.data_ptr();
        } else if (PyDict_SetItem(d, names.hidden_out, Py_None) != 0) {
            throw PyError();
        }
        put(d, names.token_group, grp);
        put(d, names.origin, origin);
        put_int(d, names.n_vis, sizes[s]);
        put_int(d, names.S, S_s);
        Py inputs(PyTuple_Pack(3, qs.items[s], ks.items[s], hid));   // alive until the caller is done with the result
        if (!inputs.p || PyDict_SetItem(d, names._inputs, inputs.p) != 0) throw PyError();
    }
    const size_t need = api.metok_prefill_prune_schedule_workspace_bytes(n_levels, dt, Hq, Hkv, Lt, S, dh, n_vis, alpha, r, n0);
    if (need == 0) return PyLong_FromLong(METOK_ERR_INVALID_ARG);
    const Workspace ws = workspace(need, dev);
    const at::Tensor status = empty_i32(1, dev);
    st = api.metok_prefill_prune_schedule(lv, n_levels, dt, Hq, Hkv, Lt, S, dh, D, vis_start, n_vis, alpha, r, n0, scale,
                                          (int32_t*)status.data_ptr(), ws.buf.data_ptr(), ws.buf.numel(), current_stream());
    if (st != METOK_OK) return PyLong_FromLong(st);
    Py wrapped(THPVariable_Wrap(status));
    if (!wrapped.p) throw PyError();
    for (int s = 0; s < n_levels; ++s)
        if (PyDict_SetItem(PyList_GET_ITEM(list.p, s), names.status, wrapped.p) != 0) throw PyError();
    Py_INCREF(list.p);
    return list.p;
}

// k_layers, v_layers, S_cur, policy, vis_start, n_vis, l1, keep_ratio, scores, keep_idx, keep_len, new_len
PyObject* kv_compact(PyObject* const* a, Py_ssize_t n) {
    want(n, 12);
    Seq ks(a[0]), vs(a[1]);
    const int L = (int)ks.n;
    if (L < 1) fail(PyExc_ValueError, "%s is empty", "k_layers");
    if (vs.n != L) fail(PyExc_ValueError, "%s must hold one tensor per layer", "v_layers");
    std::vector<void*> kp(L), vp(L);
    for (int l = 0; l < L; ++l) {
        kp[l] = cuda_contig(ks.items[l], "k/v layer").data_ptr();
        vp[l] = cuda_contig(vs.items[l], "k/v layer").data_ptr();
    }
    const at::Tensor& k0 = of_dims(ks.items[0], "k/v layer", 3);
    const int Hkv = (int)k0.size(0), S_cap = (int)k0.size(1), dh = (int)k0.size(2), dt = dtype_code(k0);
    const at::Device dev = k0.device();
    const int S_cur = (int)integer(a[2]), policy = (int)integer(a[3]), vis_start = (int)integer(a[4]), n_vis = (int)integer(a[5]),
              l1 = (int)integer(a[6]);
    const double ratio = number(a[7]);
    at::Tensor scores, keep, len, new_len;
    int per_layer = 0;
    if (a[8] != Py_None) {
        scores = cuda_contig(a[8], "scores");
        per_layer = scores.dim() == 2;
    }
    if (a[9] == Py_None) {
        keep = empty({L, S_cur}, at::kInt, dev);
        len = empty_i32(L, dev);
    } else {
        keep = tensor(a[9], "keep_idx");
        len = tensor(a[10], "keep_len");
    }
    new_len = a[11] == Py_None ? empty_i32(L, dev) : tensor(a[11], "new_len");
    const Workspace ws = workspace(api.metok_kv_compact_workspace_bytes(dt, L, Hkv, S_cur, dh, policy, n_vis), dev);
    const int st = api.metok_kv_compact(kp.data(), vp.data(), dt, L, Hkv, S_cap, S_cur, dh, policy, l1, ratio, vis_start, n_vis,
                                        scores.defined() ? (const float*)scores.data_ptr() : nullptr, per_layer,
                                        (int32_t*)keep.data_ptr(), (int32_t*)len.data_ptr(), (int32_t*)new_len.data_ptr(),
                                        ws.buf.data_ptr(), ws.buf.numel(), current_stream());
    if (st != METOK_OK) return PyLong_FromLong(st);
    Py res(PyDict_New());
    if (!res.p) throw PyError();
    put(res.p, names.keep_idx, keep);
    put(res.p, names.keep_len, len);
    put(res.p, names.new_len, new_len);
    put(res.p, names.status, ws.status);
    Py_INCREF(res.p);
    return res.p;
}

// Runs a call and turns its failures into Python exceptions.
template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    try {
        return F(args, n);
    } catch (const PyError&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

#define FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&guarded<fn>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    FAST("workspace", py_workspace),
    FAST("segment_events", segment_events),
    FAST("segment_score_events", segment_score_events),
    FAST("compress_vision", compress_vision),
    FAST("retention_budgets", retention_budgets),
    FAST("prefill_prune", prefill_prune),
    FAST("prefill_prune_schedule", prefill_prune_schedule),
    FAST("kv_compact", kv_compact),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_metok_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__metok_calls(void) {
#define X(name)                                                  \
    names.name = PyUnicode_InternFromString(#name);              \
    if (!names.name) return nullptr;
    METOK_HOST_NAMES(X)
#undef X
    return PyModule_Create(&module);
}
