// Python side of the C ABI: argument marshalling from torch tensors to the entry points of sv.h, as a CPython module.
//
// A layer of a verification step is two or three kernel launches (about 2.5 us of host time each), and a short one runs
// for less than 10 us, so what the host spends between launches is what a small call costs: the same marshalling in
// Python (type, device, dtype and layout checks per tensor, a ctypes call of 16 arguments) took 10-12 us per entry
// point.  Here a tensor is unpacked and checked in a few tens of nanoseconds: back to back, an eager layer of a small model
// (4K context) went from 30.5 to 12.3 us, an eager 32-layer step from 995 to 499 us.  The checks and the errors are those of
// the Python binding: a tensor that is not a contiguous CUDA tensor of the expected type raises TypeError before
// anything is launched, and the sv_status of the call is returned for the caller to map.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <string.h>

#include <ATen/core/CachingHostAllocator.h>
#include <ATen/EmptyTensor.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "sv.h"

namespace {

// A failed argument check: the Python exception is set, the call returns NULL.
struct ArgError {};

const at::Tensor &tensor(PyObject *o, at::ScalarType type, const char *name)
{
    if (THPVariable_Check(o)) {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (t.is_cuda() && t.scalar_type() == type && t.is_contiguous()) return t;
    }
    PyErr_Format(PyExc_TypeError, "%s: expected a contiguous CUDA tensor of torch.%s", name,
                 type == at::kBFloat16 ? "bfloat16" : type == at::kFloat ? "float32" : type == at::kByte ? "uint8" : "int32");
    throw ArgError{};
}

// Device pointer of a tensor argument (None: NULL).
void *ptr(PyObject *o, at::ScalarType type, const char *name)
{
    return o == Py_None ? nullptr : tensor(o, type, name).data_ptr();
}
void *bf16(PyObject *o, const char *name) { return ptr(o, at::kBFloat16, name); }
float *f32(PyObject *o, const char *name) { return static_cast<float *>(ptr(o, at::kFloat, name)); }
int32_t *i32(PyObject *o, const char *name) { return static_cast<int32_t *>(ptr(o, at::kInt, name)); }

long long integer(PyObject *o)
{
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw ArgError{};
    return v;
}
int32_t int32(PyObject *o)
{
    const long long v = integer(o);
    if (v < INT32_MIN || v > INT32_MAX) {
        PyErr_SetString(PyExc_OverflowError, "value does not fit in 32 bits");
        throw ArgError{};
    }
    return (int32_t)v;
}
bool truth(PyObject *o)
{
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw ArgError{};
    return v != 0;
}

// A ctypes structure (sv_geom, sv_kv) by its bytes.
template <class T>
T structure(PyObject *o, const char *name)
{
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
        PyErr_Format(PyExc_TypeError, "expected an %s", name);
        throw ArgError{};
    }
    const bool fits = view.len == (Py_ssize_t)sizeof(T);
    T v;
    if (fits) memcpy(&v, view.buf, sizeof(T));
    PyBuffer_Release(&view);
    if (!fits) {
        PyErr_Format(PyExc_TypeError, "expected an %s", name);
        throw ArgError{};
    }
    return v;
}
sv_geom geometry(PyObject *o) { return structure<sv_geom>(o, "sv_geom"); }
sv_kv cache(PyObject *o) { return structure<sv_kv>(o, "sv_kv"); }

// The stream argument of the binding: a torch stream, or None for the current one.
void *stream(PyObject *o)
{
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw ArgError{};
    void *s = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (!s && PyErr_Occurred()) throw ArgError{};
    return s;
}

// Last dimension of a list tensor: the row length max_sel.
int32_t row_length(PyObject *o, const char *name) { return (int32_t)tensor(o, at::kInt, name).size(-1); }

struct Scratch {
    void *p;
    size_t bytes;
};
Scratch scratch(PyObject *o)
{
    if (o == Py_None) return {nullptr, 0};
    if (!THPVariable_Check(o) || !THPVariable_Unpack(o).is_cuda()) {
        PyErr_SetString(PyExc_TypeError, "workspace must be a CUDA tensor");
        throw ArgError{};
    }
    const at::Tensor &t = THPVariable_Unpack(o);
    return {t.data_ptr(), (size_t)t.nbytes()};
}

// Every method: exactly N positional arguments, body returns a PyObject*.
template <class F>
PyObject *checked(Py_ssize_t n, Py_ssize_t want, F body)
{
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
        return nullptr;
    }
    try {
        return body();
    } catch (const ArgError &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
PyObject *status(sv_status st) { return PyLong_FromLong(st); }

// The library call itself, without the interpreter lock: a launch waits when the queue of its device is full, and the threads that
// drive other devices go on meanwhile.  All arguments are taken from Python before it (the caller holds the objects).  An eager layer
// of a small model, back to back: 11.9 us with the lock held, 11.9-12.1 without.
template <class F>
sv_status unlocked(F call)
{
    struct Unlocked {
        PyThreadState *const state = PyEval_SaveThread();
        ~Unlocked() { PyEval_RestoreThread(state); }
    } guard;
    return call();
}

// geom, kv, reps, block_begin, block_end, stream, reps_bf16
PyObject *block_reps(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 7, [&] {
        const sv_geom g = geometry(a[0]);
        const sv_kv kv = cache(a[1]);
        const int32_t begin = int32(a[3]), end = int32(a[4]);
        const bool half = truth(a[6]);
        void *const reps = half ? bf16(a[2], "reps_bf16") : f32(a[2], "reps"), *const s = stream(a[5]);
        return status(unlocked([&] {
            return half ? sv_block_reps_bf16(&g, &kv, begin, end, reps, s) : sv_block_reps(&g, &kv, begin, end, static_cast<float *>(reps), s);
        }));
    });
}

// geom, q, reps, seq_lens, budget_blocks, n_sink, n_local, out_idx, out_cnt, reuse_prev, prev_idx, prev_cnt, out_scores,
// stream, reps_bf16
PyObject *select_blocks(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 15, [&] {
        const sv_geom g = geometry(a[0]);
        const int32_t max_sel = row_length(a[7], "out_idx");
        const void *q = bf16(a[1], "q");
        const int32_t *lens = i32(a[3], "seq_lens"), *budget = i32(a[4], "budget_blocks");
        const int32_t sink = int32(a[5]), local = int32(a[6]);
        int32_t *idx = i32(a[7], "out_idx"), *cnt = i32(a[8], "out_cnt");
        const int32_t reuse = truth(a[9]) ? 1 : 0;
        const int32_t *pi = i32(a[10], "prev_idx"), *pc = i32(a[11], "prev_cnt");
        float *scores = f32(a[12], "out_scores");
        const bool half = truth(a[14]);
        const void *const reps = half ? bf16(a[2], "reps_bf16") : f32(a[2], "reps");
        void *const s = stream(a[13]);
        return status(unlocked([&] {
            if (half)
                return sv_select_blocks_bf16reps(&g, q, reps, lens, budget, sink, local, reuse, pi, pc, idx, cnt, max_sel, scores, s);
            return sv_select_blocks(&g, q, static_cast<const float *>(reps), lens, budget, sink, local, reuse, pi, pc, idx, cnt, max_sel,
                                    scores, s);
        }));
    });
}

// geom, q, kv, draft_k, draft_v, parent, sel_idx, sel_cnt, out, lse, workspace, softmax_scale, status_word, stream, entry
// (entry 0: sv_verify_attn, 1: sv_verify_attn_reused, 2: sv_verify_attn_noalloc)
PyObject *verify_attn(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 15, [&] {
        const sv_geom g = geometry(a[0]);
        const sv_kv kv = cache(a[2]);
        const int32_t max_sel = a[6] == Py_None ? g.max_blocks : row_length(a[6], "sel_idx");
        const void *q = bf16(a[1], "q"), *dk = bf16(a[3], "draft_k"), *dv = bf16(a[4], "draft_v");
        const int32_t *parent = i32(a[5], "parent"), *idx = i32(a[6], "sel_idx"), *cnt = i32(a[7], "sel_cnt");
        void *out = bf16(a[8], "out");
        float *lse = f32(a[9], "lse");
        const Scratch ws = scratch(a[10]);
        const double scale = PyFloat_AsDouble(a[11]);
        if (scale == -1.0 && PyErr_Occurred()) throw ArgError{};
        int32_t *word = i32(a[12], "status_word");
        void *s = stream(a[13]);
        const long long entry = integer(a[14]);
        return status(unlocked([&] {
            switch (entry) {
                case 0: return sv_verify_attn(&g, q, &kv, dk, dv, parent, idx, cnt, max_sel, (float)scale, out, lse, ws.p, ws.bytes, word, s);
                case 1: return sv_verify_attn_reused(&g, q, &kv, dk, dv, parent, idx, cnt, max_sel, (float)scale, out, lse, ws.p, ws.bytes, word, s);
                default: return sv_verify_attn_noalloc(&g, q, &kv, dk, dv, parent, idx, cnt, max_sel, (float)scale, out, lse, word, s);
            }
        }));
    });
}

// geom, k_pool, v_pool, block_table, seq_lens, draft_k, draft_v, accept_idx, n_accept, seq_lens_out, reps, stream
PyObject *kv_append(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 12, [&] {
        const sv_geom g = geometry(a[0]);
        const int32_t pages = (int32_t)tensor(a[1], at::kBFloat16, "k_pool").size(0);
        void *const k = bf16(a[1], "k_pool"), *const v = bf16(a[2], "v_pool");
        const int32_t *const table = i32(a[3], "block_table"), *const lens = i32(a[4], "seq_lens");
        const void *const dk = bf16(a[5], "draft_k"), *const dv = bf16(a[6], "draft_v");
        const int32_t *const rows = i32(a[7], "accept_idx"), *const n_rows = i32(a[8], "n_accept");
        const int32_t most = row_length(a[7], "accept_idx");
        int32_t *const lens_out = i32(a[9], "seq_lens_out");
        float *const reps = f32(a[10], "reps");
        void *const s = stream(a[11]);
        return status(unlocked([&] { return sv_kv_append(&g, k, v, pages, table, lens, dk, dv, rows, n_rows, most, lens_out, reps, s); }));
    });
}

// p_target, p_draft, tokens, parent, u_accept, u_next, path, n_path, next_token, alpha, stream
PyObject *accept(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 11, [&] {
        const at::Tensor &pt = tensor(a[0], at::kFloat, "p_target");
        const int32_t S = (int32_t)pt.size(0), T = (int32_t)pt.size(1), V = (int32_t)pt.size(2);
        const float *const target = f32(a[0], "p_target"), *const draft = f32(a[1], "p_draft");
        const int32_t *const tokens = i32(a[2], "tokens"), *const parent = i32(a[3], "parent");
        const float *const u_accept = f32(a[4], "u_accept"), *const u_next = f32(a[5], "u_next");
        int32_t *const path = i32(a[6], "path"), *const n_path = i32(a[7], "n_path"), *const next = i32(a[8], "next_token");
        float *const alpha = f32(a[9], "alpha");
        void *const s = stream(a[10]);
        return status(unlocked([&] {
            return sv_accept(S, T, V, target, draft, tokens, parent, u_accept, u_next, path, n_path, next, alpha, s);
        }));
    });
}

// One layer of a verification step: selection (an anchor layer) into sel_idx / sel_cnt or the reuse of what is there, then
// attention, on the current stream.
// geom, kv, q, reps [layers][...], layer, seq_lens, budget, n_sink, n_local, sel_idx, sel_cnt, draft_k, draft_v, parent, out,
// lse, workspace, status_word, anchor, behind_own_layer -> (status, whether it is the selection's)
PyObject *verify_layer(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 20, [&]() -> PyObject * {
        const sv_geom g = geometry(a[0]);
        const sv_kv kv = cache(a[1]);
        const void *q = bf16(a[2], "q");
        int32_t *idx = i32(a[9], "sel_idx"), *cnt = i32(a[10], "sel_cnt");
        const int32_t max_sel = row_length(a[9], "sel_idx");
        const void *dk = bf16(a[11], "draft_k"), *dv = bf16(a[12], "draft_v");
        const int32_t *parent = i32(a[13], "parent");
        void *out = bf16(a[14], "out");
        float *lse = f32(a[15], "lse");
        const Scratch ws = scratch(a[16]);
        int32_t *word = i32(a[17], "status_word");
        const bool anchor = truth(a[18]), behind = truth(a[19]);
        void *s = stream(Py_None);
        const float *r = nullptr;
        const int32_t *lens = nullptr, *budget = nullptr;
        int32_t sink = 0, local = 0;
        if (anchor) {
            const at::Tensor &reps = tensor(a[3], at::kFloat, "reps");
            long long layer = integer(a[4]);
            if (layer < 0) layer += reps.size(0);
            r = reps.data_ptr<float>() + layer * reps.stride(0);
            lens = i32(a[5], "seq_lens"), budget = i32(a[6], "budget_blocks"), sink = int32(a[7]), local = int32(a[8]);
        }
        auto attn = behind && !anchor ? sv_verify_attn_reused : sv_verify_attn;
        bool selecting = anchor;
        const sv_status st = unlocked([&] {
            if (anchor) {
                const sv_status sel = sv_select_blocks(&g, q, r, lens, budget, sink, local, 0, nullptr, nullptr, idx, cnt, max_sel, nullptr, s);
                if (sel != SV_OK) return sel;
            }
            selecting = false;
            return attn(&g, q, &kv, dk, dv, parent, idx, cnt, max_sel, 0.f, out, lse, ws.p, ws.bytes, word, s);
        });
        if (st != SV_OK) return Py_BuildValue("(iO)", (int)st, selecting ? Py_True : Py_False);
        Py_RETURN_NONE;
    });
}

// ---------------------------------------------------------------------- a stack of layers

// Per-layer host flags as bytes.
const uint8_t *flags(PyObject *o, int32_t n)
{
    if (o == Py_None) return nullptr;
    if (!PyBytes_Check(o) || PyBytes_GET_SIZE(o) != n) {
        PyErr_SetString(PyExc_TypeError, "expected one byte per layer");
        throw ArgError{};
    }
    return reinterpret_cast<const uint8_t *>(PyBytes_AS_STRING(o));
}

// The layers of an engine: its table (uint8 tensor [n_layers][row bytes]) and the page table and lengths of a layer's sv_kv.
sv_layers stack(PyObject *table, PyObject *kv)
{
    const at::Tensor &t = tensor(table, at::kByte, "layer table");
    const sv_kv first = cache(kv);
    return {t.data_ptr(), first.block_table, first.seq_lens, (int32_t)t.size(0)};
}

// Pointer of a tensor stacked over all layers, or null when the argument is something else (a list of per-layer tensors, a
// strided view): the caller then goes layer by layer.
void *stacked(PyObject *o, int64_t n_layers)
{
    if (!THPVariable_Check(o)) return nullptr;
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.is_cuda() || t.scalar_type() != at::kBFloat16 || !t.is_contiguous() || t.dim() != 5 || t.size(0) != n_layers) return nullptr;
    return t.data_ptr();
}

// geom, kv -> the layer's row of a layer table, as bytes
PyObject *layer_row(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 2, [&]() -> PyObject * {
        const sv_geom g = geometry(a[0]);
        const sv_kv kv = cache(a[1]);
        PyObject *row = PyBytes_FromStringAndSize(nullptr, (Py_ssize_t)sv_layer_table_bytes(1));
        if (!row) return nullptr;
        const sv_status st = sv_layer_table(&g, &kv, 1, PyBytes_AS_STRING(row));
        if (st == SV_OK) return row;
        Py_DECREF(row);
        return status(st);
    });
}

// geom, n_layers, max_sel -> bytes
PyObject *workspace_bytes_layers(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 3, [&] {
        const sv_geom g = geometry(a[0]);
        return PyLong_FromSize_t(sv_workspace_bytes_layers(&g, int32(a[1]), int32(a[2])));
    });
}

// geom, n_layers, max_sel -> bytes
PyObject *workspace_bytes_host_step(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 3, [&] {
        const sv_geom g = geometry(a[0]);
        return PyLong_FromSize_t(sv_workspace_bytes_host_step(&g, int32(a[1]), int32(a[2])));
    });
}

// geom, table, kv, which (bytes or None), block_begin, block_end, reps
PyObject *block_reps_layers(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 7, [&] {
        const sv_geom g = geometry(a[0]);
        const sv_layers layers = stack(a[1], a[2]);
        const uint8_t *const which = flags(a[3], layers.n_layers);
        const int32_t begin = int32(a[4]), end = int32(a[5]);
        float *const reps = f32(a[6], "reps");
        void *const s = stream(Py_None);
        return status(unlocked([&] { return sv_block_reps_layers(&g, &layers, which, begin, end, reps, s); }));
    });
}

// Layers first .. end - 1 of a step on the current stream: the selections of their anchors in one launch, their attention in
// another (dense: attention only).  geom, table, kv, first, end, anchors, q, draft_k, draft_v, parent, out, reps, budget, n_sink,
// n_local, idx, cnt (None: dense), workspace, status_word -> None, (status, whether it is the selection's), or False when the
// inputs are not stacked tensors
PyObject *verify_layers(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 19, [&]() -> PyObject * {
        const sv_geom g = geometry(a[0]);
        const sv_layers layers = stack(a[1], a[2]);
        const int32_t first = int32(a[3]), end = int32(a[4]);
        const void *q = stacked(a[6], layers.n_layers), *dk = stacked(a[7], layers.n_layers), *dv = stacked(a[8], layers.n_layers);
        void *out = stacked(a[10], layers.n_layers);
        if (!q || !dk || !dv || !out) Py_RETURN_FALSE;
        const uint8_t *anchors = flags(a[5], layers.n_layers);
        const int32_t *parent = i32(a[9], "parent");
        const bool dense = a[15] == Py_None;
        int32_t *idx = i32(a[15], "idx"), *cnt = i32(a[16], "cnt");
        const int32_t max_sel = dense ? g.max_blocks : row_length(a[15], "idx");
        const Scratch ws = scratch(a[17]);
        void *s = stream(Py_None);
        int32_t *const word = i32(a[18], "status_word");
        const float *const reps = dense ? nullptr : f32(a[11], "reps");
        const int32_t *const budget = dense ? nullptr : i32(a[12], "budget_blocks");
        const int32_t sink = dense ? 0 : int32(a[13]), local = dense ? 0 : int32(a[14]);
        bool selecting = !dense;
        const sv_status st = unlocked([&] {
            if (!dense) {
                const sv_status sel = sv_select_blocks_layers(&g, &layers, first, end, anchors, q, reps, budget, sink, local, idx, cnt, max_sel, s);
                if (sel != SV_OK) return sel;
            }
            selecting = false;
            return sv_verify_attn_layers(&g, &layers, first, end, anchors, q, dk, dv, parent, idx, cnt, max_sel, 0.f, out, ws.p, ws.bytes, word, s);
        });
        if (st != SV_OK) return Py_BuildValue("(iO)", (int)st, selecting ? Py_True : Py_False);
        Py_RETURN_NONE;
    });
}

// Pointer of a stacked host tensor, or null: as stacked().
void *stacked_host(PyObject *o, const at::Tensor &like)
{
    if (!THPVariable_Check(o)) return nullptr;
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.is_cpu() || t.scalar_type() != at::kBFloat16 || !t.is_contiguous() || !t.sizes().equals(like.sizes())) return nullptr;
    return t.data_ptr();
}

void destroy_host_step(PyObject *capsule) { sv_host_step_destroy(static_cast<sv_host_step *>(PyCapsule_GetPointer(capsule, "sv_host_step"))); }

PyObject *host_step(PyObject *, PyObject *const *, Py_ssize_t n)
{
    return checked(n, 0, [&]() -> PyObject * {
        sv_host_step *h = sv_host_step_create();
        if (h) return PyCapsule_New(h, "sv_host_step", destroy_host_step);
        return status(SV_ERR_CUDA);
    });
}

// step, geom, table, kv, anchors, chunk_end (sequence of int), q_host, draft_k_host, draft_v_host, q, draft_k, draft_v, parent, reps, budget,
// n_sink, n_local, idx, cnt, out, out_host, workspace, status_word, refresh_tail, refresh_which (bytes or None),
// stream_in, stream_out
// -> status, or False when the tensors are not stacked ones.  chunk_end None: without chunks (the streams are then not looked at), and
// False also where that has no form
PyObject *verify_step_from_host(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 27, [&]() -> PyObject * {
        const bool direct = a[5] == Py_None;
        sv_host_step *h = direct ? nullptr : static_cast<sv_host_step *>(PyCapsule_GetPointer(a[0], "sv_host_step"));
        if (!h && !direct) throw ArgError{};
        const sv_geom g = geometry(a[1]);
        const sv_layers layers = stack(a[2], a[3]);
        void *dev[4], *host[4];   // q, draft K, draft V, out
        for (int i = 0; i < 4; ++i) {
            PyObject *d = i < 3 ? a[9 + i] : a[19], *o = i < 3 ? a[6 + i] : a[20];
            dev[i] = stacked(d, layers.n_layers);
            if (!dev[i]) Py_RETURN_FALSE;
            const at::Tensor &t = THPVariable_Unpack(d);
            if (t.size(1) != g.n_seq || t.size(2) != g.n_draft || t.size(3) != (i == 1 || i == 2 ? g.n_kv_heads : g.n_q_heads) || t.size(4) != g.head_dim)
                Py_RETURN_FALSE;
            host[i] = stacked_host(o, t);
            if (!host[i]) Py_RETURN_FALSE;
        }
        int32_t ends[SV_MAX_HOST_CHUNKS];
        const Py_ssize_t chunks = direct ? 0 : PySequence_Fast_GET_SIZE(a[5]);
        if (chunks > SV_MAX_HOST_CHUNKS) Py_RETURN_FALSE;
        for (Py_ssize_t c = 0; c < chunks; ++c) ends[c] = int32(PySequence_Fast_GET_ITEM(a[5], c));
        const Scratch ws = scratch(a[21]);
        const uint8_t *const anchors = flags(a[4], layers.n_layers), *const which = flags(a[24], layers.n_layers);
        const int32_t *const parent = i32(a[12], "parent"), *const budget = i32(a[14], "budget_blocks");
        float *const reps = f32(a[13], "reps");
        const int32_t sink = int32(a[15]), local = int32(a[16]), max_sel = row_length(a[17], "idx");
        int32_t *const idx = i32(a[17], "idx"), *const cnt = i32(a[18], "cnt"), *const word = i32(a[22], "status_word");
        const bool refresh = truth(a[23]);
        void *const s = stream(Py_None), *const in = direct ? s : stream(a[25]), *const back = direct ? s : stream(a[26]);
        const sv_status st = unlocked([&] {
            if (direct)
                return sv_verify_step_from_host_direct(&g, &layers, anchors, host[0], host[1], host[2], dev[0], dev[1], dev[2], parent, reps, budget,
                                                       sink, local, idx, cnt, max_sel, dev[3], host[3], ws.p, ws.bytes, word, refresh, which, s);
            return sv_verify_step_from_host(h, &g, &layers, anchors, ends, (int32_t)chunks, host[0], host[1], host[2], dev[0], dev[1], dev[2],
                                            parent, reps, budget, sink, local, idx, cnt, max_sel, dev[3], host[3], ws.p, ws.bytes, word,
                                            refresh, which, in, back, s);
        });
        if (direct && st == SV_ERR_UNSUPPORTED) Py_RETURN_FALSE;
        // the allocator of pinned memory must not hand these out again before the copies are through
        const auto device = c10::cuda::current_device();
        for (int i = 0; i < 4; ++i) {
            const at::Tensor &t = THPVariable_Unpack(i < 3 ? a[6 + i] : a[20]);
            void *const context = t.storage().data_ptr().get_context();
            if (!direct) at::getHostAllocator(at::kCUDA)->record_event(
                host[i], context, c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(i < 3 ? in : back), device).unwrap());
            at::getHostAllocator(at::kCUDA)->record_event(host[i], context, c10::cuda::getCurrentCUDAStream().unwrap());
        }
        return status(st);
    });
}

// geom, table, kv, draft_k, draft_v, path, n_path, seq_lens, counters, reps -> status, or False when the drafts are not stacked tensors
PyObject *kv_append_layers(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 10, [&]() -> PyObject * {
        const sv_geom g = geometry(a[0]);
        const sv_layers layers = stack(a[1], a[2]);
        const void *dk = stacked(a[3], layers.n_layers), *dv = stacked(a[4], layers.n_layers);
        int32_t *lens = i32(a[7], "seq_lens");
        if (!dk || !dv || lens != layers.seq_lens) Py_RETURN_FALSE;
        const int32_t *const rows = i32(a[5], "accept_idx"), *const n_rows = i32(a[6], "n_accept");
        const int32_t most = row_length(a[5], "accept_idx");
        uint32_t *const counters = reinterpret_cast<uint32_t *>(i32(a[8], "counters"));
        float *const reps = f32(a[9], "reps");
        void *const s = stream(Py_None);
        return status(unlocked([&] { return sv_kv_append_layers(&g, &layers, dk, dv, rows, n_rows, most, lens, counters, reps, s); }));
    });
}

// An uninitialised tensor with a storage of its own on the current device, past the dispatcher (for outputs that a kernel writes whole).
at::Tensor fresh(at::IntArrayRef sizes)
{
    return at::Tensor(at::detail::empty_generic(sizes, c10::cuda::CUDACachingAllocator::get(), c10::DispatchKeySet(c10::DispatchKey::CUDA), at::kInt,
                                                std::nullopt));
}

// accept with the outputs allocated here: p_target, p_draft, tokens, parent, u_accept, u_next, n_seq, n_draft
// -> (path, n_path, next_token), or a status
PyObject *accept_new(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return checked(n, 8, [&]() -> PyObject * {
        const at::Tensor &pt = tensor(a[0], at::kFloat, "p_target"), &pd = tensor(a[1], at::kFloat, "p_draft");
        const at::Tensor &tok = tensor(a[2], at::kInt, "tokens");
        const int64_t S = integer(a[6]), T = integer(a[7]);
        if (pt.dim() != 3 || pt.size(0) != S || pt.size(1) != T || !pd.sizes().equals(pt.sizes()) || !tok.sizes().equals({S, T})) {
            PyErr_SetString(PyExc_ValueError, "sv_accept: shapes disagree");
            throw ArgError{};
        }
        // Three tensors of their own: parts of one allocation are 0.2 us faster, and one that grows (resize_) runs over the next.  Acceptance, the
        // copy and the commit around it: 14.98 us with at::empty, 13.77 past the dispatcher; 13.37 as parts where this takes 13.60.
        at::Tensor path, n_path, next;
        {
            const c10::cuda::CUDAGuard guard(tok.device());
            path = fresh({S, T}), n_path = fresh({S}), next = fresh({S});
        }
        const int32_t V = (int32_t)pt.size(2), *const tokens = tok.data_ptr<int32_t>(), *const parent = i32(a[3], "parent");
        const float *const target = pt.data_ptr<float>(), *const draft = pd.data_ptr<float>();
        const float *const u_accept = f32(a[4], "u_accept"), *const u_next = f32(a[5], "u_next");
        void *const s = stream(Py_None);
        const sv_status st = unlocked([&] {
            return sv_accept((int32_t)S, (int32_t)T, V, target, draft, tokens, parent, u_accept, u_next, path.data_ptr<int32_t>(),
                             n_path.data_ptr<int32_t>(), next.data_ptr<int32_t>(), nullptr, s);
        });
        if (st != SV_OK) return status(st);
        return Py_BuildValue("(NNN)", THPVariable_Wrap(path), THPVariable_Wrap(n_path), THPVariable_Wrap(next));
    });
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(block_reps), METHOD(select_blocks), METHOD(verify_attn), METHOD(kv_append), METHOD(accept),
                         METHOD(verify_layer), METHOD(layer_row), METHOD(workspace_bytes_layers), METHOD(workspace_bytes_host_step), METHOD(block_reps_layers),
                         METHOD(verify_layers), METHOD(kv_append_layers), METHOD(accept_new), METHOD(host_step), METHOD(verify_step_from_host), {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Argument marshalling for the entry points of sv.h.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
