// Native half of the Python binding: checks the tensors, allocates what the caller did not pass, and calls the C ABI
// on the current stream.
//
// A call of the library is one to six short launches; done from Python (attribute look-ups, ctypes conversions
// of twenty arguments, torch.cuda.current_stream alone 3.2 us) the calls of a decoding step took 24 us on the host for
// 16 us of device time.  The functions take positional arguments in the order of their Python wrappers
// (binding.py), which hold the names, the defaults and the documentation.  The library's entry points arrive as
// addresses (bind), so that this module works with whichever build of the library the process has loaded.
#include <Python.h>

#include <vector>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/pulsar.h"

namespace {

#define PULSAR_ENTRIES(X)                                                                                          \
    X(pulsar_maxidf_select_workspace_bytes) X(pulsar_maxidf_select) X(pulsar_chunk_select_workspace_bytes)         \
    X(pulsar_chunk_select) X(pulsar_phase1_workspace_bytes) X(pulsar_phase1_attn) X(pulsar_pack_summary_kv)        \
    X(pulsar_gather_kv_rows) X(pulsar_phase1_attn_sharded) X(pulsar_causal_varlen_attn) X(pulsar_retain_block_kv)  \
    X(pulsar_phase2_choose_splits) X(pulsar_phase2_workspace_bytes) X(pulsar_phase2_attn)                          \
    X(pulsar_phase2_generate_workspace_bytes) X(pulsar_phase2_generate_step) X(pulsar_lse_merge_strided)           \
    X(pulsar_rope_apply_qk) X(pulsar_encode_step)

struct Entries {
#define X(name) decltype(&::name) name = nullptr;
    PULSAR_ENTRIES(X)
#undef X
} g;
PyObject* g_error = nullptr;                     // PulsarError(call, status)

// ---- arguments ------------------------------------------------------------------------------------------------------
struct Fail {};                                  // a Python error is set

[[noreturn]] void raise(PyObject* type, const std::string& text) {
    PyErr_SetString(type, text.c_str());
    throw Fail{};
}

struct Args {
    PyObject* const* v;
    Py_ssize_t n, i = 0;
    PyObject* next() {
        if (i >= n) raise(PyExc_TypeError, "too few arguments");
        return v[i++];
    }
    int64_t integer() {
        const int64_t x = PyLong_AsLongLong(next());
        if (x == -1 && PyErr_Occurred()) throw Fail{};
        return x;
    }
    // Sizes the C ABI takes as int32: a value outside it is outside every shape the kernels cover.
    int32_t i32() {
        const int64_t x = integer();
        if (x > INT32_MAX || x < INT32_MIN) raise(PyExc_OverflowError, "integer argument does not fit 32 bits");
        return static_cast<int32_t>(x);
    }
    double real() {
        const double x = PyFloat_AsDouble(next());
        if (x == -1.0 && PyErr_Occurred()) throw Fail{};
        return x;
    }
    bool truth() {
        const int x = PyObject_IsTrue(next());
        if (x < 0) throw Fail{};
        return x != 0;
    }
    // A tensor argument, or an undefined tensor for None.
    at::Tensor tensor() {
        PyObject* o = next();
        if (o == Py_None) return {};
        if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string("expected a tensor, got ") + Py_TYPE(o)->tp_name);
        return THPVariable_Unpack(o);
    }
    // The same with the requirements of the kernels.
    at::Tensor needed(at::ScalarType dtype, const char* name, int64_t dim = 0) {
        at::Tensor t = tensor();
        if (!t.defined() || !t.is_cuda() || t.scalar_type() != dtype || !t.is_contiguous())
            raise(PyExc_TypeError, std::string(name) + ": expected a contiguous CUDA tensor of " + at::toString(dtype) +
                                       (t.defined() ? std::string(", got ") + at::toString(t.scalar_type()) + " on " + t.device().str()
                                                    : std::string(", got None")));
        if (dim > 0 && t.dim() != dim) raise(PyExc_ValueError, std::string(name) + ": expected " + std::to_string(dim) + " dimensions");
        return t;
    }
    at::Tensor bf16(const char* name, int64_t dim = 0) { return needed(at::kBFloat16, name, dim); }
    at::Tensor i32s(const char* name) { return needed(at::kInt, name); }
    std::vector<int32_t> sequence() {
        PyObject* fast = PySequence_Fast(next(), "expected a sequence of integers");
        if (!fast) throw Fail{};
        std::vector<int32_t> out(static_cast<size_t>(PySequence_Fast_GET_SIZE(fast)));
        for (size_t k = 0; k < out.size(); ++k) {
            PyObject* x = PyNumber_Long(PySequence_Fast_GET_ITEM(fast, static_cast<Py_ssize_t>(k)));
            const long long value = x ? PyLong_AsLongLong(x) : -1;
            Py_XDECREF(x);
            if (value == -1 && PyErr_Occurred()) { Py_DECREF(fast); throw Fail{}; }
            out[k] = static_cast<int32_t>(value);
        }
        Py_DECREF(fast);
        return out;
    }
};

template <typename T> T* ptr(const at::Tensor& t) { return t.defined() ? static_cast<T*>(t.data_ptr()) : nullptr; }
const uint16_t* in16(const at::Tensor& t) { return ptr<uint16_t>(t); }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor empty(at::IntArrayRef sizes, at::ScalarType dtype, const at::Tensor& like) {
    return at::empty(sizes, like.options().dtype(dtype));
}
at::Tensor workspace_or(const at::Tensor& given, size_t bytes, const at::Tensor& like) {
    return given.defined() ? given : empty({static_cast<int64_t>(bytes > 256 ? bytes : 256)}, at::kByte, like);
}

// Calls an entry point without the GIL (a full launch queue makes a launch wait) and raises what it reports.
template <typename F> void call(const char* name, F&& f) {
    int32_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    if (rc == PULSAR_OK) return;
    PyObject* e = PyObject_CallFunction(g_error, "si", name, static_cast<int>(rc));
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Fail{};
}

PyObject* result(std::initializer_list<at::Tensor> ts) {
    PyObject* out = PyTuple_New(static_cast<Py_ssize_t>(ts.size()));
    if (!out) throw Fail{};
    Py_ssize_t i = 0;
    for (const at::Tensor& t : ts) {
        PyObject* o = Py_None;
        if (t.defined()) o = THPVariable_Wrap(t);
        else Py_INCREF(o);
        PyTuple_SET_ITEM(out, i++, o);
    }
    return out;
}

template <PyObject* (*F)(Args&)> PyObject* entry(PyObject*, PyObject* const* v, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    try {
        Args a{v, n};
        return F(a);
    } catch (const Fail&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// ---- selection ------------------------------------------------------------------------------------------------------
// The first n entries along the first dimension, fewer if there are not as many (t[:n]).
at::Tensor head(const at::Tensor& t, int64_t n) { return t.slice(0, 0, n); }

struct SelectShape {
    int32_t V, block, chunk, k, sink;
    int64_t L, B, C;
    SelectShape(Args& a, int64_t L_) : L(L_) {
        V = a.i32(); block = a.i32(); chunk = a.i32(); k = a.i32(); sink = a.i32();
        B = block > 0 ? (L + block - 1) / block : 0;               // the last block may be shorter
        C = chunk > 0 ? (static_cast<int64_t>(block) + chunk - 1) / chunk : 0;
    }
    static int64_t pos(int64_t x) { return x > 0 ? x : 0; }
    int64_t prefix() const { return sink + pos(B - 1) * k * chunk; }
    at::Tensor sel_buf(const at::Tensor& like) const { return empty({pos(B) * pos(k) + 4}, at::kInt, like); }
    at::Tensor prefix_buf(const at::Tensor& like) const {
        return empty({pos(sink) + pos(B - 1) * pos(k) * pos(chunk) + 4}, at::kInt, like);
    }
    at::Tensor len_buf(const at::Tensor& like) const { return empty({B > 1 ? B : 1}, at::kInt, like); }
};

// (token_ids, vocab, block, chunk, k, sink, df, idf, workspace, status, sel_buf, prefix_idx, prefix_len)
PyObject* maxidf_select(Args& a) {
    at::Tensor ids = a.i32s("token_ids");
    SelectShape z(a, ids.numel());
    at::Tensor df = a.tensor(), idf = a.tensor(), ws = a.tensor(), status = a.tensor(), sel = a.tensor(), pidx = a.tensor(),
               plen = a.tensor();
    if (!sel.defined()) {
        sel = z.sel_buf(ids);
        pidx = z.prefix_buf(ids);
        plen = z.len_buf(ids);
    }
    if (!ws.defined()) ws = workspace_or(ws, g.pulsar_maxidf_select_workspace_bytes(z.L, z.V, z.block, z.chunk, z.k, z.sink), ids);
    call("pulsar_maxidf_select", [&, st = stream()] {
        return g.pulsar_maxidf_select(ptr<uint32_t>(ids), z.L, z.V, z.block, z.chunk, z.k, z.sink, ptr<int32_t>(sel),
                                      ptr<int32_t>(pidx), ptr<int32_t>(plen), ptr<uint32_t>(df), ptr<float>(idf), ptr<void>(ws),
                                      static_cast<size_t>(ws.numel()), ptr<int32_t>(status), st);
    });
    return result({head(sel, z.B * z.k).view({z.B, z.k}), head(pidx, z.prefix()), head(plen, z.B)});
}

// (token_ids, vocab, block, chunk, k, sink, mode, want_score, workspace, status)
PyObject* chunk_select(Args& a) {
    at::Tensor ids = a.i32s("token_ids");
    SelectShape z(a, ids.numel());
    const int32_t mode = a.i32();
    const bool want_score = a.truth();
    at::Tensor ws = a.tensor(), status = a.tensor(), sel = z.sel_buf(ids), pidx = z.prefix_buf(ids), plen = z.len_buf(ids), score;
    if (want_score) score = empty({z.B > 1 ? z.B : 1, z.C > 1 ? z.C : 1}, at::kDouble, ids);
    if (!ws.defined())
        ws = workspace_or(ws, g.pulsar_chunk_select_workspace_bytes(z.L, z.V, z.block, z.chunk, z.k, z.sink, mode), ids);
    call("pulsar_chunk_select", [&, st = stream()] {
        return g.pulsar_chunk_select(ptr<uint32_t>(ids), z.L, z.V, z.block, z.chunk, z.k, z.sink, mode, ptr<int32_t>(sel),
                                     ptr<int32_t>(pidx), ptr<int32_t>(plen), ptr<double>(score), ptr<void>(ws),
                                     static_cast<size_t>(ws.numel()), ptr<int32_t>(status), st);
    });
    return result({head(sel, z.B * z.k).view({z.B, z.k}), head(pidx, z.prefix()), head(plen, z.B), score});
}

// ---- Phase 1 --------------------------------------------------------------------------------------------------------
struct Qkv {
    at::Tensor Q, K, V;
    int64_t rows;
    int32_t Hq, Hkv, d;
    explicit Qkv(Args& a) : Q(a.bf16("Q", 3)), K(a.bf16("K")), V(a.bf16("V")) {
        rows = Q.size(0);
        Hq = static_cast<int32_t>(Q.size(1));
        d = static_cast<int32_t>(Q.size(2));
        if (K.dim() < 2) raise(PyExc_ValueError, "K: expected 3 dimensions");
        Hkv = static_cast<int32_t>(K.size(1));
    }
    at::Tensor lse(bool want, const at::Tensor& given) const {
        return given.defined() || !want ? given : empty({rows, Hq}, at::kFloat, Q);
    }
};

// (Q, K, V, block, prefix_idx, prefix_len, scale, want_lse, retain_copy, out, lse_out, workspace, status)
PyObject* phase1_attn(Args& a) {
    Qkv x(a);
    const int32_t block = a.i32();
    at::Tensor pidx = a.tensor(), plen = a.i32s("prefix_len");
    if (!pidx.defined() || !pidx.is_cuda() || pidx.scalar_type() != at::kInt || !pidx.is_contiguous())
        raise(PyExc_TypeError, "prefix_idx: expected a contiguous CUDA tensor of Int");
    const int32_t total = static_cast<int32_t>(pidx.numel());
    const float scale = static_cast<float>(a.real());
    const bool want_lse = a.truth(), retain = a.truth();
    at::Tensor out = a.tensor(), lse = a.tensor(), ws = a.tensor(), status = a.tensor(), Kr, Vr;
    if (!out.defined()) out = at::empty_like(x.Q);
    lse = x.lse(want_lse, lse);
    if (retain) {
        Kr = at::empty_like(x.K);
        Vr = at::empty_like(x.V);
    }
    if (!ws.defined()) ws = workspace_or(ws, g.pulsar_phase1_workspace_bytes(x.rows, x.Hq, x.Hkv, x.d, block, total), x.Q);
    call("pulsar_phase1_attn", [&, st = stream()] {
        return g.pulsar_phase1_attn(in16(x.Q), in16(x.K), in16(x.V), x.rows, x.Hq, x.Hkv, x.d, block,
                                    total > 0 ? ptr<int32_t>(pidx) : nullptr, ptr<int32_t>(plen), total, scale,
                                    ptr<uint16_t>(out), ptr<float>(lse), ptr<uint16_t>(Kr), ptr<uint16_t>(Vr), ptr<void>(ws),
                                    static_cast<size_t>(ws.numel()), ptr<int32_t>(status), st);
    });
    return result({out, lse, Kr, Vr});
}

// (Q, K, V, block, K_prefix, V_prefix, prefix_len_local, scale, want_lse, out, lse_out, workspace, status)
PyObject* phase1_attn_sharded(Args& a) {
    Qkv x(a);
    const int32_t block = a.i32();
    at::Tensor Kp = a.tensor(), Vp = a.tensor(), plen = a.i32s("prefix_len_local");
    const int32_t total = Kp.defined() ? static_cast<int32_t>(Kp.size(0)) : 0;
    if (total > 0)
        for (const at::Tensor* t : {&Kp, &Vp})
            if (!t->defined() || !t->is_cuda() || t->scalar_type() != at::kBFloat16 || !t->is_contiguous())
                raise(PyExc_TypeError, "K_prefix, V_prefix: expected contiguous CUDA tensors of BFloat16");
    const float scale = static_cast<float>(a.real());
    const bool want_lse = a.truth();
    at::Tensor out = a.tensor(), lse = a.tensor(), ws = a.tensor(), status = a.tensor();
    if (!out.defined()) out = at::empty_like(x.Q);
    lse = x.lse(want_lse, lse);
    ws = workspace_or(ws, 256, x.Q);
    call("pulsar_phase1_attn_sharded", [&, st = stream()] {
        return g.pulsar_phase1_attn_sharded(in16(x.Q), in16(x.K), in16(x.V), x.rows, x.Hq, x.Hkv, x.d, block,
                                            total > 0 ? in16(Kp) : nullptr, total > 0 ? in16(Vp) : nullptr, total,
                                            ptr<int32_t>(plen), scale, ptr<uint16_t>(out), ptr<float>(lse), ptr<void>(ws),
                                            static_cast<size_t>(ws.numel()), ptr<int32_t>(status), st);
    });
    return result({out, lse});
}

// (Q, K, V, cu_seqlens, scale, want_lse, out, workspace, status)
PyObject* causal_varlen_attn(Args& a) {
    Qkv x(a);
    const std::vector<int32_t> cu = a.sequence();
    const float scale = static_cast<float>(a.real());
    const bool want_lse = a.truth();
    at::Tensor out = a.tensor(), ws = a.tensor(), status = a.tensor(), lse = x.lse(want_lse, {});
    if (!out.defined()) out = at::empty_like(x.Q);
    ws = workspace_or(ws, 256, x.Q);
    call("pulsar_causal_varlen_attn", [&, st = stream()] {
        return g.pulsar_causal_varlen_attn(in16(x.Q), in16(x.K), in16(x.V), x.rows, cu.data(),
                                           static_cast<int32_t>(cu.size()) - 1, x.Hq, x.Hkv, x.d, scale, ptr<uint16_t>(out),
                                           ptr<float>(lse), ptr<void>(ws), static_cast<size_t>(ws.numel()),
                                           ptr<int32_t>(status), st);
    });
    return result({out, lse});
}

// (K, V, cu_seqlens, block)
PyObject* retain_block_kv(Args& a) {
    at::Tensor K = a.bf16("K"), V = a.bf16("V");
    if (K.dim() < 3) raise(PyExc_ValueError, "K: expected 3 dimensions");
    const std::vector<int32_t> cu = a.sequence();
    const int32_t block = a.i32(), n_seq = static_cast<int32_t>(cu.size()) - 1;
    std::vector<int64_t> sizes = K.sizes().vec();
    sizes[0] = static_cast<int64_t>(n_seq) * block;
    at::Tensor Kr = empty(sizes, at::kBFloat16, K), Vr = at::empty_like(Kr);
    call("pulsar_retain_block_kv", [&, st = stream()] {
        return g.pulsar_retain_block_kv(in16(K), in16(V), K.size(0), cu.data(), n_seq, block, static_cast<int32_t>(K.size(1)),
                                        static_cast<int32_t>(K.size(2)), ptr<uint16_t>(Kr), ptr<uint16_t>(Vr), st);
    });
    return result({Kr, Vr});
}

// (K, V, block, sel_chunks, block_ids, n_blocks, chunk, k, sink, K_send, V_send, status)
PyObject* pack_summary_kv(Args& a) {
    at::Tensor K = a.bf16("K"), V = a.bf16("V");
    const int32_t block = a.i32();
    at::Tensor sel = a.i32s("sel_chunks"), ids = a.i32s("block_ids");
    const int32_t n_blocks = a.i32(), chunk = a.i32(), k = a.i32(), sink = a.i32();
    at::Tensor Ks = a.bf16("K_send"), Vs = a.bf16("V_send"), status = a.tensor();
    const int32_t Hkv = static_cast<int32_t>(K.size(-2)), d = static_cast<int32_t>(K.size(-1));
    call("pulsar_pack_summary_kv", [&, st = stream()] {
        return g.pulsar_pack_summary_kv(in16(K), in16(V), static_cast<int32_t>(ids.numel()), block, Hkv, d, ptr<int32_t>(sel),
                                        ptr<int32_t>(ids), n_blocks, chunk, k, sink, ptr<uint16_t>(Ks), ptr<uint16_t>(Vs),
                                        ptr<int32_t>(status), st);
    });
    Py_RETURN_NONE;
}

// (K, V, idx, K_out, V_out, status)
PyObject* gather_kv_rows(Args& a) {
    at::Tensor K = a.bf16("K"), V = a.bf16("V"), idx = a.i32s("idx"), Ko = a.bf16("K_out"), Vo = a.bf16("V_out"), status = a.tensor();
    const int32_t Hkv = static_cast<int32_t>(K.size(-2)), d = static_cast<int32_t>(K.size(-1));
    call("pulsar_gather_kv_rows", [&, st = stream()] {
        return g.pulsar_gather_kv_rows(in16(K), in16(V), K.size(0), Hkv, d, ptr<int32_t>(idx), static_cast<int32_t>(idx.numel()),
                                       ptr<uint16_t>(Ko), ptr<uint16_t>(Vo), ptr<int32_t>(status), st);
    });
    Py_RETURN_NONE;
}

// ---- Phase 2 --------------------------------------------------------------------------------------------------------
struct Query {
    at::Tensor Q, K, V;
    int32_t nq, Hq, Hkv, d;
    void shape() {
        nq = static_cast<int32_t>(Q.size(0));
        Hq = static_cast<int32_t>(Q.size(1));
        d = static_cast<int32_t>(Q.size(2));
        if (K.dim() < 2) raise(PyExc_ValueError, "Kblocks: expected 3 dimensions");
        Hkv = static_cast<int32_t>(K.size(-2));
    }
};

// (Qq, K, V, n_blocks, block, scale, n_splits, want_partials, out, lse_out, workspace, status, part_O, part_LSE)
PyObject* phase2_attn(Args& a) {
    Query x;
    x.Q = a.bf16("Qq", 3);
    x.K = a.bf16("Kblocks");
    x.V = a.bf16("Vblocks");
    x.shape();
    const int32_t B = a.i32(), block = a.i32();
    const float scale = static_cast<float>(a.real());
    int32_t splits = a.i32();
    const bool want_partials = a.truth();
    at::Tensor out = a.tensor(), lse = a.tensor(), ws = a.tensor(), status = a.tensor(), pO = a.tensor(), pL = a.tensor();
    if (!out.defined()) out = at::empty_like(x.Q);
    if (!lse.defined()) lse = empty({x.nq, x.Hq}, at::kFloat, x.Q);
    if (pO.defined()) {
        for (const at::Tensor* t : {&pO, &pL})
            if (!t->defined() || !t->is_cuda() || t->scalar_type() != at::kFloat || !t->is_contiguous())
                raise(PyExc_TypeError, "partials: expected contiguous CUDA tensors of Float");
    } else if (want_partials) {
        pO = empty({splits, x.nq, x.Hq, x.d}, at::kFloat, x.Q);
        pL = empty({splits, x.nq, x.Hq}, at::kFloat, x.Q);
    }
    if (!ws.defined()) {
        if (splits == 0 && !pO.defined()) splits = g.pulsar_phase2_choose_splits(x.nq, B, block, x.Hq, x.Hkv, x.d);
        ws = workspace_or(ws, g.pulsar_phase2_workspace_bytes(x.nq, B, block, x.Hq, x.Hkv, x.d, splits), x.Q);
    }
    call("pulsar_phase2_attn", [&, st = stream()] {
        return g.pulsar_phase2_attn(in16(x.Q), x.nq, in16(x.K), in16(x.V), B, block, x.Hq, x.Hkv, x.d, scale, splits,
                                    ptr<uint16_t>(out), ptr<float>(lse), ptr<float>(pO), ptr<float>(pL), ptr<void>(ws),
                                    static_cast<size_t>(ws.numel()), ptr<int32_t>(status), st);
    });
    return result({out, lse, pO, pL});
}

// (Qnew, Knew, Vnew, K, V, n_blocks, block, Kgen, Vgen, gen_len, scale, n_splits, out, workspace, status)
PyObject* phase2_generate_step(Args& a) {
    Query x;
    x.Q = a.bf16("Qnew", 3);
    at::Tensor Kn = a.bf16("Knew"), Vn = a.bf16("Vnew");
    x.K = a.bf16("Kblocks");
    x.V = a.bf16("Vblocks");
    x.shape();
    const int32_t B = a.i32(), block = a.i32();
    at::Tensor Kg = a.bf16("Kgen"), Vg = a.bf16("Vgen");
    const int32_t gen_len = a.i32();
    const float scale = static_cast<float>(a.real());
    int32_t splits = a.i32();
    at::Tensor out = a.tensor(), ws = a.tensor(), status = a.tensor(), lse = empty({x.nq, x.Hq}, at::kFloat, x.Q);
    if (splits == 0) splits = g.pulsar_phase2_choose_splits(x.nq, B, block, x.Hq, x.Hkv, x.d);
    if (!out.defined()) out = at::empty_like(x.Q);
    if (!ws.defined())
        ws = workspace_or(ws, g.pulsar_phase2_generate_workspace_bytes(x.nq, B, block, x.Hq, x.Hkv, x.d, splits), x.Q);
    call("pulsar_phase2_generate_step", [&, st = stream()] {
        return g.pulsar_phase2_generate_step(in16(x.Q), in16(Kn), in16(Vn), x.nq, in16(x.K), in16(x.V), B, block,
                                             ptr<uint16_t>(Kg), ptr<uint16_t>(Vg), gen_len, static_cast<int32_t>(Kg.size(0)),
                                             x.Hq, x.Hkv, x.d, scale, splits, ptr<uint16_t>(out), ptr<float>(lse), ptr<void>(ws),
                                             static_cast<size_t>(ws.numel()), ptr<int32_t>(status), st);
    });
    return result({out, lse});
}

// (token_ids, vocab, block, chunk, k, sink, Q, K, V, Qq, scale, n_splits, status, sel_buf, prefix_idx, prefix_len, O1, LSE1, O2,
//  LSE2, ws_select, ws_phase1, ws_phase2): the three calls of a step with everything preallocated; LSE1 and LSE2 may be None
PyObject* encode_step(Args& a) {
    at::Tensor ids = a.i32s("token_ids");
    SelectShape z(a, ids.numel());
    Qkv x(a);
    at::Tensor Qq = a.bf16("Qq", 3);
    const float scale = static_cast<float>(a.real());
    const int32_t splits = a.i32();
    at::Tensor status = a.tensor();
    const int64_t nq = Qq.size(0);
    if (x.rows != z.L) raise(PyExc_ValueError, "one token id per row of Q, K and V");
    if (Qq.size(1) != x.Hq || Qq.size(2) != x.d) raise(PyExc_ValueError, "Qq: expected the heads and the head size of Q");
    const auto output = [&](at::ScalarType dtype, const char* name, int64_t n) {
        at::Tensor t = a.needed(dtype, name);
        if (t.numel() < n) raise(PyExc_ValueError, std::string(name) + ": expected at least " + std::to_string(n) + " entries");
        return t;
    };
    const auto lse = [&](const char* name, int64_t n) {
        if (a.i < a.n && a.v[a.i] == Py_None) return a.tensor();
        return output(at::kFloat, name, n);
    };
    at::Tensor sel = output(at::kInt, "sel_chunks", z.B * z.k), pidx = output(at::kInt, "prefix_idx", z.prefix()),
               plen = output(at::kInt, "prefix_len", z.B), O1 = output(at::kBFloat16, "O", x.rows * x.Hq * x.d),
               LSE1 = lse("LSE", x.rows * x.Hq), O2 = output(at::kBFloat16, "O2", nq * x.Hq * x.d), LSE2 = lse("LSE2", nq * x.Hq),
               ws_s = output(at::kByte, "selection workspace", 0), ws_1 = output(at::kByte, "Phase-1 workspace", 0),
               ws_2 = output(at::kByte, "Phase-2 workspace", 0);                       // (their sizes are the library's to check)
    call("pulsar_encode_step", [&, st = stream()] {
        return g.pulsar_encode_step(ptr<uint32_t>(ids), z.L, z.V, z.block, z.chunk, z.k, z.sink, ptr<int32_t>(sel), ptr<int32_t>(pidx),
                                    ptr<int32_t>(plen), ptr<void>(ws_s), static_cast<size_t>(ws_s.numel()), in16(x.Q), in16(x.K),
                                    in16(x.V), x.Hq, x.Hkv, x.d, static_cast<int32_t>(z.prefix()), scale, ptr<uint16_t>(O1),
                                    ptr<float>(LSE1), ptr<void>(ws_1), static_cast<size_t>(ws_1.numel()), in16(Qq),
                                    static_cast<int32_t>(nq), splits, ptr<uint16_t>(O2), ptr<float>(LSE2), ptr<void>(ws_2),
                                    static_cast<size_t>(ws_2.numel()), ptr<int32_t>(status), st);
    });
    return result({head(sel, z.B * z.k).view({z.B, z.k}), head(pidx, z.prefix()), head(plen, z.B)});
}

// (part_O, part_LSE, n_parts, stride_O, stride_LSE, rows, d, out, lse_out)
PyObject* lse_merge_strided(Args& a) {
    at::Tensor pO = a.needed(at::kFloat, "part_O"), pL = a.needed(at::kFloat, "part_LSE");
    const int32_t n_parts = a.i32();
    const int64_t stride_O = a.integer(), stride_L = a.integer(), rows = a.integer();
    const int32_t d = a.i32();
    at::Tensor out = a.tensor(), lse = a.tensor();
    if (!out.defined() || (out.scalar_type() != at::kFloat && out.scalar_type() != at::kBFloat16))
        raise(PyExc_TypeError, "out must be float32 or bfloat16");
    call("pulsar_lse_merge_strided", [&, st = stream()] {
        return g.pulsar_lse_merge_strided(ptr<float>(pO), ptr<float>(pL), n_parts, stride_O, stride_L, rows, d, ptr<void>(out),
                                          out.scalar_type() == at::kFloat ? 1 : 0, ptr<float>(lse), st);
    });
    Py_RETURN_NONE;
}

// (Q, K, positions, theta, q_out, k_out, status)
PyObject* rope_apply_qk(Args& a) {
    at::Tensor Q = a.bf16("Q", 3), K = a.bf16("K"), pos = a.i32s("positions");
    const double theta = a.real();
    at::Tensor Qo = a.tensor(), Ko = a.tensor(), status = a.tensor();
    const int64_t rows = Q.size(0), d = Q.size(2);
    if (K.dim() < 3 || K.size(0) != rows || K.size(2) != d || pos.numel() != rows)
        raise(PyExc_ValueError, "Q, K and positions must cover the same rows and head size");
    if (!Qo.defined()) Qo = at::empty_like(Q);
    if (!Ko.defined()) Ko = at::empty_like(K);
    call("pulsar_rope_apply_qk", [&, st = stream()] {
        return g.pulsar_rope_apply_qk(in16(Q), ptr<uint16_t>(Qo), static_cast<int32_t>(Q.size(1)), in16(K), ptr<uint16_t>(Ko),
                                      static_cast<int32_t>(K.size(1)), rows, static_cast<int32_t>(d), ptr<int32_t>(pos), theta,
                                      ptr<int32_t>(status), st);
    });
    return result({Qo, Ko});
}

// bind({name: address}, error class): the library build to call.
PyObject* bind(Args& a) {
    PyObject* table = a.next();
    PyObject* error = a.next();
#define X(name)                                                                                     \
    {                                                                                               \
        PyObject* o = PyDict_GetItemString(table, #name);                                           \
        void* p = o ? PyLong_AsVoidPtr(o) : nullptr;                                                \
        if (!p) raise(PyExc_ValueError, "no address for " #name);                                   \
        g.name = reinterpret_cast<decltype(&::name)>(p);                                              \
    }
    PULSAR_ENTRIES(X)
#undef X
    Py_INCREF(error);
    Py_XSETREF(g_error, error);
    Py_RETURN_NONE;
}

#define M(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {M(bind), M(maxidf_select), M(chunk_select), M(phase1_attn), M(phase1_attn_sharded), M(causal_varlen_attn),
                         M(retain_block_kv), M(pack_summary_kv), M(gather_kv_rows), M(phase2_attn), M(phase2_generate_step),
                         M(lse_merge_strided), M(rope_apply_qk), M(encode_step), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
