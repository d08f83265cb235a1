// Native side of the Python binding: the hot entry points (forward, hybrid, block lists, 8-bit operands, backward,
// decode) with torch tensors in and out.  It checks and marshals the arguments, allocates the outputs on torch's
// caching allocator and calls the C entry points of libattnfuse on the current stream; it does no arithmetic.
//
// Why it is native: a small call is bound by its host time, and marshalling the same arguments with ctypes took more of it
// than the launch.  Back-to-back calls, ctypes against this module: forward at B = 1, 2 heads, S = 128, D = 64 21.9 us
// against 8.2 us; decode at 32 q / 8 kv heads, 4096 keys, D = 128 19.7 us against 10.3 us.
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/attnfuse.h"

namespace {

// entry points of libattnfuse, bound once by binding.py from the library it has loaded
struct Api {
    decltype(&attnfuse_strerror) strerror_;
    decltype(&attnfuse_fwd) fwd;
    decltype(&attnfuse_fwd_scratch) fwd_scratch;
    decltype(&attnfuse_fwd_scratch_bytes) fwd_scratch_bytes;
    decltype(&attnfuse_fwd_hybrid) fwd_hybrid;
    decltype(&attnfuse_fwd_hybrid_workspace_bytes) fwd_hybrid_workspace_bytes;
    decltype(&attnfuse_fwd_blocks) fwd_blocks;
    decltype(&attnfuse_fwd_fp8) fwd_fp8;
    decltype(&attnfuse_bwd) bwd;
    decltype(&attnfuse_bwd_blocks) bwd_blocks;
    decltype(&attnfuse_bwd_onepass_workspace_bytes) bwd_onepass_workspace_bytes;
    decltype(&attnfuse_decode) decode;
    decltype(&attnfuse_decode_splits) decode_splits;
    decltype(&attnfuse_decode_workspace_bytes) decode_workspace_bytes;
} api;
PyObject* error_class = nullptr;

// attribute names, interned once
struct Names {
    PyObject *theta, *rotary_dim, *pos_offset, *causal, *window, *alibi_slopes, *nb, *row_ptr, *col_idx, *col_ptr, *row_idx,
        *row_order, *col_order, *pair_ptr, *pair_idx, *pair_order, *col_longest, *listed;
} names;

struct Raised {};   // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* msg) {
    PyErr_SetString(type, msg);
    throw Raised();
}
void require(bool ok, const char* msg) {
    if (!ok) raise(PyExc_AssertionError, msg);
}
[[noreturn]] void raise_status(int code, const char* msg) {
    PyObject* e = PyObject_CallFunction(error_class, "is", code, msg);
    if (e) {
        PyErr_SetObject(error_class, e);
        Py_DECREF(e);
    }
    throw Raised();
}

// An owned attribute of a spec object.
struct Attr {
    PyObject* v;
    Attr(PyObject* o, PyObject* name) : v(PyObject_GetAttr(o, name)) {
        if (!v) throw Raised();
    }
    Attr(const Attr&) = delete;
    ~Attr() { Py_DECREF(v); }
    long as_int() const {
        const long r = PyLong_AsLong(v);
        if (r == -1 && PyErr_Occurred()) throw Raised();
        return r;
    }
    double as_double() const {
        const double r = PyFloat_AsDouble(v);
        if (r == -1.0 && PyErr_Occurred()) throw Raised();
        return r;
    }
    bool as_bool() const {
        const int r = PyObject_IsTrue(v);
        if (r < 0) throw Raised();
        return r != 0;
    }
};

// A tensor argument; None gives nullptr.  Tensors must live on a CUDA device.
const at::Tensor* tensor(PyObject* o) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch.Tensor");
    const at::Tensor* t = &THPVariable_Unpack(o);
    if (!t->is_cuda()) raise_status(-2, "tensor is not on a CUDA device (there is no CPU path)");
    return t;
}
const at::Tensor& need(PyObject* o) {
    const at::Tensor* t = tensor(o);
    if (!t) raise(PyExc_TypeError, "a tensor is required here, not None");
    return *t;
}
void* ptr(const at::Tensor* t) { return t ? t->data_ptr() : nullptr; }

// float(o): a number, a one-element tensor, a text
double number(PyObject* o) {
    PyObject* f = PyNumber_Float(o);
    if (!f) throw Raised();
    const double r = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return r;
}
// int(o), its low 32 bits: also of a float or a text
int integer(PyObject* o) {
    PyObject* l = PyNumber_Long(o);
    if (!l) throw Raised();
    const unsigned long r = PyLong_AsUnsignedLongMask(l);
    Py_DECREF(l);
    if (r == static_cast<unsigned long>(-1) && PyErr_Occurred()) throw Raised();
    return static_cast<int>(r);
}
at::ScalarType dtype(PyObject* o) {
    if (!THPDtype_Check(o)) raise(PyExc_TypeError, "expected a torch.dtype");
    return reinterpret_cast<THPDtype*>(o)->scalar_type;
}
bool truth(PyObject* o) {
    const int r = PyObject_IsTrue(o);
    if (r < 0) throw Raised();
    return r != 0;
}
af_dtype out_code(at::ScalarType t) { return t == at::kFloat ? AF_F32 : AF_BF16; }

af_rope rope_of(PyObject* spec) {
    return {static_cast<float>(Attr(spec, names.theta).as_double()), static_cast<int>(Attr(spec, names.rotary_dim).as_int()),
            static_cast<int>(Attr(spec, names.pos_offset).as_int())};
}
af_mask mask_of(PyObject* spec) {
    af_mask m;
    m.causal = Attr(spec, names.causal).as_bool() ? 1 : 0;
    m.window = integer(Attr(spec, names.window).v);
    const Attr slopes(spec, names.alibi_slopes);
    const at::Tensor* sl = tensor(slopes.v);
    require(!sl || (sl->scalar_type() == at::kFloat && sl->is_contiguous()), "alibi_slopes: fp32, contiguous");
    m.alibi_slopes = static_cast<const float*>(ptr(sl));
    return m;
}
const int* index_list(PyObject* mask, PyObject* name) {
    const Attr a(mask, name);
    return static_cast<const int*>(need(a.v).data_ptr());
}
af_blocks blocks_of(PyObject* mask, int64_t S) {
    require(Attr(mask, names.nb).as_int() == (S + 127) / 128, "block mask of another sequence length");
    return {128, index_list(mask, names.row_ptr), index_list(mask, names.col_idx), index_list(mask, names.col_ptr),
            index_list(mask, names.row_idx), index_list(mask, names.row_order), index_list(mask, names.col_order),
            index_list(mask, names.pair_ptr), index_list(mask, names.pair_idx), index_list(mask, names.pair_order),
            integer(Attr(mask, names.col_longest).v), integer(Attr(mask, names.listed).v)};
}

af_strides strides_of(const at::Tensor& t) {
    require(t.dim() == 4 && t.stride(3) == 1, "expected a 4-D tensor with a contiguous last dimension");
    return {t.stride(0), t.stride(1), t.stride(2)};
}
at::Tensor empty(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) {
    return at::detail::empty_cuda(sizes, type, like.device(), std::nullopt);
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Does the memory belong to the private pool that torch makes for a graph?  (A user's own pools have a zero there.)
bool in_graph_pool(const void* p) {
    const size_t a = reinterpret_cast<size_t>(p);
    for (const auto& s : c10::cuda::CUDACachingAllocator::snapshot({0, 0}, false).segments)
        if (s.address <= a && a - s.address < s.total_size) return s.owner_private_pool_id.first != 0;
    return false;
}

// Memory that a call works faster with but does not need: from torch's allocator, on the device and for the stream of the launch (its
// reuse is then ordered).  An undefined tensor where there is none to be had, for whatever reason: the call must not fail over it.
// `allocates`: the call allocates its outputs anyway.  One with outputs of the caller's own allocates nothing while its stream is being
// captured (a capture that torch does not know of would be broken by it), and no capture of another stream, by this thread or
// another, may be broken by a cudaMalloc here: the thread's capture mode is relaxed meanwhile.
// A captured launch writes the memory at every replay, long after this call has given it back: only the pool of torch's own graph,
// which nobody outside the graph is served from, is lent to one.
at::Tensor scratch_if_any(size_t bytes, bool allocates) {
    try {
        const bool captured = c10::cuda::currentStreamCaptureStatusMayInitCtx() != c10::cuda::CaptureStatus::None;
        if (captured && !allocates) return {};
        const c10::cuda::CUDAStreamCaptureModeGuard relaxed(cudaStreamCaptureModeRelaxed);
        at::Tensor t = at::detail::empty_cuda({static_cast<int64_t>(bytes)}, at::kByte, c10::Device(c10::kCUDA, c10::cuda::current_device()), std::nullopt);
        if ((reinterpret_cast<uintptr_t>(t.data_ptr()) & 15) == 0 && (!captured || in_graph_pool(t.data_ptr()))) return t;
    } catch (const std::exception&) {   // (any allocator's: torch's own raises several, one plugged in by the user its own)
    }
    return {};
}

// Runs a C entry point without the interpreter lock (a launch may block while the device's queue is full).  The arguments are
// plain values, evaluated by the caller while it holds the lock: data_ptr() of a tensor without storage throws.
template <typename... P, typename... A>
void call(af_status (*entry_point)(P...), A... args) {
    int code;
    {
        struct Released {
            PyThreadState* state = PyEval_SaveThread();
            ~Released() { PyEval_RestoreThread(state); }
        } released;
        code = static_cast<int>(entry_point(args...));
    }
    if (code != 0) raise_status(code, api.strerror_(static_cast<af_status>(code)));
}

// The caller's own object, or a new tensor.
struct Out {
    PyObject* given;   // borrowed, nullptr when allocated here
    at::Tensor t;
    bool any = true;
    Out(PyObject* o, bool wanted, at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) : given(nullptr) {
        if (const at::Tensor* g = tensor(o)) {
            given = o;
            t = *g;
        } else if (wanted) {
            t = empty(sizes, type, like);
        } else {
            any = false;
        }
    }
    void* data() const { return any ? t.data_ptr() : nullptr; }
    PyObject* result() {
        if (given) return Py_NewRef(given);
        if (!any) Py_RETURN_NONE;
        return THPVariable_Wrap(std::move(t));
    }
};
PyObject* pair(Out& a, Out& b) {
    PyObject* x = a.result();
    PyObject* y = x ? b.result() : nullptr;
    PyObject* r = y ? PyTuple_Pack(2, x, y) : nullptr;
    Py_XDECREF(x);
    Py_XDECREF(y);
    if (!r) throw Raised();
    return r;
}

// q [B,Hq,S,D], k and v [B,Hkv,S,D] bf16
struct Qkv {
    const at::Tensor &q, &k, &v;
    af_shape sh;
    af_strides sq, skv;
    int group;
    Qkv(PyObject* q_, PyObject* k_, PyObject* v_, bool check = true) : q(need(q_)), k(need(k_)), v(need(v_)) {
        require(q.dim() == 4 && k.dim() == 4, "q, k, v: [B, H, S, D]");
        if (check) {
            require(q.scalar_type() == at::kBFloat16 && k.scalar_type() == at::kBFloat16 && v.scalar_type() == at::kBFloat16,
                    "q, k, v: bf16");
            require(k.sizes() == v.sizes() && k.strides() == v.strides() && k.size(0) == q.size(0) && k.size(2) == q.size(2) &&
                        k.size(3) == q.size(3),
                    "k and v: [B, Hkv, S, D] of q's B, S, D, with the same strides");
        }
        sh = {static_cast<int>(q.size(0)), static_cast<int>(q.size(1)), static_cast<int>(k.size(1)), static_cast<int>(q.size(2)),
              static_cast<int>(q.size(3))};
        sq = strides_of(q);
        skv = strides_of(k);
        group = sh.Hkv > 0 ? sh.Hq / sh.Hkv : 0;
    }
};

void check_args(Py_ssize_t got, Py_ssize_t want) {
    if (got != want) raise(PyExc_TypeError, "wrong number of arguments");
}

// fwd(q, k, v, rope, table, mask, scale, out, lse, out_dtype, want_lse)
PyObject* fwd(PyObject* const* a, Py_ssize_t n) {
    check_args(n, 11);
    Qkv x(a[0], a[1], a[2]);
    const af_rope r = rope_of(a[3]);
    const at::Tensor* table = tensor(a[4]);
    const af_mask m = mask_of(a[5]);
    const float scale = static_cast<float>(number(a[6]));
    Out o(a[7], true, x.q.sizes(), dtype(a[9]), x.q);
    Out l(a[8], truth(a[10]), {x.sh.B, x.sh.Hq, x.sh.S}, at::kFloat, x.q);
    require(o.t.is_contiguous() && (o.t.scalar_type() == at::kBFloat16 || o.t.scalar_type() == at::kFloat), "out: contiguous, bf16 or fp32");
    const size_t bytes = api.fwd_scratch_bytes(&x.sh, &r, &m, x.group);
    const at::Tensor scratch = bytes ? scratch_if_any(bytes, !(o.given && (l.given || !l.any))) : at::Tensor();
    const bool lent = scratch.defined();
    call(api.fwd_scratch, &x.sh, x.q.data_ptr(), x.k.data_ptr(), x.v.data_ptr(), &x.sq, &x.skv, &r, ptr(table), &m, x.group, scale,
         o.data(), out_code(o.t.scalar_type()), static_cast<float*>(l.data()), lent ? scratch.data_ptr() : nullptr,
         lent ? scratch.nbytes() : size_t{0}, stream());
    return pair(o, l);
}

// fwd_hybrid(q, k, v, rope, table, mask, scale, out, lse, out_dtype, want_lse, workspace)
PyObject* fwd_hybrid(PyObject* const* a, Py_ssize_t n) {
    check_args(n, 12);
    Qkv x(a[0], a[1], a[2]);
    const af_rope r = rope_of(a[3]);
    const at::Tensor* table = tensor(a[4]);
    const af_mask m = mask_of(a[5]);
    const float scale = static_cast<float>(number(a[6]));
    Out o(a[7], true, x.q.sizes(), dtype(a[9]), x.q);
    Out l(a[8], truth(a[10]), {x.sh.B, x.sh.Hq, x.sh.S}, at::kFloat, x.q);
    require(o.t.is_contiguous() && (o.t.scalar_type() == at::kBFloat16 || o.t.scalar_type() == at::kFloat), "out: contiguous, bf16 or fp32");
    const at::Tensor* given = tensor(a[11]);
    const at::Tensor ws = given ? *given : empty({static_cast<int64_t>(api.fwd_hybrid_workspace_bytes(&x.sh))}, at::kByte, x.q);
    call(api.fwd_hybrid, &x.sh, x.q.data_ptr(), x.k.data_ptr(), x.v.data_ptr(), &x.sq, &x.skv, &r, ptr(table), &m, x.group,
         scale, o.data(), out_code(o.t.scalar_type()), static_cast<float*>(l.data()), ws.data_ptr(), ws.nbytes(), stream());
    return pair(o, l);
}

// fwd_blocks(q, k, v, rope, table, mask, scale, blocks, out, lse, out_dtype)
PyObject* fwd_blocks(PyObject* const* a, Py_ssize_t n) {
    check_args(n, 11);
    Qkv x(a[0], a[1], a[2]);
    const af_rope r = rope_of(a[3]);
    const at::Tensor* table = tensor(a[4]);
    const af_mask m = mask_of(a[5]);
    const float scale = static_cast<float>(number(a[6]));
    const af_blocks bl = blocks_of(a[7], x.sh.S);
    Out o(a[8], true, x.q.sizes(), dtype(a[10]), x.q);
    Out l(a[9], true, {x.sh.B, x.sh.Hq, x.sh.S}, at::kFloat, x.q);
    call(api.fwd_blocks, &x.sh, x.q.data_ptr(), x.k.data_ptr(), x.v.data_ptr(), &x.sq, &x.skv, &r, ptr(table), &m, x.group,
         scale, &bl, o.data(), out_code(o.t.scalar_type()), static_cast<float*>(l.data()), stream());
    return pair(o, l);
}

// 8-bit codes, contiguous; elements of another size are taken as that many codes each
at::Tensor codes(PyObject* o) {
    const at::Tensor& t = need(o);
    at::Tensor c = t.element_size() == 1 ? t : t.view(at::kByte);
    require(c.is_contiguous() && c.dim() == 4, "q8, k8, vt8: contiguous 4-D tensors of 8-bit codes");
    return c;
}

// fwd_fp8(q8, k8, vt8, mask, scale, scale_q, scale_k, scale_v, out_dtype)
PyObject* fwd_fp8(PyObject* const* a, Py_ssize_t n) {
    check_args(n, 9);
    const at::Tensor q = codes(a[0]), k = codes(a[1]), v = codes(a[2]);
    const int64_t B = q.size(0), Hq = q.size(1), S = q.size(2), D = q.size(3), Hkv = k.size(1);
    require(k.sizes() == at::IntArrayRef({B, Hkv, S, D}) && v.sizes() == at::IntArrayRef({B, Hkv, D, S}), "k8: [B, Hkv, S, D], vt8: [B, Hkv, D, S]");
    const af_mask m = mask_of(a[3]);
    const float scale = static_cast<float>(number(a[4])), s_q = static_cast<float>(number(a[5])), s_k = static_cast<float>(number(a[6])),
                s_v = static_cast<float>(number(a[7]));
    Out o(Py_None, true, q.sizes(), dtype(a[8]), q);
    Out l(Py_None, true, {B, Hq, S}, at::kFloat, q);
    const af_shape sh = {static_cast<int>(B), static_cast<int>(Hq), static_cast<int>(Hkv), static_cast<int>(S), static_cast<int>(D)};
    call(api.fwd_fp8, &sh, q.data_ptr(), k.data_ptr(), v.data_ptr(), &m, Hkv > 0 ? static_cast<int>(Hq / Hkv) : 0, scale, s_q,
         s_k, s_v, o.data(), out_code(o.t.scalar_type()), static_cast<float*>(l.data()), stream());
    return pair(o, l);
}

// bwd(q, k, v, o, lse, d_o, rope, table, mask, scale, dq_dtype, dkv_dtype, workspace, blocks)
PyObject* bwd(PyObject* const* a, Py_ssize_t n) {
    check_args(n, 14);
    Qkv x(a[0], a[1], a[2], false);
    const at::Tensor &o = need(a[3]), &lse = need(a[4]), &d_o = need(a[5]);
    require(o.is_contiguous() && d_o.is_contiguous() && lse.is_contiguous(), "o, d_o, lse: contiguous");
    require(o.scalar_type() == at::kBFloat16 && d_o.scalar_type() == at::kBFloat16 && lse.scalar_type() == at::kFloat, "o, d_o: bf16; lse: fp32");
    const af_rope r = rope_of(a[6]);
    const at::Tensor* table = tensor(a[7]);
    const af_mask m = mask_of(a[8]);
    const float scale = static_cast<float>(number(a[9]));
    const at::ScalarType tq = dtype(a[10]), tkv = dtype(a[11]);
    const at::Tensor* given = tensor(a[12]);
    const at::Tensor ws = given ? *given : empty({static_cast<int64_t>(api.bwd_onepass_workspace_bytes(&x.sh))}, at::kByte, x.q);
    Out dq(Py_None, true, x.q.sizes(), tq, x.q), dk(Py_None, true, x.k.sizes(), tkv, x.q), dv(Py_None, true, x.k.sizes(), tkv, x.q);
    if (a[13] != Py_None) {
        const af_blocks bl = blocks_of(a[13], x.sh.S);
        call(api.bwd_blocks, &x.sh, x.q.data_ptr(), x.k.data_ptr(), x.v.data_ptr(), o.data_ptr(),
             static_cast<const float*>(lse.data_ptr()), d_o.data_ptr(), &x.sq, &x.skv, &r, ptr(table), &m, x.group, scale, &bl,
             dq.data(), out_code(tq), dk.data(), dv.data(), out_code(tkv), ws.data_ptr(), ws.numel(), stream());
    } else {
        call(api.bwd, &x.sh, x.q.data_ptr(), x.k.data_ptr(), x.v.data_ptr(), o.data_ptr(),
             static_cast<const float*>(lse.data_ptr()), d_o.data_ptr(), &x.sq, &x.skv, &r, ptr(table), &m, x.group, scale,
             dq.data(), out_code(tq), dk.data(), dv.data(), out_code(tkv), ws.data_ptr(), ws.numel(), stream());
    }
    PyObject* g[3] = {dq.result(), dk.result(), dv.result()};
    PyObject* t = g[0] && g[1] && g[2] ? PyTuple_Pack(3, g[0], g[1], g[2]) : nullptr;
    for (PyObject* y : g) Py_XDECREF(y);
    if (!t) throw Raised();
    return t;
}

// decode(q, k, v, mask, scale, n_splits, out, lse, workspace, want_lse)
PyObject* decode(PyObject* const* a, Py_ssize_t n) {
    check_args(n, 10);
    const at::Tensor &q = need(a[0]), &k = need(a[1]), &v = need(a[2]);
    require(q.scalar_type() == at::kBFloat16 && k.scalar_type() == at::kBFloat16 && v.scalar_type() == at::kBFloat16, "q, k, v: bf16");
    require(q.dim() == 3 && q.is_contiguous() && k.dim() == 4, "q: [B, Hq, D], contiguous; k, v: [B, Hkv, N, D]");
    require(k.sizes() == v.sizes() && k.strides() == v.strides() && k.size(0) == q.size(0) && k.size(3) == q.size(2),
            "k and v: [B, Hkv, N, D] of q's B and D, with the same strides");
    const af_mask m = mask_of(a[3]);
    const float scale = static_cast<float>(number(a[4]));
    int n_splits = static_cast<int>(PyLong_AsLong(a[5]));
    if (n_splits == -1 && PyErr_Occurred()) throw Raised();
    const af_shape sh = {static_cast<int>(q.size(0)), static_cast<int>(q.size(1)), static_cast<int>(k.size(1)), static_cast<int>(k.size(2)),
                         static_cast<int>(q.size(2))};
    const af_strides skv = strides_of(k);
    Out o(a[6], true, q.sizes(), at::kBFloat16, q);
    Out l(a[7], truth(a[9]), {sh.B, sh.Hq}, at::kFloat, q);
    if (n_splits <= 0) n_splits = api.decode_splits(&sh);
    const at::Tensor* given = tensor(a[8]);
    at::Tensor ws;
    if (given) {
        ws = *given;
    } else {   // (a caller's own workspace must have been cleared once)
        ws = empty({static_cast<int64_t>(api.decode_workspace_bytes(&sh, n_splits))}, at::kByte, q);
        ws.zero_();
    }
    call(api.decode, &sh, q.data_ptr(), k.data_ptr(), v.data_ptr(), &skv, &m, sh.Hkv > 0 ? sh.Hq / sh.Hkv : 0, scale, o.data(),
         static_cast<float*>(l.data()), n_splits, ws.data_ptr(), ws.nbytes(), stream());
    return pair(o, l);
}

template <PyObject* (*F)(PyObject* const*, Py_ssize_t)>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    try {
        return F(args, n);
    } catch (const Raised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

// bind(addresses, error_class): addresses of the C entry points by name (a dict of ints)
PyObject* bind(PyObject*, PyObject* args) {
    PyObject *d, *cls;
    if (!PyArg_ParseTuple(args, "O!O", &PyDict_Type, &d, &cls)) return nullptr;
    bool ok = true;
    auto get = [&](const char* name, auto& slot) {
        PyObject* v = PyDict_GetItemString(d, name);
        void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
        if (!p) {
            ok = false;
            if (!PyErr_Occurred()) PyErr_Format(PyExc_KeyError, "%s", name);
            return;
        }
        slot = reinterpret_cast<std::remove_reference_t<decltype(slot)>>(p);
    };
    get("attnfuse_strerror", api.strerror_);
    get("attnfuse_fwd", api.fwd);
    get("attnfuse_fwd_scratch", api.fwd_scratch);
    get("attnfuse_fwd_scratch_bytes", api.fwd_scratch_bytes);
    get("attnfuse_fwd_hybrid", api.fwd_hybrid);
    get("attnfuse_fwd_hybrid_workspace_bytes", api.fwd_hybrid_workspace_bytes);
    get("attnfuse_fwd_blocks", api.fwd_blocks);
    get("attnfuse_fwd_fp8", api.fwd_fp8);
    get("attnfuse_bwd", api.bwd);
    get("attnfuse_bwd_blocks", api.bwd_blocks);
    get("attnfuse_bwd_onepass_workspace_bytes", api.bwd_onepass_workspace_bytes);
    get("attnfuse_decode", api.decode);
    get("attnfuse_decode_splits", api.decode_splits);
    get("attnfuse_decode_workspace_bytes", api.decode_workspace_bytes);
    if (!ok) return nullptr;
    Py_XSETREF(error_class, Py_NewRef(cls));
    Py_RETURN_NONE;
}

#define AF_FASTCALL(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<f>))
PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, nullptr},
    {"fwd", AF_FASTCALL(fwd), METH_FASTCALL, nullptr},
    {"fwd_hybrid", AF_FASTCALL(fwd_hybrid), METH_FASTCALL, nullptr},
    {"fwd_blocks", AF_FASTCALL(fwd_blocks), METH_FASTCALL, nullptr},
    {"fwd_fp8", AF_FASTCALL(fwd_fp8), METH_FASTCALL, nullptr},
    {"bwd", AF_FASTCALL(bwd), METH_FASTCALL, nullptr},
    {"decode", AF_FASTCALL(decode), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_torch_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__torch_binding(void) {
    auto intern = [](const char* s) { return PyUnicode_InternFromString(s); };
    names = {intern("theta"),   intern("rotary_dim"), intern("pos_offset"), intern("causal"),    intern("window"),   intern("alibi_slopes"),
             intern("nb"),      intern("row_ptr"),    intern("col_idx"),    intern("col_ptr"),   intern("row_idx"),  intern("row_order"),
             intern("col_order"), intern("pair_ptr"), intern("pair_idx"),   intern("pair_order"), intern("col_longest"),
             intern("listed")};
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "ABI_TAG", AF_ABI_TAG) < 0) Py_CLEAR(m);
    return m;
}
