// The hot part of the Python binding as a CPython extension: argument checks, output and workspace allocation, the call
// into libbased.so and the autograd node.  The functions take their arguments by position, in the order of the Python
// functions of binding.py that forward to them (which hold the signatures and defaults); an optional tensor is None.
// Errors are the ones the Python checks raise: ValueError, TypeError, and binding.BasedError for a status of the library.
#include <Python.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/device_lazy_init.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>

#include <algorithm>
#include <stdexcept>
#include <string>

#include "based.h"

namespace {
using at::Tensor;

struct TypeFault : std::runtime_error { using std::runtime_error::runtime_error; };
struct StatusFault : std::runtime_error {
    based_status status;
    StatusFault(based_status s, const char* where) : std::runtime_error(where), status(s) {}
};
[[noreturn]] void value_error(const std::string& what) { throw std::invalid_argument(what); }

// ---------------------------------------------------------------------------------------------- arguments
const Tensor kNone;

const Tensor& tensor(PyObject* o) {
    if (o == Py_None) return kNone;
    if (!THPVariable_Check(o)) throw TypeFault(std::string("expected a tensor, got ") + Py_TYPE(o)->tp_name);
    return THPVariable_Unpack(o);
}
// a CUDA tensor, contiguous; or an undefined one for None
const Tensor& dev(PyObject* o) {
    const Tensor& t = tensor(o);
    if (!t.defined()) return t;
    if (!t.is_cuda()) value_error("libbased takes CUDA tensors only (there is no CPU path)");
    if (!t.is_contiguous()) value_error("tensors must be contiguous");
    return t;
}
const Tensor& need(PyObject* o, const char* name) {
    const Tensor& t = dev(o);
    if (!t.defined()) throw TypeFault(std::string(name) + " is required");
    return t;
}
int integer(PyObject* o) {
    const long x = PyLong_AsLong(o);
    if (x == -1 && PyErr_Occurred()) {
        PyErr_Clear();
        throw TypeFault("expected an integer");
    }
    return static_cast<int>(x);
}
float number(PyObject* o) {
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) {
        PyErr_Clear();
        throw TypeFault("expected a number");
    }
    return static_cast<float>(x);
}
// None: the current stream; else the handle of a stream as an integer
void* stream_of(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) {
        PyErr_Clear();
        throw TypeFault("expected a stream handle");
    }
    return p;
}
based_dtype dtype_code(const Tensor& t) {
    if (t.scalar_type() == at::kFloat) return BASED_F32;
    if (t.scalar_type() == at::kBFloat16) return BASED_BF16;
    throw TypeFault(std::string("unsupported io dtype ") + c10::toString(t.scalar_type()));
}
const void* cptr(const Tensor& t) { return t.defined() ? t.const_data_ptr() : nullptr; }
void* ptr(const Tensor& t) { return t.defined() ? t.mutable_data_ptr() : nullptr; }
float* fptr(const Tensor& t) { return static_cast<float*>(ptr(t)); }
int size(const Tensor& t, int i) { return static_cast<int>(t.size(i)); }
void dims(const Tensor& t, int n, const char* name) {
    if (t.dim() != n) value_error(std::string(name) + " must have " + std::to_string(n) + " dimensions");
}
std::string text(at::IntArrayRef s) {
    std::string r = "(";
    for (size_t i = 0; i < s.size(); ++i) r += (i ? ", " : "") + std::to_string(s[i]);
    return r + ")";
}
bool shape_is(const Tensor& t, at::IntArrayRef s) { return t.sizes() == s; }
// the same number of elements of the same type: enough where the kernels take a contiguous array and the caller may hold it
// in another shape (a step's k as [B,H,1,d], its output as [B,1,C])
bool fills(const Tensor& t, const Tensor& like) { return t.numel() == like.numel() && t.scalar_type() == like.scalar_type(); }

// ---------------------------------------------------------------------------------------------- checks
void check_qkv(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& out) {
    if (k.sizes() != q.sizes() || v.dim() != q.dim() ||
        v.sizes().slice(0, v.dim() - 1) != q.sizes().slice(0, q.dim() - 1) || k.scalar_type() != q.scalar_type() ||
        v.scalar_type() != q.scalar_type())
        value_error("q, k, v shapes/dtypes disagree");
    if (out.defined() && (out.sizes() != v.sizes() || out.scalar_type() != v.scalar_type()))
        value_error("out must have the shape and dtype of v");
}
void check_state(const Tensor& kv, const Tensor& z, int B, int H, int d_feat, int d_v, int flags, bool required) {
    if (!kv.defined() && !z.defined()) {
        if (required) value_error("kv_state and z_state are required");
        return;
    }
    if (!kv.defined() || !z.defined()) value_error("kv_state and z_state come together");
    if (kv.scalar_type() != at::kFloat || z.scalar_type() != at::kFloat) throw TypeFault("state tensors are fp32");
    const int rows = (flags & BASED_STATE_SYM) ? BASED_D_SYM : 1 + d_feat + d_feat * d_feat;
    if (!shape_is(kv, {B, H, rows, d_v}) || !shape_is(z, {B, H, rows})) {
        const std::string b = std::to_string(B), h = std::to_string(H), r = std::to_string(rows);
        value_error("state shapes must be kv [" + b + "," + h + "," + r + "," + std::to_string(d_v) + "] and z [" + b + "," + h +
                    "," + r + "] for these flags, got " + text(kv.sizes()) + " and " + text(z.sizes()));
    }
}
void check_caches(const Tensor& kc, const Tensor& vc, const Tensor& q, const char* what) {
    if (kc.dim() != 4 || !shape_is(kc, {q.size(0), q.size(1), kc.size(2), q.size(2)}) || vc.sizes() != kc.sizes() ||
        kc.scalar_type() != q.scalar_type() || vc.scalar_type() != q.scalar_type())
        value_error(std::string("cache shapes/dtypes disagree with ") + what);
}
void check(based_status st, const char* where) {
    if (st != BASED_OK) throw StatusFault(st, where);
}
// a tensor like t, which is contiguous (at::empty_like takes 0.85 us, 0.1 of it to look at the strides)
Tensor fresh(const Tensor& t) { return at::empty(t.sizes(), t.options()); }
// a workspace of at least `need` bytes: the caller's, or a fresh one that lives as long as this object (memory of torch's
// allocator, as a tensor would hold it but without the tensor: 0.3 us for 0.7).  It belongs to the call's own stream, which may
// be another than the current one: only what follows on that stream is given it again.
struct Workspace {
    c10::DataPtr own;
    void* data = nullptr;
    size_t bytes = 0;
    Workspace(const Tensor& given, size_t need, const Tensor& like, void* stream) {
        if (need == 0 || (given.defined() && given.nbytes() >= need)) {
            if (!given.defined()) return;
            data = given.mutable_data_ptr();
            bytes = given.nbytes();
            return;
        }
        const c10::cuda::CUDAGuard on(like.device());
        c10::cuda::OptionalCUDAStreamGuard of;
        if (stream != c10::cuda::getCurrentCUDAStream().stream())
            of.reset_stream(c10::cuda::getStreamFromExternal(static_cast<cudaStream_t>(stream), like.get_device()));
        own = c10::cuda::CUDACachingAllocator::get()->allocate(need);
        data = own.get();
        bytes = need;
    }
};
// the same for scratch that a call can do without: nothing where the device has no room for it
Workspace optional_workspace(size_t bytes, const Tensor& like, void* stream) {
    try {
        return Workspace(kNone, bytes, like, stream);
    } catch (const c10::OutOfMemoryError&) {
        return Workspace(kNone, 0, like, stream);
    }
}
// the library's calls run without the interpreter lock: a launch can wait for room in the stream's queue
template <typename F> based_status unlocked(F f) {
    based_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return st;
}

// ---------------------------------------------------------------------------------------------- calls
Tensor prefill_call(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& kv, const Tensor& z, Tensor out, int flags,
                    const Tensor& workspace, void* stream) {
    const int B = size(q, 0), H = size(q, 1), L = size(q, 2), d_feat = size(q, 3), d_v = size(v, 3);
    const based_dtype io = dtype_code(q);
    if (!out.defined()) out = fresh(v);
    size_t need = based_prefill_workspace_bytes(B, H, L, d_feat, d_v, io);
    if (need <= BASED_WORDS_BYTES && !(flags & BASED_STATE_CONTINUE)) need = 0;
    const Workspace ws(workspace, need, q, stream);
    check(based_prefill(cptr(q), cptr(k), cptr(v), ptr(out), fptr(kv), fptr(z), B, H, L, d_feat, d_v, io, flags, ws.data, ws.bytes,
                        stream),
          "based_prefill");
    return out;
}
struct Gradients { Tensor dq, dk, dv; };
Gradients backward_call(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& dout, const Tensor& out, int flags,
                        const Tensor& workspace, void* stream) {
    const int B = size(q, 0), H = size(q, 1), L = size(q, 2), d_feat = size(q, 3), d_v = size(v, 3);
    const based_dtype io = dtype_code(q);
    const size_t need = based_prefill_backward_workspace_bytes(B, H, L, d_v, io);
    // (a caller's workspace of that size is used as it is)
    const size_t parts = io == BASED_F32 && !workspace.defined() ? based_f32_parts_bytes(B, H, L, d_feat, d_v, 1) : 0;
    Workspace ws = optional_workspace(parts, q, stream);
    if (ws.bytes < need) ws = Workspace(workspace, need, q, stream);
    Gradients g{fresh(q), fresh(k), fresh(v)};
    const based_status st =
        out.defined() ? based_prefill_backward_with_out(cptr(q), cptr(k), cptr(v), cptr(out), cptr(dout), ptr(g.dq), ptr(g.dk),
                                                        ptr(g.dv), B, H, L, d_feat, d_v, io, flags, ws.data, ws.bytes, stream)
                      : based_prefill_backward(cptr(q), cptr(k), cptr(v), cptr(dout), ptr(g.dq), ptr(g.dk), ptr(g.dv), B, H, L,
                                               d_feat, d_v, io, flags, ws.data, ws.bytes, stream);
    check(st, "based_prefill_backward");
    return g;
}

PyObject* wrap(const Tensor& t) { return THPVariable_Wrap(t); }
PyObject* wrap(std::initializer_list<Tensor> ts) {
    PyObject* r = PyTuple_New(static_cast<Py_ssize_t>(ts.size()));
    Py_ssize_t i = 0;
    for (const Tensor& t : ts) PyTuple_SET_ITEM(r, i++, wrap(t));
    return r;
}

// q, k, v, out, kv_state, z_state, flags, workspace, stream
PyObject* prefill(PyObject* const* a) {
    const Tensor &q = need(a[0], "q"), &k = need(a[1], "k"), &v = need(a[2], "v"), &out = dev(a[3]), &kv = dev(a[4]), &z = dev(a[5]),
                 &ws = dev(a[7]);
    const int flags = integer(a[6]);
    dims(q, 4, "q");
    check_qkv(q, k, v, out);
    check_state(kv, z, size(q, 0), size(q, 1), size(q, 3), size(v, 3), flags, (flags & BASED_STATE_CONTINUE) != 0);
    void* stream = stream_of(a[8]);
    Tensor r;
    std::exception_ptr fault;
    Py_BEGIN_ALLOW_THREADS
    try {
        r = prefill_call(q, k, v, kv, z, out, flags, ws, stream);
    } catch (...) {
        fault = std::current_exception();
    }
    Py_END_ALLOW_THREADS
    if (fault) std::rethrow_exception(fault);
    return wrap(r);
}

// q, k, v, dout, flags, workspace, stream, out
PyObject* prefill_backward(PyObject* const* a) {
    const Tensor &q = need(a[0], "q"), &k = need(a[1], "k"), &v = need(a[2], "v"), &dout = need(a[3], "dout"), &ws = dev(a[5]),
                 &out = dev(a[7]);
    dims(q, 4, "q");
    check_qkv(q, k, v, out);
    if (dout.sizes() != v.sizes() || dout.scalar_type() != v.scalar_type())
        value_error("dout must have the shape and dtype of v");
    const int flags = integer(a[4]);
    void* stream = stream_of(a[6]);
    Gradients g;
    std::exception_ptr fault;
    Py_BEGIN_ALLOW_THREADS
    try {
        g = backward_call(q, k, v, dout, out, flags, ws, stream);
    } catch (...) {
        fault = std::current_exception();
    }
    Py_END_ALLOW_THREADS
    if (fault) std::rethrow_exception(fault);
    return wrap({g.dq, g.dk, g.dv});
}

// q, k, v, kv_state, z_state, flags, out, stream, name of the entry point (for the error message)
PyObject* decode_step(PyObject* const* a) {
    const Tensor &q = need(a[0], "q"), &k = need(a[1], "k"), &v = need(a[2], "v"), &kv = dev(a[3]), &z = dev(a[4]);
    Tensor out = dev(a[6]);
    dims(q, 3, "q");
    check_qkv(q, k, v, out);
    const int B = size(q, 0), H = size(q, 1), d_feat = size(q, 2), d_v = size(v, 2), flags = integer(a[5]);
    check_state(kv, z, B, H, d_feat, d_v, flags, true);
    const based_dtype io = dtype_code(q);
    void* stream = stream_of(a[7]);
    if (!out.defined()) out = fresh(v);
    const based_status st = unlocked([&] {
        return based_decode_step_flags(cptr(q), cptr(k), cptr(v), fptr(kv), fptr(z), ptr(out), B, H, d_feat, d_v, io, flags, stream);
    });
    check(st, PyUnicode_AsUTF8(a[8]));
    return wrap(out);
}

// q, k, v, out, window, softmax_scale, stream
PyObject* swa(PyObject* const* a) {
    const Tensor &q = need(a[0], "q"), &k = need(a[1], "k"), &v = need(a[2], "v");
    Tensor out = dev(a[3]);
    dims(q, 4, "q");
    check_qkv(q, k, v, out);
    if (v.sizes() != q.sizes()) value_error("the sliding-window mixer takes q, k, v of one shape");
    const int window = integer(a[4]);
    const float scale = number(a[5]);
    const based_dtype io = dtype_code(q);
    void* stream = stream_of(a[6]);
    if (!out.defined()) out = fresh(v);
    const based_status st = unlocked([&] {
        return swa_forward(cptr(q), cptr(k), cptr(v), ptr(out), size(q, 0), size(q, 1), size(q, 2), size(q, 3), window, scale, io, stream);
    });
    check(st, "swa_forward");
    return wrap(out);
}

// q, k, v, k_cache, v_cache, pos (an integer, or an int32 tensor with one entry per sequence), out, softmax_scale, stream
PyObject* swa_decode(PyObject* const* a) {
    const Tensor &q = need(a[0], "q"), &k = need(a[1], "k"), &v = need(a[2], "v"), &kc = need(a[3], "k_cache"), &vc = need(a[4], "v_cache");
    const bool ragged = THPVariable_Check(a[5]);
    const Tensor& positions = ragged ? dev(a[5]) : kNone;
    Tensor out = dev(a[6]);
    dims(q, 3, "q");
    if (ragged) {
        check_qkv(q, k, v, out);
        if (v.sizes() != q.sizes()) value_error("the sliding-window mixer takes q, k, v of one shape");
    } else {
        if (!fills(k, q) || !fills(v, q)) value_error("q, k, v shapes/dtypes disagree");
        if (out.defined() && !fills(out, v)) value_error("out must have the shape and dtype of v");
    }
    check_caches(kc, vc, q, "q");
    const int B = size(q, 0), H = size(q, 1), d = size(q, 2), window = size(kc, 2);
    if (ragged && (positions.scalar_type() != at::kInt || !shape_is(positions, {B})))
        value_error("pos is an int32 tensor with one entry per sequence");
    const int pos = ragged ? 0 : integer(a[5]);
    const float scale = number(a[7]);
    const based_dtype io = dtype_code(q);
    void* stream = stream_of(a[8]);
    if (!out.defined()) out = fresh(v);
    const based_status st = unlocked([&] {
        return ragged ? swa_decode_step_ragged(cptr(q), cptr(k), cptr(v), ptr(kc), ptr(vc), ptr(out), B, H, d, window,
                                               static_cast<const int*>(cptr(positions)), scale, io, stream)
                      : swa_decode_step(cptr(q), cptr(k), cptr(v), ptr(kc), ptr(vc), ptr(out), B, H, d, window, pos, scale, io, stream);
    });
    check(st, ragged ? "swa_decode_step_ragged" : "swa_decode_step");
    return wrap(out);
}

// q, k, v, kv_state, z_state, qw, kw, vw, k_cache, v_cache, pos_state, out, out_w, flags, softmax_scale, stream
PyObject* generation_step(PyObject* const* a) {
    const Tensor &q = need(a[0], "q"), &k = need(a[1], "k"), &v = need(a[2], "v"), &kv = dev(a[3]), &z = dev(a[4]),
                 &qw = need(a[5], "qw"), &kw = need(a[6], "kw"), &vw = need(a[7], "vw"), &kc = need(a[8], "k_cache"),
                 &vc = need(a[9], "v_cache"), &pos = need(a[10], "pos_state");
    Tensor out = dev(a[11]), out_w = dev(a[12]);
    dims(q, 3, "q");
    dims(qw, 3, "qw");
    check_qkv(q, k, v, out);
    const int B = size(q, 0), H = size(q, 1), d_feat = size(q, 2), d_v = size(v, 2), flags = integer(a[13]);
    check_state(kv, z, B, H, d_feat, d_v, flags, true);
    const int Hw = size(qw, 1), d_w = size(qw, 2);
    const auto dt = q.scalar_type();
    if (size(qw, 0) != B || kw.sizes() != qw.sizes() || vw.sizes() != qw.sizes() || qw.scalar_type() != dt ||
        kw.scalar_type() != dt || vw.scalar_type() != dt)
        value_error("qw, kw, vw must be [B,H_w,d_w] in the io dtype");
    check_caches(kc, vc, qw, "qw");
    if (pos.scalar_type() != at::kInt || pos.numel() != 2) value_error("pos_state is an int32 tensor {position, ticket}");
    if (out_w.defined() && (out_w.sizes() != vw.sizes() || out_w.scalar_type() != dt))
        value_error("out_w must have the shape and dtype of vw");
    const float scale = number(a[14]);
    const based_dtype io = dtype_code(q);
    void* stream = stream_of(a[15]);
    if (!out.defined()) out = fresh(v);
    if (!out_w.defined()) out_w = fresh(vw);
    const int window = size(kc, 2);
    const based_status st = unlocked([&] {
        return based_generation_step(cptr(q), cptr(k), cptr(v), fptr(kv), fptr(z), ptr(out), cptr(qw), cptr(kw), cptr(vw), ptr(kc),
                                     ptr(vc), ptr(out_w), B, H, d_feat, d_v, Hw, d_w, window, static_cast<int*>(ptr(pos)), scale, io,
                                     flags, stream);
    });
    check(st, "based_generation_step");
    return wrap({out, out_w});
}

struct GenerationGraph {
    based_generation_graph* graph;
    Tensor in[6];                              // q, k, v, qw, kw, vw: the buffers of the last token's inputs
    Tensor written[7];                         // state, caches, position and outputs
    c10::Device device() const { return in[0].device(); }
    // the steps belong on the current stream of the graph's own device, whichever device is current
    void* stream() const { return c10::cuda::getCurrentCUDAStream(in[0].get_device()).stream(); }
};
bool overlap(const Tensor& a, const Tensor& b) {
    const char *x = static_cast<const char*>(a.const_data_ptr()), *y = static_cast<const char*>(b.const_data_ptr());
    return x < y + b.nbytes() && y < x + a.nbytes();
}
constexpr const char* kGraphName = "based_generation_graph";
void free_graph(PyObject* capsule) {
    GenerationGraph* g = static_cast<GenerationGraph*>(PyCapsule_GetPointer(capsule, kGraphName));
    if (!g) return;
    {
        c10::cuda::OptionalCUDAGuard on;
        try {
            on.set_device(g->device());
        } catch (...) {                        // (at the interpreter's end the device may be gone)
        }
        based_generation_graph_destroy(g->graph);
    }
    delete g;
}
GenerationGraph& graph_of(PyObject* o) {
    GenerationGraph* g = static_cast<GenerationGraph*>(PyCapsule_GetPointer(o, kGraphName));
    if (!g) {
        PyErr_Clear();
        throw TypeFault("expected a generation graph");
    }
    return *g;
}
// q, k, v, kv_state, z_state, qw, kw, vw, k_cache, v_cache, pos_state, out, out_w, flags, softmax_scale (all tensors live as
// long as the graph: the caller sees to it)
PyObject* generation_graph(PyObject* const* a) {
    Tensor t[13];
    for (int i = 0; i < 13; ++i) t[i] = need(a[i], "every tensor of a generation graph");
    const Tensor &q = t[0], &v = t[2], &kv = t[3], &z = t[4], &qw = t[5], &kc = t[8];
    check_qkv(q, t[1], v, t[11]);
    const int B = size(q, 0), H = size(q, 1), d_feat = size(q, 2), d_v = size(v, 2), flags = integer(a[13]);
    check_state(kv, z, B, H, d_feat, d_v, flags, true);
    check_caches(kc, t[9], qw, "qw");
    const float scale = number(a[14]);
    const based_dtype io = dtype_code(q);
    based_generation_graph* made = nullptr;
    const based_status st = unlocked([&] {
        return based_generation_graph_create(ptr(q), ptr(t[1]), ptr(v), fptr(kv), fptr(z), ptr(t[11]), ptr(qw), ptr(t[6]), ptr(t[7]),
                                             ptr(kc), ptr(t[9]), ptr(t[12]), B, H, d_feat, d_v, size(qw, 1), size(qw, 2),
                                             size(kc, 2), static_cast<int*>(ptr(t[10])), scale, io, flags, &made);
    });
    check(st, "based_generation_graph_create");
    return PyCapsule_New(new GenerationGraph{made, {q, t[1], v, qw, t[6], t[7]}, {kv, z, kc, t[9], t[10], t[11], t[12]}},
                         kGraphName, free_graph);
}
// graph, q, k, v, qw, kw, vw -> whether the step was launched on these inputs; False: they have to be copied into the
// buffers first (another dtype, shape or layout, or they overlap the buffers or something that the step writes, such as the
// outputs of the step before)
PyObject* generation_graph_step(PyObject* const* a) {
    GenerationGraph& g = graph_of(a[0]);
    const void* p[6];
    for (int i = 0; i < 6; ++i) {
        const Tensor &t = tensor(a[1 + i]), &own = g.in[i];
        if (!t.defined() || t.scalar_type() != own.scalar_type() || t.sizes() != own.sizes() || t.device() != own.device() ||
            !t.is_contiguous() || (reinterpret_cast<uintptr_t>(t.const_data_ptr()) & 15))
            Py_RETURN_FALSE;
        p[i] = t.const_data_ptr();
        for (const Tensor& b : g.in)
            if (overlap(t, b)) Py_RETURN_FALSE;
        for (const Tensor& b : g.written)
            if (overlap(t, b)) Py_RETURN_FALSE;
    }
    const c10::cuda::CUDAGuard on(g.device());
    void* stream = g.stream();
    const based_status st = unlocked([&] { return based_generation_graph_step(g.graph, p[0], p[1], p[2], p[3], p[4], p[5], stream); });
    check(st, "based_generation_graph_step");
    Py_RETURN_TRUE;
}
// graph: the step on what the buffers hold
PyObject* generation_graph_replay(PyObject* const* a) {
    GenerationGraph& g = graph_of(a[0]);
    const c10::cuda::CUDAGuard on(g.device());
    void* stream = g.stream();
    const based_status st = unlocked([&] {
        return based_generation_graph_step(g.graph, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, stream);
    });
    check(st, "based_generation_graph_step");
    Py_RETURN_NONE;
}

// a, g, h, b2, conv_state, out, step (bool), stream
PyObject* baseconv(PyObject* const* p) {
    const Tensor &a = need(p[0], "a"), &g = need(p[1], "g"), &h = need(p[2], "h"), &b2 = need(p[3], "b2"), &state = dev(p[4]);
    Tensor out = dev(p[5]);
    const bool step = p[6] == Py_True;
    dims(a, step ? 2 : 3, "a");
    if (h.dim() < 1) value_error("h must be [width, C]");
    const int B = size(a, 0), N = step ? 1 : size(a, 1), C = static_cast<int>(a.size(-1)), width = size(h, 0);
    if (!(step ? fills(g, a) : g.sizes() == a.sizes() && g.scalar_type() == a.scalar_type()) || h.scalar_type() != at::kFloat ||
        b2.scalar_type() != at::kFloat)
        value_error("a, g disagree or the filter/bias are not fp32");
    if (h.numel() != static_cast<int64_t>(width) * C || (step ? b2.numel() != C : h.dim() < 2 || h.size(1) != C || !shape_is(b2, {C})))
        value_error("filter/bias shapes disagree with C");
    if (out.defined() && !fills(out, a)) value_error("out must have the shape and dtype of a");
    if (state.defined() && (!shape_is(state, {B, width - 1, C}) || state.scalar_type() != a.scalar_type()))
        value_error("conv_state must be [B, width-1, C] in the io dtype");
    const based_dtype io = dtype_code(a);
    void* stream = stream_of(p[7]);
    if (!out.defined()) out = fresh(a);
    auto filter = static_cast<const float*>(cptr(h)), bias = static_cast<const float*>(cptr(b2));
    const based_status st = unlocked([&] {
        return step ? baseconv_gate_step(cptr(a), cptr(g), filter, bias, ptr(state), ptr(out), B, C, width, io, stream)
                    : baseconv_gate_forward(cptr(a), cptr(g), filter, bias, ptr(out), B, N, C, width, io, stream);
    });
    check(st, step ? "baseconv_gate_step" : "baseconv_gate_forward");
    return wrap(out);
}

// Python's exception for a status of the library
void set_status_error(const StatusFault& e) {
    PyObject* mod = PyImport_ImportModule("paper_2402_18668_b200.binding");
    PyObject* cls = mod ? PyObject_GetAttrString(mod, "BasedError") : nullptr;
    PyObject* err = cls ? PyObject_CallFunction(cls, "is", static_cast<int>(e.status), e.what()) : nullptr;
    if (err) PyErr_SetObject(cls, err);
    Py_XDECREF(err);
    Py_XDECREF(cls);
    Py_XDECREF(mod);
}

// ---------------------------------------------------------------------------------------------- autograd
// An output gradient usually comes back from a projection with the heads of a token side by side, [B,L,H,d_v] seen as
// [B,H,L,d_v].
bool tokens_first(const Tensor& g, at::ScalarType dt) {
    if (g.is_contiguous() || g.dim() != 4 || !g.is_cuda() || g.scalar_type() != dt) return false;
    const int64_t B = g.size(0), H = g.size(1), L = g.size(2), d = g.size(3);
    return g.stride(3) == 1 && g.stride(1) == d && g.stride(2) == H * d && (B == 1 || g.stride(0) == L * H * d);
}
// bf16 gradients of such an output gradient as it lies (the copy ahead was 6.5 us and a launch of a step of B4 H16 L2048 d_v64: 158.8
// -> 150.0 us); undefined tensors where there is no such route
Gradients backward_bf16_as_it_lies(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& dout, const Tensor& out, int flags,
                                   void* stream) {
    const int B = size(q, 0), H = size(q, 1), L = size(q, 2), d_feat = size(q, 3), d_v = size(v, 3);
    if (dout.sizes() != v.sizes() || (reinterpret_cast<uintptr_t>(dout.const_data_ptr()) & 15) ||
        (static_cast<int64_t>(L) * H * d_v * 2 >> 39) != 0 || static_cast<int64_t>(B) * H > 65532 || static_cast<int64_t>(B) * H * L > 0x7fffffff)
        return {};
    const Workspace ws(kNone, based_prefill_backward_workspace_bytes(B, H, L, d_v, BASED_BF16), q, stream);
    Gradients g{fresh(q), fresh(k), fresh(v)};
    check(based_prefill_backward_tokens_first_with_out(cptr(q), cptr(k), cptr(v), cptr(out), dout.const_data_ptr(), ptr(g.dq), ptr(g.dk),
                                                       ptr(g.dv), B, H, L, d_feat, d_v, BASED_BF16, flags, ws.data, ws.bytes, stream),
          "based_prefill_backward");
    return g;
}
// fp32 gradients of such an output gradient as it lies; undefined tensors where there is no such route
Gradients backward_as_it_lies(const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& dout, int flags, void* stream) {
    const int B = size(q, 0), H = size(q, 1), L = size(q, 2), d_feat = size(q, 3), d_v = size(v, 3);
    if (dout.sizes() != v.sizes() || (reinterpret_cast<uintptr_t>(dout.const_data_ptr()) & 15)) return {};
    const size_t parts = based_f32_parts_bytes(B, H, L, d_feat, d_v, 1);
    // On multiply-adds every tile of dout is read several times, in rows: with many tokens the copy ahead is the faster (32768 of
    // d_v 112 473 us for 475, 8192 of d_v 128 124 for 123)
    if (parts == 0 && static_cast<int64_t>(B) * H * L > 16384) return {};
    const size_t bytes = std::max(based_prefill_backward_workspace_bytes(B, H, L, d_v, BASED_F32), parts);
    const Workspace ws = optional_workspace(bytes, q, stream);
    if (!ws.data) return {};
    Gradients g{fresh(q), fresh(k), fresh(v)};
    const based_status st = based_prefill_backward_tokens_first(cptr(q), cptr(k), cptr(v), dout.const_data_ptr(), ptr(g.dq), ptr(g.dk),
                                                                ptr(g.dv), B, H, L, d_feat, d_v, BASED_F32, flags, ws.data, ws.bytes,
                                                                stream);
    if (st == BASED_ERR_UNSUPPORTED) return {};
    check(st, "based_prefill_backward");
    return g;
}
// The output gradient as the backward pass takes it: the library has a copy kernel for that layout.
Tensor heads_first(const Tensor& g, at::ScalarType dt, void* stream) {
    if (!tokens_first(g, dt)) return g.contiguous().to(dt);
    const int64_t B = g.size(0), H = g.size(1), L = g.size(2), d = g.size(3);
    const Tensor out = at::empty({B, H, L, d}, g.options());
    const based_status st = based_tokens_to_heads(g.const_data_ptr(), ptr(out), static_cast<int>(B), static_cast<int>(H),
                                                  static_cast<int>(L), static_cast<int>(d * g.element_size()), stream);
    return st == BASED_OK ? out : g.contiguous();
}
// the fp32 forward pass on the tensor cores; an undefined tensor where there is no such route
Tensor forward_by_parts(const Tensor& q, const Tensor& k, const Tensor& v, int flags, void* stream) {
    const int B = size(q, 0), H = size(q, 1), L = size(q, 2), d_feat = size(q, 3), d_v = size(v, 3);
    const size_t bytes = based_f32_parts_bytes(B, H, L, d_feat, d_v, 0);
    if (bytes == 0 || (flags & ~BASED_NUMERATOR_ONLY)) return {};
    const Workspace ws = optional_workspace(bytes, q, stream);
    if (!ws.data) return {};
    Tensor out = fresh(v);
    auto in = [](const Tensor& t) { return static_cast<const float*>(t.const_data_ptr()); };
    const based_status st = based_prefill_f32_parts(in(q), in(k), in(v), static_cast<float*>(ptr(out)), B, H, L, d_feat, d_v, flags,
                                                    ws.data, ws.bytes, stream);
    if (st == BASED_ERR_UNSUPPORTED) return {};
    check(st, "based_prefill");
    return out;
}
struct LinearAttention : torch::autograd::Function<LinearAttention> {
    static Tensor forward(torch::autograd::AutogradContext* ctx, const Tensor& q_, const Tensor& k_, const Tensor& v_, int64_t flags) {
        const Tensor q = q_.contiguous(), k = k_.contiguous(), v = v_.contiguous();
        if (!q.is_cuda() || !k.is_cuda() || !v.is_cuda()) value_error("libbased takes CUDA tensors only (there is no CPU path)");
        dims(q, 4, "q");
        check_qkv(q, k, v, kNone);
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        Tensor out = q.scalar_type() == at::kFloat ? forward_by_parts(q, k, v, static_cast<int>(flags), stream) : Tensor();
        if (!out.defined()) out = prefill_call(q, k, v, kNone, kNone, Tensor(), static_cast<int>(flags), kNone, stream);
        ctx->save_for_backward({q, k, v, out});
        ctx->saved_data["flags"] = flags;
        return out;
    }
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext* ctx, torch::autograd::variable_list grads) {
        const auto saved = ctx->get_saved_variables();
        const Tensor &q = saved[0], &k = saved[1], &v = saved[2], &out = saved[3];
        void* stream = c10::cuda::getCurrentCUDAStream().stream();
        const int flags = static_cast<int>(ctx->saved_data["flags"].toInt());
        try {
            Gradients g;
            if (grads[0].defined() && tokens_first(grads[0], q.scalar_type()))
                g = q.scalar_type() == at::kFloat ? backward_as_it_lies(q, k, v, grads[0], flags, stream)
                                                  : backward_bf16_as_it_lies(q, k, v, grads[0], out, flags, stream);
            if (!g.dq.defined()) {
                const Tensor dout = grads[0].defined() ? heads_first(grads[0], q.scalar_type(), stream) : at::zeros_like(v);
                g = backward_call(q, k, v, dout, out, flags, kNone, stream);
            }
            return {g.dq, g.dk, g.dv, Tensor()};
        } catch (const StatusFault& e) {
            // autograd's worker thread: the engine hands a Python exception on to the thread that called backward
            pybind11::gil_scoped_acquire lock;
            set_status_error(e);
            python_error err;
            err.persist();
            throw err;
        }
    }
};

// q, k, v, flags
PyObject* linear_attention(PyObject* const* a) {
    const Tensor q = tensor(a[0]), k = tensor(a[1]), v = tensor(a[2]);
    if (!q.defined() || !k.defined() || !v.defined()) throw TypeFault("q, k and v are required");
    const int64_t flags = integer(a[3]);
    Tensor r;
    std::exception_ptr fault;
    Py_BEGIN_ALLOW_THREADS
    try {
        r = LinearAttention::apply(q, k, v, flags);
    } catch (...) {
        fault = std::current_exception();
    }
    Py_END_ALLOW_THREADS
    if (fault) std::rethrow_exception(fault);
    return wrap(r);
}

// ---------------------------------------------------------------------------------------------- module
// Everything but the faults of this file is torch's to translate: its own error types, and Python exceptions that passed
// through C++ (python_error, from a saved-tensor hook for instance), which go on as they are.
PyObject* translated(std::exception_ptr fault) {
    HANDLE_TH_ERRORS
    std::rethrow_exception(fault);
    END_HANDLE_TH_ERRORS
}
template <PyObject* (*F)(PyObject* const*), int N>
PyObject* guarded(PyObject*, PyObject* const* args, Py_ssize_t n) {
    try {
        if (n != N) throw TypeFault("wrong number of arguments");
        return F(args);
    } catch (const StatusFault& e) {
        set_status_error(e);
    } catch (const TypeFault& e) {
        PyErr_SetString(PyExc_TypeError, e.what());
    } catch (const std::invalid_argument& e) {
        PyErr_SetString(PyExc_ValueError, e.what());
    } catch (...) {
        return translated(std::current_exception());
    }
    return nullptr;
}
template <PyObject* (*F)(PyObject* const*), int N> PyMethodDef method(const char* name) {
    return {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&guarded<F, N>)), METH_FASTCALL, nullptr};
}
PyMethodDef methods[] = {method<prefill, 9>("prefill"), method<prefill_backward, 8>("prefill_backward"),
                         method<decode_step, 9>("decode_step"), method<swa, 7>("swa"), method<swa_decode, 9>("swa_decode"),
                         method<generation_step, 16>("generation_step"), method<baseconv, 8>("baseconv"),
                         method<generation_graph, 15>("generation_graph"), method<generation_graph_step, 7>("generation_graph_step"),
                         method<generation_graph_replay, 1>("generation_graph_replay"),
                         method<linear_attention, 4>("linear_attention"), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};
}  // namespace

PyMODINIT_FUNC PyInit__native(void) { return PyModule_Create(&module); }
