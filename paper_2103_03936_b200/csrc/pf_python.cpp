// The Python side of the library: argument marshalling from torch tensors to the C ABI of include/pf.h,
// as one CPython extension module (_pf_native) linked against libpf.so.
//
// It exists because the calls it serves are short: a layer forward at a small batch runs a few
// microseconds on the GPU, and marshalling it through ctypes cost 15-20 us of host time per call
// (attribute look-ups on the tensors, one conversion per argument, torch.empty through the dispatcher).
// Here a call checks its tensors, takes its outputs and its workspace from torch's caching allocator
// and enters the C function without leaving native code.
//
// Every function takes the keyword arguments of its wrapper in binding.py by position.  `prepare` calls
// return (Prepared, outputs): an object that issues the C call with these arguments when it is called.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <functional>
#include <string>
#include <vector>

#include "pf.h"

namespace {

PyObject* g_pf_error = nullptr;      // binding.PfError, set once by binding.py

struct PyError {                     // becomes a Python exception of this type
    PyObject* type;
    std::string what;
};
[[noreturn]] void value_error(const std::string& s) { throw PyError{PyExc_ValueError, s}; }

const at::Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) throw PyError{PyExc_TypeError, std::string(name) + ": need a torch tensor"};
    return THPVariable_Unpack(o);
}
// An optional tensor argument: None gives an undefined tensor.
at::Tensor optional(PyObject* o, const char* name) {
    return o == Py_None ? at::Tensor() : at::Tensor(tensor(o, name));
}

int dtype_code(const at::Tensor& t) {
    if (t.scalar_type() == at::kBFloat16) return PF_BF16;
    if (t.scalar_type() == at::kFloat) return PF_F32;
    throw PyError{PyExc_TypeError, std::string("unsupported dtype ") + c10::toString(t.scalar_type())};
}
void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }

// Row pitch of a 2-D CUDA matrix with unit column stride (0 for an absent one).
int64_t pitch(const at::Tensor& t, const char* name) {
    if (!t.defined()) return 0;
    if (!t.is_cuda() || t.dim() != 2 || (t.size(1) > 1 && t.stride(1) != 1))
        value_error(std::string(name) + ": need a 2-D CUDA tensor with unit column stride");
    return t.size(0) > 1 ? t.stride(0) : std::max<int64_t>(t.stride(0), t.size(1));
}

at::Tensor empty(at::IntArrayRef shape, at::ScalarType type, const at::Tensor& like) {
    if (!like.is_cuda()) value_error("need CUDA tensors");
    return at::detail::empty_cuda(shape, type, like.device(), std::nullopt);
}

struct Stream {
    cudaStream_t s;
    bool current;        // the stream that torch's allocator orders its blocks by
};
Stream stream_of(PyObject* o) {
    const cudaStream_t cur = c10::cuda::getCurrentCUDAStream().stream();
    if (o == Py_None) return {cur, true};
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) throw python_error();
    void* p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw python_error();
    return {static_cast<cudaStream_t>(p), static_cast<cudaStream_t>(p) == cur};
}

// The caller's workspace, or a block of torch's caching allocator.  Such a block goes back to the
// allocator when the wrapper returns, while kernels that use it may still be queued: that is safe on
// torch's current stream (blocks are reused in stream order) and is made safe on any other stream by
// recording that stream on the block.
struct Workspace {
    at::Tensor given;
    c10::DataPtr own;
    void* p = nullptr;
    size_t bytes = 0;
};
Workspace workspace(PyObject* o, size_t need, const at::Tensor& like, const Stream& st) {
    Workspace w;
    if (o != Py_None) {
        w.given = tensor(o, "workspace");
        w.p = w.given.data_ptr();
        w.bytes = static_cast<size_t>(w.given.numel());
        return w;
    }
    w.bytes = std::max<size_t>(need, 256);
    const c10::Device cur(c10::kCUDA, c10::cuda::current_device());
    if (like.device() != cur) {              // tensors of another device: a block of that device
        w.given = empty({static_cast<int64_t>(w.bytes)}, at::kByte, like);
        w.p = w.given.data_ptr();
        if (!st.current)
            c10::cuda::CUDACachingAllocator::recordStream(w.given.storage().data_ptr(),
                                                          c10::cuda::getStreamFromExternal(st.s, like.device().index()));
        return w;
    }
    w.own = c10::cuda::CUDACachingAllocator::get()->allocate(w.bytes);
    w.p = w.own.get();
    if (!st.current) c10::cuda::CUDACachingAllocator::recordStream(w.own, c10::cuda::getStreamFromExternal(st.s, cur.index()));
    return w;
}

void check(int status, const char* where) {
    if (status == PF_OK) return;
    PyObject* e = PyObject_CallFunction(g_pf_error, "is", status, where);
    if (e) {
        PyErr_SetObject(g_pf_error, e);
        Py_DECREF(e);
    }
    throw python_error();
}

// ---------------------------------------------------------------------------- prepared calls
struct PreparedState {
    std::function<int()> call;
    const char* where;
    std::vector<at::Tensor> keep;
    Workspace ws;
};
struct Prepared {
    PyObject_HEAD
    PreparedState* st;
};
PyObject* prepared_call(PyObject* self, PyObject*, PyObject*) {
    HANDLE_TH_ERRORS
    PreparedState* st = reinterpret_cast<Prepared*>(self)->st;
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = st->call();
    Py_END_ALLOW_THREADS
    check(status, st->where);
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}
void prepared_free(PyObject* self) {
    PyTypeObject* type = Py_TYPE(self);
    delete reinterpret_cast<Prepared*>(self)->st;
    PyObject_Free(self);
    Py_DECREF(type);
}
PyType_Slot g_prepared_slots[] = {{Py_tp_call, reinterpret_cast<void*>(prepared_call)},
                                  {Py_tp_dealloc, reinterpret_cast<void*>(prepared_free)},
                                  {Py_tp_doc, const_cast<char*>("A C call with its arguments marshalled once; keeps its tensors alive.")},
                                  {0, nullptr}};
PyType_Spec g_prepared_spec = {"_pf_native.Prepared", sizeof(Prepared), 0, Py_TPFLAGS_DEFAULT | Py_TPFLAGS_DISALLOW_INSTANTIATION, g_prepared_slots};
PyTypeObject* g_prepared_type = nullptr;

// Issues the call now (returns `out`), or wraps it (returns (Prepared, out)); steals `out`.
template <typename F>
PyObject* issue(bool prepare, F&& f, const char* where, Workspace&& ws, std::vector<at::Tensor> keep, PyObject* out) {
    if (!out) throw python_error();
    if (!prepare) {
        int st;
        Py_BEGIN_ALLOW_THREADS
        st = f();
        Py_END_ALLOW_THREADS
        if (st != PF_OK) {
            Py_DECREF(out);
            check(st, where);
        }
        return out;
    }
    Prepared* p = PyObject_New(Prepared, g_prepared_type);
    if (!p) {
        Py_DECREF(out);
        throw python_error();
    }
    p->st = new PreparedState{std::function<int()>(std::forward<F>(f)), where, std::move(keep), std::move(ws)};
    return Py_BuildValue("(NN)", reinterpret_cast<PyObject*>(p), out);
}

PyObject* wrap(const at::Tensor& t) {
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}
PyObject* tuple(std::initializer_list<at::Tensor> ts) {
    PyObject* out = PyTuple_New(static_cast<Py_ssize_t>(ts.size()));
    if (!out) return nullptr;
    Py_ssize_t i = 0;
    for (const at::Tensor& t : ts) PyTuple_SET_ITEM(out, i++, wrap(t));
    return out;
}
bool truth(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw python_error();
    return v == 1;
}
int64_t integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
}

template <PyObject* (*body)(PyObject* const*)>
PyObject* entry_impl(PyObject* const* a) {
    HANDLE_TH_ERRORS
    try {
        return body(a);
    } catch (const PyError& e) {
        PyErr_SetString(e.type, e.what.c_str());
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}
template <PyObject* (*body)(PyObject* const*), int kArgs>
PyObject* entry(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != kArgs) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", kArgs, n);
        return nullptr;
    }
    return entry_impl<body>(a);
}

void rows_cols(const at::Tensor& t, const char* name, int64_t* rows, int64_t* cols) {
    if (t.dim() != 2) value_error(std::string(name) + ": need a 2-D CUDA tensor with unit column stride");
    *rows = t.size(0);
    *cols = t.size(1);
}

// ---------------------------------------------------------------------------- linear
// 0 x, 1 U, 2 V, 3 bias, 4 act, 5 y, 6 T_stash, 7 want_stash, 8 workspace, 9 stream, 10 prepare, 11 with_act
PyObject* linear_fwd(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const int dt = dtype_code(x);
    int64_t m, k, n, r;
    rows_cols(x, "x", &m, &k);
    rows_cols(V, "V", &n, &r);
    if (U.dim() != 2 || U.size(0) != k || U.size(1) != r) value_error("U must be [k, r] and V [n, r]");
    const at::Tensor bias = optional(a[3], "bias");
    if (bias.defined() && (bias.dim() != 1 || bias.size(0) != n || bias.scalar_type() != x.scalar_type() || !bias.is_contiguous()))
        value_error("bias must be a contiguous [n] tensor of x's dtype");
    const int act = static_cast<int>(integer(a[4]));
    at::Tensor y = optional(a[5], "y"), T = optional(a[6], "T_stash");
    if (!y.defined()) y = empty({m, n}, x.scalar_type(), x);
    if (!T.defined() && truth(a[7])) T = empty({m, r}, x.scalar_type(), x);
    const Stream st = stream_of(a[9]);
    Workspace ws = workspace(a[8], a[8] == Py_None ? pf_lowrank_linear_workspace(m, k, n, r, dt, 0) : 0, x, st);
    auto f = [=, px = ptr(x), pu = ptr(U), pv = ptr(V), pb = ptr(bias), py = ptr(y), pt = ptr(T), ldx = pitch(x, "x"),
              ldu = pitch(U, "U"), ldv = pitch(V, "V"), ldy = pitch(y, "y"), ldt = pitch(T, "T_stash"), wp = ws.p, wb = ws.bytes, s = st.s] {
        return pf_lowrank_linear_fwd_act(px, ldx, pu, ldu, pv, ldv, pb, act, py, ldy, pt, ldt, m, k, n, r, dt, wp, wb, s);
    };
    const bool prepare = truth(a[10]);
    std::vector<at::Tensor> keep;
    if (prepare) keep = {x, U, V, bias, y, T};
    return issue(prepare, f, truth(a[11]) ? "pf_lowrank_linear_fwd_act" : "pf_lowrank_linear_fwd", std::move(ws), std::move(keep),
                 T.defined() ? tuple({y, T}) : wrap(y));
}

// 0 x, 1 U, 2 V, 3 y, 4 T_stash, 5 stream
PyObject* linear_fwd_static(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const at::Tensor& y = tensor(a[3], "y");
    const at::Tensor T = optional(a[4], "T_stash");
    const int dt = dtype_code(x);
    int64_t m, k, n, r;
    rows_cols(x, "x", &m, &k);
    rows_cols(V, "V", &n, &r);
    if (U.dim() != 2 || U.size(0) != k || U.size(1) != r) value_error("U must be [k, r] and V [n, r]");
    const Stream st = stream_of(a[5]);
    const int64_t ldx = pitch(x, "x"), ldu = pitch(U, "U"), ldv = pitch(V, "V"), ldy = pitch(y, "y"), ldt = pitch(T, "T_stash");
    auto f = [=, px = ptr(x), pu = ptr(U), pv = ptr(V), py = ptr(y), pt = ptr(T), s = st.s] {
        return pf_lowrank_linear_fwd_static(px, ldx, pu, ldu, pv, ldv, py, ldy, pt, ldt, m, k, n, r, dt, s);
    };
    return issue(false, f, "pf_lowrank_linear_fwd_static", Workspace(), {}, T.defined() ? tuple({y, T}) : wrap(y));
}

unsigned grad_flags(PyObject* accumulate, PyObject* f32) {
    return (truth(accumulate) ? PF_GRAD_ACCUMULATE : 0u) | (truth(f32) ? PF_GRAD_F32 : 0u);
}

// 0 x, 1 U, 2 V, 3 dY, 4 T_stash, 5 need_dX, 6 dX, 7 dU, 8 dV, 9 accumulate, 10 grads_f32, 11 workspace, 12 stream, 13 prepare
PyObject* linear_bwd(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const at::Tensor& dY = tensor(a[3], "dY");
    const at::Tensor T = optional(a[4], "T_stash");
    const int dt = dtype_code(x);
    int64_t m, k, n, r;
    rows_cols(x, "x", &m, &k);
    rows_cols(V, "V", &n, &r);
    const unsigned flags = grad_flags(a[9], a[10]);
    const at::ScalarType gdt = (flags & PF_GRAD_F32) ? at::kFloat : x.scalar_type();
    at::Tensor dX = optional(a[6], "dX"), dU = optional(a[7], "dU"), dV = optional(a[8], "dV");
    if ((flags & PF_GRAD_ACCUMULATE) && (!dU.defined() || !dV.defined())) value_error("accumulate=True needs the dU and dV to add to");
    if (!dX.defined() && truth(a[5])) dX = empty({m, k}, x.scalar_type(), x);
    if (!dU.defined()) dU = empty({k, r}, gdt, x);
    if (!dV.defined()) dV = empty({n, r}, gdt, x);
    if (dU.scalar_type() != gdt || dV.scalar_type() != gdt)
        value_error("dU and dV must be float32 with grads_f32=True and of x's dtype otherwise");
    const Stream st = stream_of(a[12]);
    Workspace ws = workspace(a[11], a[11] == Py_None ? pf_lowrank_linear_workspace(m, k, n, r, dt, 1) : 0, x, st);
    auto f = [=, px = ptr(x), pu = ptr(U), pv = ptr(V), pdy = ptr(dY), pt = ptr(T), pdx = ptr(dX), pdu = ptr(dU), pdv = ptr(dV),
              ldx = pitch(x, "x"), ldu = pitch(U, "U"), ldv = pitch(V, "V"), lddy = pitch(dY, "dY"), ldt = pitch(T, "T_stash"),
              lddx = pitch(dX, "dX"), lddu = pitch(dU, "dU"), lddv = pitch(dV, "dV"), wp = ws.p, wb = ws.bytes, s = st.s] {
        return pf_lowrank_linear_bwd_ex(px, ldx, pu, ldu, pv, ldv, pdy, lddy, pt, ldt, pdx, lddx, pdu, lddu, pdv, lddv, m, k, n, r, dt,
                                        flags, wp, wb, s);
    };
    const bool prepare = truth(a[13]);
    std::vector<at::Tensor> keep;
    if (prepare) keep = {x, U, V, dY, T, dX, dU, dV};
    return issue(prepare, f, flags ? "pf_lowrank_linear_bwd_ex" : "pf_lowrank_linear_bwd", std::move(ws), std::move(keep),
                 tuple({dX, dU, dV}));
}

// 0 y, 1 dY, 2 act, 3 want_dbias, 4 dbias, 5 workspace, 6 stream
PyObject* bias_act_bwd(PyObject* const* a) {
    const at::Tensor y = optional(a[0], "y");
    const at::Tensor& dY = tensor(a[1], "dY");
    const int dt = dtype_code(dY);
    const int act = static_cast<int>(integer(a[2]));
    int64_t m, n;
    rows_cols(dY, "dY", &m, &n);
    at::Tensor db = optional(a[4], "dbias");
    if (!db.defined() && truth(a[3])) db = empty({n}, dY.scalar_type(), dY);
    const Stream st = stream_of(a[6]);
    Workspace ws = workspace(a[5], db.defined() && a[5] == Py_None ? pf_bias_act_bwd_workspace(m, n) : 0, dY, st);
    auto f = [=, py = ptr(y), pdy = ptr(dY), pdb = ptr(db), ldy = pitch(y, "y"), lddy = pitch(dY, "dY"), wp = ws.p, wb = ws.bytes, s = st.s] {
        return pf_bias_act_bwd(py, ldy, pdy, lddy, pdb, m, n, act, dt, wp, wb, s);
    };
    return issue(false, f, "pf_bias_act_bwd", std::move(ws), {}, wrap(db));
}

// ---------------------------------------------------------------------------- grouped linear
struct Group {
    void* p;
    int64_t ld, gs;
};
// (pointer, row pitch, group stride) of a [groups, rows, cols] tensor (unit column stride), or of a 2-D
// [rows, cols] tensor shared by all groups (stride 0) where that is allowed.
Group group(const at::Tensor& t, const char* name, int64_t groups, bool may_share = false) {
    if (!t.defined()) return {nullptr, 0, 0};
    if (t.dim() == 2 && may_share) return {t.data_ptr(), pitch(t, name), 0};
    if (!t.is_cuda() || t.dim() != 3 || t.size(0) != groups || (t.size(2) > 1 && t.stride(2) != 1))
        value_error(std::string(name) + ": need a CUDA tensor [groups, rows, cols] with unit column stride");
    return {t.data_ptr(), t.size(1) > 1 ? t.stride(1) : std::max<int64_t>(t.stride(1), t.size(2)), t.stride(0)};
}

// 0 x, 1 U, 2 V, 3 y, 4 T_stash, 5 want_stash, 6 workspace, 7 stream, 8 prepare
PyObject* grouped_fwd(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const int dt = dtype_code(U);
    if (U.dim() != 3 || V.dim() != 3 || x.dim() < 2) value_error("U must be [G, k, r], V [G, n, r], x [G, m, k] or [m, k]");
    const int64_t G = U.size(0), k = U.size(1), r = U.size(2), n = V.size(1), m = x.size(-2);
    if (V.size(0) != G || V.size(2) != r || x.size(-1) != k) value_error("U must be [G, k, r], V [G, n, r], x [G, m, k] or [m, k]");
    at::Tensor y = optional(a[3], "y"), T = optional(a[4], "T_stash");
    if (!y.defined()) y = empty({G, m, n}, U.scalar_type(), U);
    if (!T.defined() && truth(a[5])) T = empty({G, m, r}, U.scalar_type(), U);
    const Stream st = stream_of(a[7]);
    const int g = static_cast<int>(G);
    Workspace ws = workspace(a[6], a[6] == Py_None ? pf_lowrank_linear_grouped_workspace(g, m, k, n, r, dt, 0) : 0, U, st);
    auto f = [=, gx = group(x, "x", G, true), gu = group(U, "U", G), gv = group(V, "V", G), gy = group(y, "y", G), gt = group(T, "T_stash", G),
              wp = ws.p, wb = ws.bytes, s = st.s] {
        return pf_lowrank_linear_grouped_fwd(g, gx.p, gx.ld, gx.gs, gu.p, gu.ld, gu.gs, gv.p, gv.ld, gv.gs, gy.p, gy.ld, gy.gs, gt.p, gt.ld,
                                             gt.gs, m, k, n, r, dt, wp, wb, s);
    };
    const bool prepare = truth(a[8]);
    std::vector<at::Tensor> keep;
    if (prepare) keep = {x, U, V, y, T};
    return issue(prepare, f, "pf_lowrank_linear_grouped_fwd", std::move(ws), std::move(keep), T.defined() ? tuple({y, T}) : wrap(y));
}

// 0 x, 1 U, 2 V, 3 dY, 4 T_stash, 5 need_dX, 6 dX, 7 dU, 8 dV, 9 workspace, 10 stream, 11 prepare
PyObject* grouped_bwd(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const at::Tensor& dY = tensor(a[3], "dY");
    const at::Tensor T = optional(a[4], "T_stash");
    const int dt = dtype_code(U);
    if (U.dim() != 3 || V.dim() != 3 || x.dim() < 2) value_error("U must be [G, k, r], V [G, n, r], x [G, m, k] or [m, k]");
    const int64_t G = U.size(0), k = U.size(1), r = U.size(2), n = V.size(1), m = x.size(-2);
    at::Tensor dX = optional(a[6], "dX"), dU = optional(a[7], "dU"), dV = optional(a[8], "dV");
    if (!dX.defined() && truth(a[5])) dX = x.dim() == 2 ? empty({m, k}, U.scalar_type(), U) : empty({G, m, k}, U.scalar_type(), U);
    if (!dU.defined()) dU = empty({G, k, r}, U.scalar_type(), U);
    if (!dV.defined()) dV = empty({G, n, r}, U.scalar_type(), U);
    const Stream st = stream_of(a[10]);
    const int g = static_cast<int>(G);
    Workspace ws = workspace(a[9], a[9] == Py_None ? pf_lowrank_linear_grouped_workspace(g, m, k, n, r, dt, 1) : 0, U, st);
    auto f = [=, gx = group(x, "x", G, true), gu = group(U, "U", G), gv = group(V, "V", G), gdy = group(dY, "dY", G), gt = group(T, "T_stash", G),
              gdx = group(dX, "dX", G, true), gdu = group(dU, "dU", G), gdv = group(dV, "dV", G), wp = ws.p, wb = ws.bytes, s = st.s] {
        return pf_lowrank_linear_grouped_bwd(g, gx.p, gx.ld, gx.gs, gu.p, gu.ld, gu.gs, gv.p, gv.ld, gv.gs, gdy.p, gdy.ld, gdy.gs, gt.p, gt.ld,
                                             gt.gs, gdx.p, gdx.ld, gdx.gs, gdu.p, gdu.ld, gdu.gs, gdv.p, gdv.ld, gdv.gs, m, k, n, r, dt, wp,
                                             wb, s);
    };
    const bool prepare = truth(a[11]);
    std::vector<at::Tensor> keep;
    if (prepare) keep = {x, U, V, dY, T, dX, dU, dV};
    return issue(prepare, f, "pf_lowrank_linear_grouped_bwd", std::move(ws), std::move(keep), tuple({dX, dU, dV}));
}

// ---------------------------------------------------------------------------- convolution
struct Conv {
    int N, H, W, C, R, O, kh, kw, Ho, Wo, stride, pad;
};
Conv conv_dims(const at::Tensor& x, const at::Tensor& U, const at::Tensor& V, PyObject* stride, PyObject* pad) {
    const struct { const at::Tensor* t; const char* name; int dims; } all[3] = {{&x, "x", 4}, {&U, "U", 4}, {&V, "V", 2}};
    for (const auto& e : all) {
        if (!e.t->is_cuda() || !e.t->is_contiguous()) value_error(std::string(e.name) + ": need a contiguous CUDA tensor");
        if (e.t->dim() != e.dims) value_error("x must be [N, H, W, C], U [kh, kw, C, R] and V [O, R]");
    }
    Conv c;
    c.N = static_cast<int>(x.size(0)); c.H = static_cast<int>(x.size(1)); c.W = static_cast<int>(x.size(2)); c.C = static_cast<int>(x.size(3));
    c.kh = static_cast<int>(U.size(0)); c.kw = static_cast<int>(U.size(1)); c.R = static_cast<int>(U.size(3));
    c.O = static_cast<int>(V.size(0));
    if (U.size(2) != c.C || V.size(1) != c.R) value_error("U must be [kh, kw, C, R] and V [O, R]");
    c.stride = static_cast<int>(integer(stride)); c.pad = static_cast<int>(integer(pad));
    if (c.stride == 0) throw PyError{PyExc_ZeroDivisionError, "integer division or modulo by zero"};
    auto out = [&](int size, int k) {        // floor division
        const int num = size + 2 * c.pad - k;
        int q = num / c.stride;
        if (num % c.stride != 0 && ((num < 0) != (c.stride < 0))) --q;
        return q + 1;
    };
    c.Ho = out(c.H, c.kh); c.Wo = out(c.W, c.kw);
    return c;
}
size_t conv_workspace(const Conv& c, int dt, int bwd) {
    return pf_lowrank_conv_workspace(c.N, c.H, c.W, c.C, c.R, c.O, c.kh, c.kw, c.stride, c.pad, dt, bwd);
}

// 0 x, 1 U, 2 V, 3 stride, 4 pad, 5 y, 6 T_stash, 7 want_stash, 8 workspace, 9 stream, 10 prepare
PyObject* conv_fwd(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const int dt = dtype_code(x);
    const Conv c = conv_dims(x, U, V, a[3], a[4]);
    at::Tensor y = optional(a[5], "y"), T = optional(a[6], "T_stash");
    if (!y.defined()) y = empty({c.N, c.Ho, c.Wo, c.O}, x.scalar_type(), x);
    if (!T.defined() && truth(a[7])) T = empty({c.N, c.Ho, c.Wo, c.R}, x.scalar_type(), x);
    const Stream st = stream_of(a[9]);
    Workspace ws = workspace(a[8], a[8] == Py_None ? conv_workspace(c, dt, 0) : 0, x, st);
    auto f = [=, px = ptr(x), pu = ptr(U), pv = ptr(V), py = ptr(y), pt = ptr(T), wp = ws.p, wb = ws.bytes, s = st.s] {
        return pf_lowrank_conv_fwd(px, pu, pv, py, pt, c.N, c.H, c.W, c.C, c.R, c.O, c.kh, c.kw, c.stride, c.pad, dt, wp, wb, s);
    };
    const bool prepare = truth(a[10]);
    std::vector<at::Tensor> keep;
    if (prepare) keep = {x, U, V, y, T};
    return issue(prepare, f, "pf_lowrank_conv_fwd", std::move(ws), std::move(keep), T.defined() ? tuple({y, T}) : wrap(y));
}

// 0 x, 1 U, 2 V, 3 dY, 4 stride, 5 pad, 6 T_stash, 7 need_dX, 8 dX, 9 dU, 10 dV, 11 accumulate, 12 grads_f32, 13 workspace,
// 14 stream, 15 prepare
PyObject* conv_bwd(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0], "x");
    const at::Tensor& U = tensor(a[1], "U");
    const at::Tensor& V = tensor(a[2], "V");
    const at::Tensor& dY = tensor(a[3], "dY");
    const int dt = dtype_code(x);
    const Conv c = conv_dims(x, U, V, a[4], a[5]);
    if (!dY.is_contiguous() || dY.dim() != 4 || dY.size(0) != c.N || dY.size(1) != c.Ho || dY.size(2) != c.Wo || dY.size(3) != c.O)
        value_error("dY must be contiguous [N, Ho, Wo, O]");
    const at::Tensor T = optional(a[6], "T_stash");
    at::Tensor dX = optional(a[8], "dX"), dU = optional(a[9], "dU"), dV = optional(a[10], "dV");
    if (!dX.defined() && truth(a[7])) dX = empty(x.sizes(), x.scalar_type(), x);
    const unsigned flags = grad_flags(a[11], a[12]);
    const at::ScalarType gdt = (flags & PF_GRAD_F32) ? at::kFloat : x.scalar_type();
    if ((flags & PF_GRAD_ACCUMULATE) && (!dU.defined() || !dV.defined())) value_error("accumulate=True needs the dU and dV to add to");
    if (!dU.defined()) dU = empty(U.sizes(), gdt, x);
    if (!dV.defined()) dV = empty(V.sizes(), gdt, x);
    if (dU.scalar_type() != gdt || dV.scalar_type() != gdt || !dU.is_contiguous() || !dV.is_contiguous())
        value_error("dU and dV must be contiguous, float32 with grads_f32=True and of x's dtype otherwise");
    const Stream st = stream_of(a[14]);
    Workspace ws = workspace(a[13], a[13] == Py_None ? conv_workspace(c, dt, 1) : 0, x, st);
    auto f = [=, px = ptr(x), pu = ptr(U), pv = ptr(V), pdy = ptr(dY), pt = ptr(T), pdx = ptr(dX), pdu = ptr(dU), pdv = ptr(dV), wp = ws.p,
              wb = ws.bytes, s = st.s] {
        return pf_lowrank_conv_bwd_ex(px, pu, pv, pdy, pt, pdx, pdu, pdv, c.N, c.H, c.W, c.C, c.R, c.O, c.kh, c.kw, c.stride, c.pad, dt, flags,
                                      wp, wb, s);
    };
    const bool prepare = truth(a[15]);
    std::vector<at::Tensor> keep;
    if (prepare) keep = {x, U, V, dY, T, dX, dU, dV};
    return issue(prepare, f, flags ? "pf_lowrank_conv_bwd_ex" : "pf_lowrank_conv_bwd", std::move(ws), std::move(keep), tuple({dX, dU, dV}));
}

// ---------------------------------------------------------------------------- flat gradient buffer
struct TensorList {
    std::vector<void*> ptrs;
    std::vector<int64_t> numels, offsets;     // offsets: prefix sums of numels, one more entry
    std::vector<at::Tensor> keep;
    at::Tensor first;
};
// The tensors of a list; `like` (or else the first one) sets the dtype that all of them must have.
TensorList tensor_list(PyObject* seq, const at::Tensor& like, const char* whose, bool keep) {
    TensorList l;
    PyObject* fast = PySequence_Fast(seq, "grads: need a sequence of tensors");
    if (!fast) throw python_error();
    struct Drop { PyObject* o; ~Drop() { Py_DECREF(o); } } drop{fast};
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
    l.ptrs.resize(n); l.numels.resize(n); l.offsets.resize(n + 1);
    at::ScalarType type = at::kFloat;
    for (Py_ssize_t i = 0; i < n; ++i) {
        const at::Tensor& t = tensor(PySequence_Fast_GET_ITEM(fast, i), "grads");
        if (i == 0) {
            l.first = t;
            const at::Tensor& ref = like.defined() ? like : t;
            dtype_code(ref);
            type = ref.scalar_type();
        }
        if (!t.is_cuda() || !t.is_contiguous() || t.scalar_type() != type)
            value_error(std::string("grads: contiguous CUDA tensors of ") + whose + " dtype");
        l.ptrs[i] = t.data_ptr();
        l.numels[i] = t.numel();
        l.offsets[i + 1] = l.offsets[i] + l.numels[i];
        if (keep) l.keep.push_back(t);
    }
    return l;
}
PyObject* offset_list(const std::vector<int64_t>& offs) {
    PyObject* out = PyList_New(static_cast<Py_ssize_t>(offs.size()));
    for (size_t i = 0; out && i < offs.size(); ++i) PyList_SET_ITEM(out, static_cast<Py_ssize_t>(i), PyLong_FromLongLong(offs[i]));
    return out;
}

// 0 grads (not empty), 1 flat, 2 stream, 3 prepare
PyObject* pack(PyObject* const* a) {
    at::Tensor flat = optional(a[1], "flat");
    const bool prepare = truth(a[3]);
    TensorList l = tensor_list(a[0], at::Tensor(), "one", prepare);
    const int dt = dtype_code(l.first), count = static_cast<int>(l.ptrs.size());
    if (!flat.defined()) flat = empty({l.offsets[count]}, l.first.scalar_type(), l.first);
    const Stream st = stream_of(a[2]);
    PyObject* out = Py_BuildValue("(NN)", wrap(flat), offset_list(l.offsets));
    std::vector<at::Tensor> keep = std::move(l.keep);
    if (prepare) keep.push_back(flat);
    l.first = at::Tensor();
    auto f = [l = std::move(l), dt, p = ptr(flat), n = flat.numel(), s = st.s, count]() mutable {
        return pf_pack_factor_grads(l.ptrs.data(), l.numels.data(), count, dt, p, n, l.offsets.data(), nullptr, 0, s);
    };
    return issue(prepare, std::move(f), "pf_pack_factor_grads", Workspace(), std::move(keep), out);
}

// 0 flat, 1 grads (not empty), 2 stream
PyObject* unpack(PyObject* const* a) {
    const at::Tensor& flat = tensor(a[0], "flat");
    TensorList l = tensor_list(a[1], flat, "flat's", false);
    const int dt = dtype_code(flat);
    const Stream st = stream_of(a[2]);
    void* p = ptr(flat);
    const int64_t n = flat.numel();
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = pf_unpack_factor_grads(p, n, l.ptrs.data(), l.numels.data(), static_cast<int>(l.ptrs.size()), dt, l.offsets.data(), nullptr, 0, st.s);
    Py_END_ALLOW_THREADS
    check(status, "pf_unpack_factor_grads");
    return offset_list(l.offsets);
}

PyObject* set_error(PyObject*, PyObject* cls) {
    Py_INCREF(cls);
    Py_XSETREF(g_pf_error, cls);
    Py_RETURN_NONE;
}

#define PF_ENTRY(name, args) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<name, args>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {PF_ENTRY(linear_fwd, 12), PF_ENTRY(linear_fwd_static, 6), PF_ENTRY(linear_bwd, 14), PF_ENTRY(bias_act_bwd, 7),
                           PF_ENTRY(grouped_fwd, 9), PF_ENTRY(grouped_bwd, 12), PF_ENTRY(conv_fwd, 11), PF_ENTRY(conv_bwd, 16),
                           PF_ENTRY(pack, 4), PF_ENTRY(unpack, 3), {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_pf_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pf_native(void) {
    g_prepared_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&g_prepared_spec));
    if (!g_prepared_type) return nullptr;
    return PyModule_Create(&g_module);
}
