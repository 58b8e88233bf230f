// Host path of the Python entry points: argument checks, output allocation and the C-ABI call in one native step.
//
// A decode step of a few sequences takes the GPU about 4 us, so what its caller waits for is the host.  Marshalling eight
// tensors through ctypes (attribute look-ups, shape tuples, pointer objects) took 13 of the 16.5 us of such a step; here it
// is about 1 us, and what is left is the allocation of the output and the kernel launch.
// The checks and the messages are those that binding.py documents; every number is computed by libqdelta.so.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/qdelta.h"

namespace {

PyObject* g_error = nullptr;                       // binding.QdeltaError

struct Raised {};                                  // a Python exception is set

[[noreturn]] void fail(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    PyErr_FormatV(g_error ? g_error : PyExc_RuntimeError, fmt, ap);
    va_end(ap);
    throw Raised{};
}
void check(int rc, const char* what) {
    if (rc != QD_OK) fail("%s failed: %s (%d)", what, qdelta_status_string(rc), rc);
}

// nullptr for None
const at::Tensor* tensor(PyObject* o, const char* name) {
    if (o == Py_None || o == nullptr) return nullptr;
    if (!THPVariable_Check(o)) { PyErr_Format(PyExc_TypeError, "%s must be a tensor, got %s", name, Py_TYPE(o)->tp_name); throw Raised{}; }
    return &THPVariable_Unpack(o);
}
const at::Tensor& needed(PyObject* o, const char* name) {
    const at::Tensor* t = tensor(o, name);
    if (!t) { PyErr_Format(PyExc_TypeError, "%s must be a tensor, got NoneType", name); throw Raised{}; }
    return *t;
}
void want_dims(const at::Tensor& t, int n) {
    if (t.dim() == n) return;
    if (t.dim() > n) PyErr_Format(PyExc_ValueError, "too many values to unpack (expected %d)", n);
    else PyErr_Format(PyExc_ValueError, "not enough values to unpack (expected %d, got %d)", n, (int)t.dim());
    throw Raised{};
}
int dtype_code(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return QD_F32;
    if (t.scalar_type() == at::kBFloat16) return QD_BF16;
    fail("unsupported dtype torch.%s", torch::getTHPDtype(t.scalar_type())->name);
}
std::string text(c10::IntArrayRef s) {
    std::string r = "(";
    for (size_t i = 0; i < s.size(); ++i) r += (i ? ", " : "") + std::to_string(s[i]);
    return r + (s.size() == 1 ? ",)" : ")");
}
// what a kernel that is given this tensor's address would trip over; empty if nothing
std::string complaint(const at::Tensor& t, at::ScalarType dt, c10::IntArrayRef shape, const char* name, bool any_dtype = false) {
    if (!t.is_cuda() || !t.is_contiguous()) return name + std::string(" must be a contiguous CUDA tensor");
    if (!any_dtype && t.scalar_type() != dt)
        return name + std::string(" must have dtype torch.") + torch::getTHPDtype(dt)->name + ", got torch." + torch::getTHPDtype(t.scalar_type())->name;
    if (t.sizes() != shape) return name + std::string(" must have shape ") + text(shape) + ", got " + text(t.sizes());
    return {};
}
// device pointer of a contiguous CUDA tensor of the given type and shape; nullptr for an absent one
void* ptr(const at::Tensor* t, at::ScalarType dt, c10::IntArrayRef shape, const char* name, bool any_dtype = false) {
    if (!t) return nullptr;
    const std::string c = complaint(*t, dt, shape, name, any_dtype);
    if (!c.empty()) fail("%s", c.c_str());
    return t->data_ptr();
}
at::Tensor empty(c10::IntArrayRef shape, at::ScalarType dt, c10::Device dev) {
    if (!dev.is_cuda()) fail("the inputs must be contiguous CUDA tensors");
    return at::Tensor(at::detail::empty_cuda(shape, dt, dev, std::nullopt));
}
qd_stream stream() { return reinterpret_cast<qd_stream>(c10::cuda::getCurrentCUDAStream().stream()); }

struct NoGil {                                     // other threads may run while kernels are enqueued
    PyThreadState* s = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(s); }
};

// What torch throws keeps its Python type: torch.OutOfMemoryError of an allocation, IndexError, TypeError, or the exception that
// a saved-tensor hook raised (non-reentrant checkpointing ends its recomputation with one).
template <class F> PyObject* guarded(F f) {
    try {
        return f();
    } catch (const Raised&) {
    } catch (...) {
        torch::translate_exception_to_python(std::current_exception());
    }
    return nullptr;
}
bool arity(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}
PyObject* own(PyObject* o) { Py_INCREF(o); return o; }

// recurrent_step(q, k, v, beta, alpha, lam, state, o)
PyObject* recurrent_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!arity(n, 8)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor &q = needed(a[0], "q"), &v = needed(a[2], "v");
        want_dims(q, 3);
        const int64_t B = q.size(0), H = q.size(1), dk = q.size(2), dv = v.size(-1);
        const at::ScalarType dt = q.scalar_type();
        const int code = dtype_code(q);
        const void* qp = ptr(&q, dt, {B, H, dk}, "q");
        const void* kp = ptr(tensor(a[1], "k"), dt, {B, H, dk}, "k");
        const void* vp = ptr(&v, dt, {B, H, dv}, "v");
        const void* bp = ptr(tensor(a[3], "beta"), dt, {B, H}, "beta");
        const void* ap = ptr(tensor(a[4], "alpha"), dt, {B, H}, "alpha");
        const void* lp = ptr(tensor(a[5], "lam"), dt, {B, H}, "lam");
        float* sp = static_cast<float*>(ptr(tensor(a[6], "state"), at::kFloat, {B, H, dk, dv}, "state"));
        at::Tensor made;
        const at::Tensor* o = tensor(a[7], "o");
        if (!o) { made = empty({B, H, dv}, dt, q.device()); o = &made; }
        void* op = ptr(o, dt, {B, H, dv}, "o");
        int rc;
        {
            NoGil ng;
            rc = qdelta_recurrent_step((int)B, (int)H, (int)dk, (int)dv, code, qp, kp, vp, bp, ap, lp, sp, op, stream());
        }
        check(rc, "qdelta_recurrent_step");
        return made.defined() ? THPVariable_Wrap(std::move(made)) : own(a[7]);
    });
}

// recurrent_steps(q, k, v, beta, alpha, lam, state, o, flags)
PyObject* recurrent_steps(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!arity(n, 9)) return nullptr;
    return guarded([&]() -> PyObject* {
        const at::Tensor &q = needed(a[0], "q"), &v = needed(a[2], "v"), &state = needed(a[6], "state");
        want_dims(q, 4);
        const int64_t B = q.size(0), S = q.size(1), H = q.size(2), dk = q.size(3), dv = v.size(-1);
        const at::ScalarType dt = q.scalar_type();
        unsigned flags = (unsigned)PyLong_AsUnsignedLong(a[8]);
        if (state.scalar_type() == at::kBFloat16) flags |= QD_STATE_BF16;
        else if (state.scalar_type() != at::kFloat) fail("state must be fp32, or bf16 for the reduced-precision state option");
        const int code = dtype_code(q);
        const void* qp = ptr(&q, dt, {B, S, H, dk}, "q");
        const void* kp = ptr(tensor(a[1], "k"), dt, {B, S, H, dk}, "k");
        const void* vp = ptr(&v, dt, {B, S, H, dv}, "v");
        const void* bp = ptr(tensor(a[3], "beta"), dt, {B, S, H}, "beta");
        const void* ap = ptr(tensor(a[4], "alpha"), dt, {B, S, H}, "alpha");
        const void* lp = ptr(tensor(a[5], "lam"), dt, {B, S, H}, "lam");
        void* sp = ptr(&state, at::kFloat, {B, H, dk, dv}, "state", true);
        at::Tensor made;
        const at::Tensor* o = tensor(a[7], "o");
        if (!o) { made = empty({B, S, H, dv}, dt, q.device()); o = &made; }
        void* op = ptr(o, dt, {B, S, H, dv}, "o");
        int rc;
        {
            NoGil ng;
            rc = qdelta_recurrent_steps((int)B, (int)S, (int)H, (int)dk, (int)dv, code, qp, kp, vp, bp, ap, lp, sp, op, flags, stream());
        }
        check(rc, "qdelta_recurrent_steps");
        return made.defined() ? THPVariable_Wrap(std::move(made)) : own(a[7]);
    });
}

struct Chunk {                                     // the inputs that forward and backward share
    qd_shape s;
    int64_t B, T, H, dk, dv;
    at::ScalarType dt;
    c10::Device dev = c10::Device(c10::kCPU);
    const void *q, *k, *v, *beta, *alpha, *lam;
    const float* h0;
    Chunk(const at::Tensor& tq, const at::Tensor* tk, const at::Tensor& tv, const at::Tensor* tb, const at::Tensor* ta,
          const at::Tensor* tl, const at::Tensor* th, int chunk) {
        want_dims(tq, 4);
        B = tq.size(0); T = tq.size(1); H = tq.size(2); dk = tq.size(3); dv = tv.size(-1);
        dt = tq.scalar_type();
        dev = tq.device();
        s = qd_shape{(int)B, (int)T, (int)H, (int)dk, (int)dv, chunk, dtype_code(tq)};
        q = ptr(&tq, dt, {B, T, H, dk}, "q");
        k = ptr(tk, dt, {B, T, H, dk}, "k");
        v = ptr(&tv, dt, {B, T, H, dv}, "v");
        beta = ptr(tb, dt, {B, T, H}, "beta");
        alpha = ptr(ta, dt, {B, T, H}, "alpha");
        lam = ptr(tl, dt, {B, T, H}, "lam");
        h0 = static_cast<const float*>(ptr(th, at::kFloat, {B, H, dk, dv}, "h0"));
    }
    Chunk(PyObject* const* a, int chunk)           // q, k, v, beta, alpha, lam, h0
        : Chunk(needed(a[0], "q"), tensor(a[1], "k"), needed(a[2], "v"), tensor(a[3], "beta"), tensor(a[4], "alpha"),
                tensor(a[5], "lam"), tensor(a[6], "h0"), chunk) {}
    at::Tensor workspace(int for_backward) const {
        const size_t n = qdelta_chunk_workspace_bytes(&s, for_backward);
        if (n == 0) fail("unsupported or invalid shape for the chunkwise kernels");
        return empty({(int64_t)n}, at::kByte, dev);
    }
};
int to_int(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw Raised{};
    return (int)v;
}

// chunk_fwd(q, k, v, beta, alpha, lam, h0, chunk, workspace, o, hT, want_hT, flags) -> (o, hT, workspace)
PyObject* chunk_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!arity(n, 13)) return nullptr;
    return guarded([&]() -> PyObject* {
        const Chunk c(a, to_int(a[7]));
        const unsigned flags = (unsigned)PyLong_AsUnsignedLong(a[12]);
        at::Tensor ws_made, o_made, hT_made;
        const at::Tensor *ws = tensor(a[8], "workspace"), *o = tensor(a[9], "o"), *hT = tensor(a[10], "hT");
        if (!ws) { ws_made = c.workspace(flags & QD_FWD_SAVE_FOR_BWD ? 1 : 0); ws = &ws_made; }
        if (!o) { o_made = empty({c.B, c.T, c.H, c.dv}, c.dt, c.dev); o = &o_made; }
        if (!hT && a[11] == Py_True) { hT_made = empty({c.B, c.H, c.dk, c.dv}, at::kFloat, c.dev); hT = &hT_made; }
        void* op = ptr(o, c.dt, {c.B, c.T, c.H, c.dv}, "o");
        float* hp = static_cast<float*>(ptr(hT, at::kFloat, {c.B, c.H, c.dk, c.dv}, "hT"));
        int rc;
        {
            NoGil ng;
            rc = qdelta_chunk_fwd(&c.s, c.q, c.k, c.v, c.beta, c.alpha, c.lam, c.h0, op, hp, ws->data_ptr(), (size_t)ws->numel(),
                                  flags, stream());
        }
        check(rc, "qdelta_chunk_fwd");
        PyObject* r = PyTuple_New(3);
        if (!r) throw Raised{};
        PyTuple_SET_ITEM(r, 0, o_made.defined() ? THPVariable_Wrap(std::move(o_made)) : own(a[9]));
        PyTuple_SET_ITEM(r, 1, hT_made.defined() ? THPVariable_Wrap(std::move(hT_made)) : own(a[10]));
        PyTuple_SET_ITEM(r, 2, ws_made.defined() ? THPVariable_Wrap(std::move(ws_made)) : own(a[8]));
        return r;
    });
}

// chunk_bwd(q, k, v, beta, alpha, lam, h0, chunk, dO, dhT, workspace, out, want_dh0, flags): fills the dict `out`
PyObject* chunk_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!arity(n, 14)) return nullptr;
    return guarded([&]() -> PyObject* {
        const Chunk c(a, to_int(a[7]));
        const unsigned flags = (unsigned)PyLong_AsUnsignedLong(a[13]);
        const void* dO = ptr(tensor(a[8], "dO"), c.dt, {c.B, c.T, c.H, c.dv}, "dO");
        const float* dhT = static_cast<const float*>(ptr(tensor(a[9], "dhT"), at::kFloat, {c.B, c.H, c.dk, c.dv}, "dhT"));
        at::Tensor ws_made;
        const at::Tensor* ws = tensor(a[10], "workspace");
        if (!ws) { ws_made = c.workspace(1); ws = &ws_made; }
        if (!PyDict_Check(a[11])) { PyErr_SetString(PyExc_TypeError, "out must be a dict"); throw Raised{}; }
        // a gradient that the caller does not supply is allocated; an unwanted one is None
        auto grad = [&](const char* name, at::ScalarType dt, c10::IntArrayRef shape, bool wanted) -> void* {
            PyObject* have = PyDict_GetItemString(a[11], name);
            if (have) return ptr(tensor(have, name), dt, shape, name);
            if (!wanted) { if (PyDict_SetItemString(a[11], name, Py_None)) throw Raised{}; return nullptr; }
            at::Tensor t = empty(shape, dt, c.dev);
            void* p = t.data_ptr();
            PyObject* w = THPVariable_Wrap(std::move(t));
            const int bad = w ? PyDict_SetItemString(a[11], name, w) : -1;
            Py_XDECREF(w);
            if (bad) throw Raised{};
            return p;
        };
        void* dq = grad("dq", c.dt, {c.B, c.T, c.H, c.dk}, true);
        void* dk = grad("dk", c.dt, {c.B, c.T, c.H, c.dk}, true);
        void* dv = grad("dv", c.dt, {c.B, c.T, c.H, c.dv}, true);
        float* db = static_cast<float*>(grad("dbeta", at::kFloat, {c.B, c.T, c.H}, true));
        float* da = static_cast<float*>(grad("dalpha", at::kFloat, {c.B, c.T, c.H}, c.alpha != nullptr));
        float* dl = static_cast<float*>(grad("dlam", at::kFloat, {c.B, c.T, c.H}, c.lam != nullptr));
        float* dh0 = static_cast<float*>(grad("dh0", at::kFloat, {c.B, c.H, c.dk, c.dv}, a[12] == Py_True));
        int rc;
        {
            NoGil ng;
            rc = qdelta_chunk_bwd(&c.s, c.q, c.k, c.v, c.beta, c.alpha, c.lam, c.h0, dO, dhT, dq, dk, dv, db, da, dl, dh0,
                                  ws->data_ptr(), (size_t)ws->numel(), flags, stream());
        }
        check(rc, "qdelta_chunk_bwd");
        return own(a[11]);
    });
}

// ---- autograd: the pair forward / backward as one node, without Python on the way ------------------------------------
// (a Python-level Function spent 120 us per pair in the interpreter, more than the kernels of a short sequence take)
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;
constexpr int kChunk = 64;

using MaybeTensor = std::optional<at::Tensor>;
const at::Tensor* maybe(const MaybeTensor& t) { return t ? &*t : nullptr; }

struct ChunkNode : torch::autograd::Function<ChunkNode> {
    static variable_list forward(AutogradContext* ctx, const at::Tensor& q, const at::Tensor& k, const at::Tensor& v,
                                 const at::Tensor& beta, const MaybeTensor& alpha, const MaybeTensor& lam, const MaybeTensor& h0,
                                 int64_t flags, bool need_grad) {
        const Chunk c(q, &k, v, &beta, maybe(alpha), maybe(lam), maybe(h0), kChunk);
        at::Tensor ws = c.workspace(need_grad ? 1 : 0);
        at::Tensor o = empty({c.B, c.T, c.H, c.dv}, c.dt, c.dev), hT = empty({c.B, c.H, c.dk, c.dv}, at::kFloat, c.dev);
        check(qdelta_chunk_fwd(&c.s, c.q, c.k, c.v, c.beta, c.alpha, c.lam, c.h0, o.data_ptr(), hT.data_ptr<float>(),
                               ws.data_ptr(), (size_t)ws.numel(), (unsigned)flags | (need_grad ? QD_FWD_SAVE_FOR_BWD : 0), stream()),
              "qdelta_chunk_fwd");
        ctx->set_materialize_grads(false);         // an unused output costs no tensor of zeros
        if (need_grad) {
            auto or_none = [](const MaybeTensor& t) { return t ? *t : at::Tensor(); };
            ctx->save_for_backward({q, k, v, beta, or_none(alpha), or_none(lam), or_none(h0), ws});
            ctx->saved_data["flags"] = flags;
        }
        return {o, hT};
    }
    // a QdeltaError from a thread of the autograd engine, which does not hold the interpreter
    [[noreturn]] static void raise(const std::string& what) {
        pybind11::gil_scoped_acquire gil;
        PyErr_SetString(g_error, what.c_str());
        python_error e;
        e.persist();
        throw std::move(e);
    }
    static variable_list backward(AutogradContext* ctx, variable_list g) {
        const variable_list in = ctx->get_saved_variables();
        const at::Tensor &q = in[0], &v = in[2], &beta = in[3], &alpha = in[4], &lam = in[5], &h0 = in[6], &ws = in[7];
        if (q.dim() != 4 || v.dim() != 4) raise("q and v must have four dimensions");
        const int64_t B = q.size(0), T = q.size(1), H = q.size(2), dk = q.size(3), dv = v.size(3);
        const at::ScalarType dt = q.scalar_type();
        const c10::Device dev = q.device();
        const qd_shape s{(int)B, (int)T, (int)H, (int)dk, (int)dv, kChunk, dt == at::kFloat ? QD_F32 : QD_BF16};
        const at::Tensor dO = g[0].defined() ? g[0].contiguous() : at::zeros_like(v);
        const at::Tensor dhT = g[1].defined() ? g[1].contiguous().to(at::kFloat) : at::Tensor();
        // Saved-tensor hooks may hand back other tensors than were saved, tensor hooks other gradients: none of them goes to a
        // kernel unseen.
        auto seen = [&](const at::Tensor& t, at::ScalarType type, c10::IntArrayRef shape, const char* name) {
            if (!t.defined()) return;
            const std::string c = complaint(t, type, shape, name);
            if (!c.empty()) raise(c);
        };
        if (dt != at::kFloat && dt != at::kBFloat16) raise("q must be fp32 or bf16");
        seen(q, dt, {B, T, H, dk}, "q"); seen(in[1], dt, {B, T, H, dk}, "k"); seen(v, dt, {B, T, H, dv}, "v");
        seen(beta, dt, {B, T, H}, "beta"); seen(alpha, dt, {B, T, H}, "alpha"); seen(lam, dt, {B, T, H}, "lam");
        seen(h0, at::kFloat, {B, H, dk, dv}, "h0"); seen(ws, at::kByte, {ws.numel()}, "the saved workspace");
        seen(dO, dt, {B, T, H, dv}, "dO"); seen(dhT, at::kFloat, {B, H, dk, dv}, "dhT");
        auto make = [&](c10::IntArrayRef shape, at::ScalarType t) { return at::Tensor(at::detail::empty_cuda(shape, t, dev, std::nullopt)); };
        at::Tensor gq = make({B, T, H, dk}, dt), gk = make({B, T, H, dk}, dt), gv = make({B, T, H, dv}, dt), gh;
        // gradients of the gates come in fp32; one conversion takes all of them to the gates' type
        const int64_t n = 1 + (alpha.defined() ? 1 : 0) + (lam.defined() ? 1 : 0);
        at::Tensor gates = make({n, B, T, H}, at::kFloat);
        float* base = gates.data_ptr<float>();
        const int64_t row = B * T * H;
        float *db = base, *da = alpha.defined() ? base + row : nullptr, *dl = lam.defined() ? base + (n - 1) * row : nullptr;
        if (h0.defined()) gh = make({B, H, dk, dv}, at::kFloat);
        auto p = [](const at::Tensor& t) -> void* { return t.defined() ? t.data_ptr() : nullptr; };
        const unsigned flags = (unsigned)ctx->saved_data["flags"].toInt() | QD_BWD_REUSE_FWD;
        const int rc = qdelta_chunk_bwd(&s, p(q), p(in[1]), p(v), p(beta), p(alpha), p(lam), (const float*)p(h0), p(dO),
                                        (const float*)p(dhT), p(gq), p(gk), p(gv), db, da, dl, (float*)p(gh), ws.data_ptr(),
                                        (size_t)ws.numel(), flags, stream());
        if (rc != QD_OK) raise("qdelta_chunk_bwd failed: " + std::string(qdelta_status_string(rc)) + " (" + std::to_string(rc) + ")");
        if (dt != at::kFloat) gates = gates.to(dt);
        return {gq, gk, gv, gates.select(0, 0), alpha.defined() ? gates.select(0, 1) : at::Tensor(),
                lam.defined() ? gates.select(0, n - 1) : at::Tensor(), gh, at::Tensor(), at::Tensor()};
    }
};

// chunk_autograd(q, k, v, beta, alpha, lam, h0, flags) -> (o, hT)
PyObject* chunk_autograd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (!arity(n, 8)) return nullptr;
    return guarded([&]() -> PyObject* {
        static const char* names[7] = {"q", "k", "v", "beta", "alpha", "lam", "h0"};
        MaybeTensor t[7];
        bool need = false;
        for (int i = 0; i < 7; ++i) {
            const at::Tensor* x = i < 4 ? &needed(a[i], names[i]) : tensor(a[i], names[i]);
            if (!x) continue;
            need = need || x->requires_grad();
            t[i] = x->contiguous();
        }
        const variable_list r = ChunkNode::apply(*t[0], *t[1], *t[2], *t[3], t[4], t[5], t[6], (int64_t)to_int(a[7]),
                                                 need && at::GradMode::is_enabled());
        PyObject* out = PyTuple_New(2);
        if (!out) throw Raised{};
        PyTuple_SET_ITEM(out, 0, THPVariable_Wrap(r[0]));
        PyTuple_SET_ITEM(out, 1, THPVariable_Wrap(r[1]));
        return out;
    });
}

PyObject* set_error(PyObject*, PyObject* e) {
    Py_XINCREF(e);
    Py_XSETREF(g_error, e);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"recurrent_step", (PyCFunction)(void*)recurrent_step, METH_FASTCALL, nullptr},
    {"recurrent_steps", (PyCFunction)(void*)recurrent_steps, METH_FASTCALL, nullptr},
    {"chunk_fwd", (PyCFunction)(void*)chunk_fwd, METH_FASTCALL, nullptr},
    {"chunk_bwd", (PyCFunction)(void*)chunk_bwd, METH_FASTCALL, nullptr},
    {"chunk_autograd", (PyCFunction)(void*)chunk_autograd, METH_FASTCALL, nullptr},
    {"set_error", set_error, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_qdelta_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__qdelta_host(void) { return PyModule_Create(&module_def); }
