// marshal.cpp -- the two compute calls of include/fibattn.h for PyTorch
// tensors: checks, output allocation and the call, natively.  binding.py holds
// the signatures; nothing of the computation is here.  A forward call of
// B1 H8 Hkv2 T64 took 36-43 us of host time interpreted (its kernels 10), and
// takes 12-13 us here (GB300, Grace host).
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <cuda_runtime_api.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/fibattn.h"

namespace {

using at::Tensor;

[[noreturn]] void value_error(const char* msg) {
    PyErr_SetString(PyExc_ValueError, msg);
    throw python_error();
}

const Tensor& tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor, not %s", name, Py_TYPE(o)->tp_name);
        throw python_error();
    }
    return THPVariable_Unpack(o);
}
// None reads as an undefined tensor.
Tensor optional(PyObject* o, const char* name) { return o == Py_None ? Tensor() : tensor(o, name); }

long as_int(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
}
double as_float(PyObject* o) {
    if (PyFloat_CheckExact(o)) return PyFloat_AS_DOUBLE(o);
    PyObject* const f = PyNumber_Float(o);        // what float() takes
    if (!f) throw python_error();
    const double v = PyFloat_AS_DOUBLE(f);
    Py_DECREF(f);
    return v;
}
bool as_bool(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) throw python_error();
    return v != 0;
}

// The base sequence: a C-contiguous float32 array (binding.py makes it one).
struct Offsets {
    Py_buffer b;
    const float* f;
    int K;
    explicit Offsets(PyObject* o) {
        if (PyObject_GetBuffer(o, &b, PyBUF_ND | PyBUF_C_CONTIGUOUS) != 0) throw python_error();
        f = static_cast<const float*>(b.buf);
        K = b.ndim > 0 ? (int)b.shape[0] : -1;    // (refused by the library, as a scalar was by len())
    }
    ~Offsets() { PyBuffer_Release(&b); }
};

void* ptr(const Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }

// Sizes, options and the checks both calls make.
struct Call {
    int B, H, T, D, W, dtype;
    fibattn_opts o;
    Call(const Tensor& q, const Tensor& k, int w, const Offsets& f, const Tensor& rk, const Tensor& res, PyObject* const* a) {
        if (q.dim() != 4 || k.dim() < 2) value_error("q must be [B,H,T,D] and k [B,Hkv,T,D]");
        B = (int)q.size(0); H = (int)q.size(1); T = (int)q.size(2); D = (int)q.size(3);
        W = w;
        const auto dt = q.scalar_type();
        if (dt != at::kFloat && dt != at::kBFloat16) {
            PyErr_Format(PyExc_TypeError, "unsupported dtype %s: fp32 or bf16", c10::toString(dt));
            throw python_error();
        }
        dtype = dt == at::kFloat ? FIBATTN_F32 : FIBATTN_BF16;
        if (rk.defined()) {
            const auto want = k.scalar_type() == at::kBFloat16 ? at::kHalf : at::kFloat;
            if (!(rk.is_cuda() && rk.device() == q.device() && rk.is_contiguous() && rk.scalar_type() == want && rk.sizes() == k.sizes()))
                value_error(want == at::kHalf ? "rotated_k must be a contiguous CUDA torch.float16 tensor of k's shape"
                                              : "rotated_k must be a contiguous CUDA torch.float32 tensor of k's shape");
        }
        if (res.defined() && !(res.is_cuda() && res.device() == q.device() && res.is_contiguous() &&
                               (size_t)(res.numel() * res.element_size()) >= fibattn_residual_bytes(B, H, T, D, W, f.K, dtype)))
            value_error("residuals must be a contiguous CUDA buffer of residual_bytes(...) bytes");
        o = fibattn_opts{};
        o.rope_base = (float)as_float(a[0]);
        o.scale = (float)as_float(a[1]);
        o.no_dedup = as_bool(a[2]) ? 0 : 1;
        o.round_offsets = as_bool(a[3]) ? 1 : 0;
        o.Hkv = (int)k.size(1);
        o.rotated_k = ptr(rk);
        o.residuals = ptr(res);
    }
};

// The library sees pointers and the extents of q (and k's heads): whatever it
// reads or writes through the others is checked to be there, before any launch.
void check_inputs(const Tensor& q, std::initializer_list<const Tensor*> ts, const char* msg) {
    for (const Tensor* t : ts)
        if (t->defined() && !(t->is_cuda() && t->is_contiguous() && t->scalar_type() == q.scalar_type())) value_error(msg);
    for (const Tensor* t : ts)
        if (t->defined() && t->device() != q.device()) value_error("the tensors of a call must be on one device");
}
void check_kv(const Tensor& q, const Tensor& k, const Tensor& v) {
    const int64_t n = q.size(0) * k.size(1) * q.size(2) * q.size(3);
    if (k.numel() != n || v.numel() != n) value_error("k and v must be [B,Hkv,T,D], with q's B, T and D");
}
// A buffer of the caller's: n entries of type dt (more are allowed).
void check_buffer(const Tensor& t, const Tensor& q, at::ScalarType dt, int64_t n, const char* name) {
    if (!t.defined() || (t.numel() >= n && t.scalar_type() == dt && t.is_contiguous() && t.device() == q.device())) return;
    PyErr_Format(PyExc_ValueError, "%s must be contiguous, %s, on q's device and hold %lld entries", name,
                 c10::toString(dt), (long long)n);
    throw python_error();
}
// (its size is checked by the library)
void check_workspace(const Tensor& ws, const Tensor& q) {
    if (ws.defined() && !(ws.is_contiguous() && ws.device() == q.device()))
        value_error("workspace must be contiguous and on q's device");
}

Tensor like(const Tensor& given, const Tensor& t) { return given.defined() ? given : at::empty(t.sizes(), t.options()); }

Tensor bytes(size_t need, const Tensor& q) {
    return at::empty({(int64_t)std::max<size_t>(need, 256)}, q.options().dtype(at::kByte));
}

// The device of a call is that of its tensors.  (A plain guard asks the runtime
// for the current device at both ends.)
struct OnDevice {
    c10::cuda::OptionalCUDAGuard guard;
    explicit OnDevice(const Tensor& q) {
        if (c10::cuda::current_device() != q.device().index()) guard.set_device(q.device());
    }
};

// The stream of a call: the current one, or the caller's.  Memory allocated
// while it stands comes from that stream's pool: a workspace released on return
// is reused by later work of the same stream only, where the current stream's
// next allocation could have had it while the kernels still ran.
struct OnStream {
    const c10::cuda::CUDAStream current;
    cudaStream_t st;
    c10::cuda::OptionalCUDAStreamGuard guard;
    OnStream(PyObject* o, const Tensor& q)
        : current(c10::cuda::getCurrentCUDAStream(q.device().index())), st(current.stream()) {
        if (o == Py_None) return;
        st = static_cast<cudaStream_t>(PyLong_AsVoidPtr(o));
        if (!st && PyErr_Occurred()) throw python_error();
        const cudaStream_t pool = st == cudaStreamLegacy ? nullptr : st;      // (two names of the default stream)
        if (pool != current.stream())
            guard.reset_stream(pool ? c10::cuda::getStreamFromExternal(pool, current.device_index())
                                    : c10::cuda::getDefaultCUDAStream(current.device_index()));
    }
    // Results made here are the caller's, who may use and drop them on the current stream.
    void results(std::initializer_list<std::pair<const Tensor*, bool>> ts) const {
        if (!guard.current_stream()) return;
        for (const auto& [t, made] : ts)
            if (made && t->defined()) t->record_stream(current);
    }
};

bool arity(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

int call_fwd(const Call& c, const Tensor& q, const Tensor& k, const Tensor& v, const Tensor& out, const Tensor& lse,
             const Tensor& ws, float alpha, const Offsets& f, void* st) {
    void *pq = ptr(q), *pk = ptr(k), *pv = ptr(v), *po = ptr(out), *pl = ptr(lse), *pw = ptr(ws);
    const size_t nw = ws.defined() ? (size_t)ws.numel() : 0;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fibattn_fwd(pq, pk, pv, po, static_cast<float*>(pl), c.B, c.H, c.T, c.D, c.W, alpha, f.f, f.K, c.dtype, &c.o, pw, nw, st);
    Py_END_ALLOW_THREADS
    return rc;
}

PyObject* tuple_of(std::initializer_list<const Tensor*> ts) {     // an undefined tensor is None
    PyObject* r = PyTuple_New((Py_ssize_t)ts.size());
    if (!r) return nullptr;
    int i = 0;
    for (const Tensor* t : ts) {
        PyObject* x = Py_None;
        if (t->defined()) x = THPVariable_Wrap(*t);
        else Py_INCREF(Py_None);
        PyTuple_SET_ITEM(r, i++, x);
    }
    return r;
}

const char kFwdInputs[] = "q, k, v must be contiguous CUDA tensors of one dtype";

// fwd(q, k, v, offsets, W, alpha, rope_base, scale, dedup, round_offsets, kernel, out, lse, workspace, rotated_k,
//     residuals, stream) -> (out, lse), or the call's status when it is not 0
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arity(n, 17)) return nullptr;
    const Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
    const Offsets f(a[3]);
    const Tensor rk = optional(a[14], "rotated_k"), res = optional(a[15], "residuals");
    Call c(q, k, (int)as_int(a[4]), f, rk, res, a + 6);
    const float alpha = (float)as_float(a[5]);
    c.o.fwd_kernel = (int)as_int(a[10]);
    const Tensor given = optional(a[11], "out");
    Tensor lse = optional(a[12], "lse"), ws = optional(a[13], "workspace");
    check_kv(q, k, v);
    check_buffer(given, q, q.scalar_type(), q.numel(), "out");
    check_buffer(lse, q, at::kFloat, q.size(0) * q.size(1) * q.size(2), "lse");
    check_workspace(ws, q);
    check_inputs(q, {&q, &k, &v}, kFwdInputs);
    const OnDevice device(q);
    const OnStream on(a[16], q);
    const Tensor out = like(given, q);
    const bool own_lse = !lse.defined();
    if (!lse.defined()) lse = at::empty({c.B, c.H, c.T}, q.options().dtype(at::kFloat));
    if (!ws.defined()) ws = bytes(fibattn_fwd_workspace_bytes(c.B, c.H, c.T, c.D, c.W, f.K, c.dtype, &c.o), q);
    const int rc = call_fwd(c, q, k, v, out, lse, ws, alpha, f, on.st);
    on.results({{&out, !given.defined()}, {&lse, own_lse}});
    return rc ? PyLong_FromLong(rc) : tuple_of({&out, &lse});
    END_HANDLE_TH_ERRORS
}

// fwd_keep(q, k, v, offsets, W, alpha, rope_base, scale, dedup, round_offsets) -> (out, lse, rotated_k, residuals or
// None): the forward of a training step on the current stream, with what its backward reads; residuals where the
// tensor-core forward applies.  Or the call's status when it is not 0.
PyObject* fwd_keep(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arity(n, 10)) return nullptr;
    const Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
    const Offsets f(a[3]);
    Call c(q, k, (int)as_int(a[4]), f, Tensor(), Tensor(), a + 6);
    const float alpha = (float)as_float(a[5]);
    check_kv(q, k, v);
    check_inputs(q, {&q, &k, &v}, kFwdInputs);
    const OnDevice device(q);
    const Tensor out = at::empty(q.sizes(), q.options());
    const Tensor lse = at::empty({c.B, c.H, c.T}, q.options().dtype(at::kFloat));
    const Tensor rk = at::empty(k.sizes(), k.options().dtype(c.dtype == FIBATTN_BF16 ? at::kHalf : at::kFloat));
    c.o.rotated_k = ptr(rk);
    void* const st = c10::cuda::getCurrentCUDAStream(q.device().index()).stream();
    const size_t nr = fibattn_residual_bytes(c.B, c.H, c.T, c.D, c.W, f.K, c.dtype);
    Tensor res;
    int rc = FIBATTN_ERR_UNSUPPORTED;
    if (nr > 0) {
        res = at::empty({(int64_t)nr}, q.options().dtype(at::kByte));
        c.o.residuals = ptr(res);
        rc = call_fwd(c, q, k, v, out, lse, Tensor(), alpha, f, st);
    }
    if (rc == FIBATTN_ERR_UNSUPPORTED) {
        res = Tensor();
        c.o.residuals = nullptr;
        rc = call_fwd(c, q, k, v, out, lse, Tensor(), alpha, f, st);
    }
    return rc ? PyLong_FromLong(rc) : tuple_of({&out, &lse, &rk, &res});
    END_HANDLE_TH_ERRORS
}

// bwd(q, k, v, offsets, W, alpha, rope_base, scale, dedup, round_offsets, kernel, out, lse, workspace, rotated_k,
//     residuals, stream, dout, dq, dk, dv, dtheta, dd, rung_grads)
//   -> (dq, dk, dv, dtheta [1] or None, dd [K] or None), or the call's status when it is not 0
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!arity(n, 24)) return nullptr;
    const Tensor &q = tensor(a[0], "q"), &k = tensor(a[1], "k"), &v = tensor(a[2], "v");
    const Tensor &lse = tensor(a[12], "lse"), &dout = tensor(a[17], "dout");
    const Offsets f(a[3]);
    const Tensor rk = optional(a[14], "rotated_k"), res = optional(a[15], "residuals"), out = optional(a[11], "out");
    Call c(q, k, (int)as_int(a[4]), f, rk, res, a + 6);
    const float alpha = (float)as_float(a[5]);
    c.o.bwd_kernel = (int)as_int(a[10]);
    const bool rung_grads = as_bool(a[23]);
    Tensor dq = optional(a[18], "dq"), dk = optional(a[19], "dk"), dv = optional(a[20], "dv");
    Tensor dth = optional(a[21], "dtheta"), dd = optional(a[22], "dd"), ws = optional(a[13], "workspace");
    check_kv(q, k, v);
    if (dout.numel() != q.numel()) value_error("dout must be of q's shape");
    check_buffer(out, q, q.scalar_type(), q.numel(), "out");
    check_buffer(lse, q, at::kFloat, q.size(0) * q.size(1) * q.size(2), "lse");
    check_buffer(dq, q, q.scalar_type(), q.numel(), "dq");
    check_buffer(dk, q, q.scalar_type(), k.numel(), "dk");
    check_buffer(dv, q, q.scalar_type(), k.numel(), "dv");
    check_buffer(dth, q, at::kFloat, 1, "dtheta");
    check_buffer(dd, q, at::kFloat, f.K, "dd");
    check_workspace(ws, q);
    check_inputs(q, {&q, &k, &v, &dout, &out}, "q, k, v, dout, out must be contiguous CUDA tensors of one dtype");
    const OnDevice device(q);
    const OnStream on(a[16], q);
    const bool own[5] = {!dq.defined(), !dk.defined(), !dv.defined(), !dth.defined(), !dd.defined()};
    dq = like(dq, q); dk = like(dk, k); dv = like(dv, v);
    if (rung_grads) {
        if (!dth.defined()) dth = at::empty({1}, q.options().dtype(at::kFloat));
        if (!dd.defined()) dd = at::empty({std::max(f.K, 1)}, q.options().dtype(at::kFloat));
    }
    if (!ws.defined()) ws = bytes(fibattn_bwd_workspace_bytes(c.B, c.H, c.T, c.D, c.W, f.K, c.dtype, &c.o), q);
    void *pq = ptr(q), *pk = ptr(k), *pv = ptr(v), *po = ptr(out), *pl = ptr(lse), *pg = ptr(dout), *pw = ptr(ws);
    void *pdq = ptr(dq), *pdk = ptr(dk), *pdv = ptr(dv), *pth = ptr(dth), *pdd = ptr(dd);
    const size_t nw = (size_t)ws.numel();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fibattn_bwd(pq, pk, pv, po, static_cast<const float*>(pl), pg, pdq, pdk, pdv, static_cast<float*>(pth),
                     static_cast<float*>(pdd), c.B, c.H, c.T, c.D, c.W, alpha, f.f, f.K, c.dtype, &c.o, pw, nw, on.st);
    Py_END_ALLOW_THREADS
    on.results({{&dq, own[0]}, {&dk, own[1]}, {&dv, own[2]}, {&dth, own[3]}, {&dd, own[4]}});
    if (rc) return PyLong_FromLong(rc);
    if (dth.defined() && !(dth.dim() == 1 && dth.size(0) == 1)) dth = dth.slice(0, 0, 1);
    if (dd.defined() && !(dd.dim() == 1 && dd.size(0) == f.K)) dd = dd.slice(0, 0, f.K);
    return tuple_of({&dq, &dk, &dv, &dth, &dd});
    END_HANDLE_TH_ERRORS
}

// alpha_of_theta(theta) -> 0.5 + sigmoid(theta), as the library computes it
PyObject* alpha_of_theta(PyObject*, PyObject* o) {
    HANDLE_TH_ERRORS
    const float th = (float)as_float(o);
    float al = 0.f;
    const int rc = fibattn_alpha_schedule(1, 1, &th, 0, &al);
    if (rc) value_error(fibattn_last_error());
    return PyFloat_FromDouble(al);
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(fwd)), METH_FASTCALL, nullptr},
    {"fwd_keep", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(fwd_keep)), METH_FASTCALL, nullptr},
    {"bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(bwd)), METH_FASTCALL, nullptr},
    {"alpha_of_theta", alpha_of_theta, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "fibattn_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_fibattn_marshal() { return PyModule_Create(&module); }
