// The Python binding's call path: takes torch tensors apart, allocates outputs, calls the C ABI.
//
// A decode step or a short prefill runs on the GPU for 7 to 15 us, less than what the same steps cost when written in
// Python with ctypes (a dozen attribute reads, the stream object, the conversion of fifteen arguments): there the host
// was the bound.  Here a call costs about a microsecond beside the launches themselves.  The interpreter lock is
// released around the library call, which may block when the launch queue is full.
// Measured through the Python entry points, back to back on one stream (ctypes -> here): one decode step of one sequence
// 9.4 -> 6.5 us, of eight 9.3 -> 8.0, plan and prefill of 1000 tokens in a small geometry 24.2 -> 13.5; the host's share of
// a decode step 10.6 -> 3.4 us.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/bf1.h"

namespace {

PyObject* g_error = nullptr;   // the binding's Bf1Error

struct PyRaised {};            // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* msg) {
    PyErr_SetString(type, msg);
    throw PyRaised();
}
void require(bool ok, const char* what) {
    if (!ok) raise(PyExc_AssertionError, what);
}
const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "expected a torch.Tensor");
    return THPVariable_Unpack(o);
}
long long integer(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyRaised();
    return v;
}
template <typename T>
T* address(PyObject* o) {
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) throw PyRaised();
    return static_cast<T*>(p);
}
float scale_of(PyObject* o) {   // None or 0: the library's default
    if (o == Py_None) return 0.f;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyRaised();
    return static_cast<float>(v);
}
void* stream_of(PyObject* o) {  // None: the current stream of the current device
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    return address<void>(o);
}
at::Tensor lse_like(const at::Tensor& q, int64_t heads, int64_t rows) {
    return at::empty({heads, rows}, q.options().dtype(at::kFloat));
}
// One library call with the interpreter lock released; an error status becomes the binding's exception.
template <typename F>
void call(F&& f) {
    int rc;
    {
        PyThreadState* state = PyEval_SaveThread();
        rc = f();
        PyEval_RestoreThread(state);
    }
    if (rc == BF1_OK) return;
    PyObject* e = PyObject_CallFunction(g_error, "is", rc, bf1_last_error());
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw PyRaised();
}
PyObject* pair(const at::Tensor& a, const at::Tensor& b) {
    PyObject *x = THPVariable_Wrap(a), *y = THPVariable_Wrap(b);
    PyObject* t = x && y ? PyTuple_Pack(2, x, y) : nullptr;
    Py_XDECREF(x);
    Py_XDECREF(y);
    return t;
}

struct Qkv {
    int64_t T, hq, hkv, d;
};
Qkv check_qkv(const at::Tensor& q, const at::Tensor& k, const at::Tensor& v) {
    for (const at::Tensor* t : {&q, &k, &v})
        require(t->is_cuda() && t->scalar_type() == at::kBFloat16 && t->is_contiguous() && t->dim() == 3,
                "q, k and v must be contiguous 3-d bf16 CUDA tensors");
    require(k.sizes() == v.sizes() && k.size(0) == q.size(0) && k.size(2) == q.size(2), "shapes of q, k and v do not match");
    return {q.size(0), q.size(1), k.size(1), q.size(2)};
}

// Every function takes positional arguments; `*`-marked ones may be None.
// plan_route(cu_seqlens, total, max_seqlen, cfg address, route address, stream*)
PyObject* plan_route(PyObject* const* a) {
    const at::Tensor& cu = tensor(a[0]);
    require(cu.is_cuda() && cu.scalar_type() == at::kInt && cu.is_contiguous(), "cu_seqlens must be a contiguous int32 CUDA tensor");
    const int32_t batch = static_cast<int32_t>(cu.numel() - 1), max_seqlen = static_cast<int32_t>(integer(a[2]));
    const int64_t total = integer(a[1]);
    const auto* cfg = address<const bf1_route_cfg>(a[3]);
    const auto* route = address<const bf1_route>(a[4]);
    void* stream = stream_of(a[5]);
    const auto* cup = static_cast<const int32_t*>(cu.data_ptr());
    call([&] { return bf1_plan_route(cup, batch, total, max_seqlen, cfg, route, stream); });
    Py_RETURN_NONE;
}

// forward(which, q, k, v, cu_seqlens, max_seqlen, scale*, out*, lse*, stream*, x, y, z)
//   which 0: bf1_attn_fwd, x = route address;  1: bf1_dense_causal_fwd, x = work tensor*;
//   2: bf1_attn_fwd_noalloc, x = total tokens, y = cfg address, z = status tensor*
PyObject* forward(PyObject* const* a) {
    const long long which = integer(a[0]);
    const at::Tensor &q = tensor(a[1]), &k = tensor(a[2]), &v = tensor(a[3]), &cu = tensor(a[4]);
    const Qkv g = check_qkv(q, k, v);
    const int32_t max_seqlen = static_cast<int32_t>(integer(a[5]));
    const float scale = scale_of(a[6]);
    const at::Tensor out = a[7] == Py_None ? at::empty_like(q) : tensor(a[7]);
    const at::Tensor lse = a[8] == Py_None ? lse_like(q, g.hq, g.T) : tensor(a[8]);
    void* stream = stream_of(a[9]);
    const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr();
    const auto* cup = static_cast<const int32_t*>(cu.data_ptr());
    const int32_t batch = static_cast<int32_t>(cu.numel() - 1), hq = g.hq, hkv = g.hkv, d = g.d;
    void* op = out.data_ptr();
    auto* lp = static_cast<float*>(lse.data_ptr());
    if (which == 0) {
        const auto* route = address<const bf1_route>(a[10]);
        call([&] { return bf1_attn_fwd(qp, kp, vp, cup, batch, g.T, max_seqlen, hq, hkv, d, scale, route, op, lp, stream); });
    } else if (which == 1) {
        auto* work = a[10] == Py_None ? nullptr : static_cast<int32_t*>(tensor(a[10]).data_ptr());
        call([&] { return bf1_dense_causal_fwd(qp, kp, vp, cup, batch, g.T, max_seqlen, hq, hkv, d, scale, op, lp, work, stream); });
    } else {
        const int64_t total = a[10] == Py_None ? g.T : integer(a[10]);
        const auto* cfg = address<const bf1_route_cfg>(a[11]);
        auto* status = a[12] == Py_None ? nullptr : static_cast<int32_t*>(tensor(a[12]).data_ptr());
        call([&] {
            return bf1_attn_fwd_noalloc(qp, kp, vp, cup, batch, total, max_seqlen, hq, hkv, d, scale, cfg, op, lp, status, stream);
        });
    }
    return pair(out, lse);
}

// backward(q, k, v, o, lse, d_o, cu_seqlens, max_seqlen, route address, scale*, workspace, stream*)
PyObject* backward(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]), &o = tensor(a[3]), &lse = tensor(a[4]),
                     &d_o = tensor(a[5]), &cu = tensor(a[6]), &ws = tensor(a[10]);
    const Qkv g = check_qkv(q, k, v);
    require(d_o.sizes() == q.sizes() && d_o.scalar_type() == at::kBFloat16 && d_o.is_contiguous(),
            "d_o must be a contiguous bf16 tensor of q's shape");
    const int32_t max_seqlen = static_cast<int32_t>(integer(a[7]));
    const auto* route = address<const bf1_route>(a[8]);
    const float scale = scale_of(a[9]);
    void* stream = stream_of(a[11]);
    const at::Tensor dq = at::empty_like(q), dk = at::empty_like(k), dv = at::empty_like(v);
    const int32_t batch = static_cast<int32_t>(cu.numel() - 1);
    const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr(), *op = o.data_ptr(), *gp = d_o.data_ptr();
    const auto* lp = static_cast<const float*>(lse.data_ptr());
    const auto* cup = static_cast<const int32_t*>(cu.data_ptr());
    void *wp = ws.data_ptr(), *dqp = dq.data_ptr(), *dkp = dk.data_ptr(), *dvp = dv.data_ptr();
    call([&] {
        return bf1_attn_bwd(qp, kp, vp, op, lp, gp, cup, batch, g.T, max_seqlen, static_cast<int32_t>(g.hq),
                            static_cast<int32_t>(g.hkv), static_cast<int32_t>(g.d), scale, route, wp, dqp, dkp, dvp, stream);
    });
    PyObject *x = THPVariable_Wrap(dq), *y = THPVariable_Wrap(dk), *z = THPVariable_Wrap(dv);
    PyObject* t = x && y && z ? PyTuple_Pack(3, x, y, z) : nullptr;
    Py_XDECREF(x);
    Py_XDECREF(y);
    Py_XDECREF(z);
    return t;
}

// plan_decode(seqlens, page_table, cfg address, plan address, stream*)
PyObject* plan_decode(PyObject* const* a) {
    const at::Tensor &seqlens = tensor(a[0]), &table = tensor(a[1]);
    require(seqlens.is_cuda() && seqlens.scalar_type() == at::kInt && table.scalar_type() == at::kInt && table.dim() == 2,
            "seqlens and the 2-d page_table must be int32 CUDA tensors");
    const auto* cfg = address<const bf1_route_cfg>(a[2]);
    const auto* plan = address<const bf1_decode_plan>(a[3]);
    void* stream = stream_of(a[4]);
    const int32_t batch = static_cast<int32_t>(table.size(0)), pages = static_cast<int32_t>(table.size(1));
    const auto *sp = static_cast<const int32_t*>(seqlens.data_ptr()), *tp = static_cast<const int32_t*>(table.data_ptr());
    call([&] { return bf1_plan_decode(sp, tp, pages, batch, cfg, plan, stream); });
    Py_RETURN_NONE;
}

// decode(q, k_pages, v_pages, seqlens, plan address, workspace, scale*, out*, lse*, stream*)
PyObject* decode(PyObject* const* a) {
    const at::Tensor &q = tensor(a[0]), &k = tensor(a[1]), &v = tensor(a[2]), &seqlens = tensor(a[3]), &ws = tensor(a[5]);
    require(q.dim() == 3 && k.dim() == 4 && k.size(1) == 64 && k.size(3) == q.size(2) && v.sizes() == k.sizes(),
            "q must be [batch, hq, d], k_pages and v_pages [pages, 64, hkv, d]");
    const auto* plan = address<const bf1_decode_plan>(a[4]);
    const float scale = scale_of(a[6]);
    const at::Tensor out = a[7] == Py_None ? at::empty_like(q) : tensor(a[7]);
    const at::Tensor lse = a[8] == Py_None ? lse_like(q, q.size(1), q.size(0)) : tensor(a[8]);
    void* stream = stream_of(a[9]);
    const int32_t batch = q.size(0), hq = q.size(1), d = q.size(2), pages = k.size(0), hkv = k.size(2);
    const void *qp = q.data_ptr(), *kp = k.data_ptr(), *vp = v.data_ptr();
    const auto* sp = static_cast<const int32_t*>(seqlens.data_ptr());
    void *wp = ws.data_ptr(), *op = out.data_ptr();
    auto* lp = static_cast<float*>(lse.data_ptr());
    call([&] { return bf1_decode_fwd(qp, kp, vp, pages, sp, batch, hq, hkv, d, scale, plan, wp, op, lp, stream); });
    return pair(out, lse);
}

// Argument count, C++ and torch exceptions.
template <PyObject* (*F)(PyObject* const*), int kArgs>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != kArgs) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", kArgs, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const PyRaised&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

PyObject* set_error(PyObject*, PyObject* type) {
    Py_INCREF(type);
    Py_XDECREF(g_error);
    g_error = type;
    Py_RETURN_NONE;
}

#define BF1_ENTRY(name, args) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<name, args>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    {"set_error", set_error, METH_O, nullptr},
    BF1_ENTRY(plan_route, 6),
    BF1_ENTRY(forward, 13),
    BF1_ENTRY(backward, 12),
    BF1_ENTRY(plan_decode, 5),
    BF1_ENTRY(decode, 10),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__host() { return PyModule_Create(&g_module); }
