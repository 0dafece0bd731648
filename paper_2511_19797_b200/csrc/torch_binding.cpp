// Native half of the Python binding: checks the tensors of a call, allocates outputs and workspace from PyTorch's
// caching allocator and calls the C-ABI library (include/tvm_attn.h).  Argument marshalling only.
//
// It exists because a call on a small problem is over on the GPU in 6 to 14 us, while the same marshalling written in
// Python (shape, stride and device comparisons, up to seven allocations, a device guard, twenty ctypes arguments) kept
// the host busy for 38 us (forward) and 55 us (backward).  Measured here (2, 2, 64, d 32), one call after another: forward 7.8
// us with the outputs allocated and 6.2 into given ones, backward 15.9 and 14.3, both in turn 22.6 to 24 from machine to
// machine.  The host alone, 20 calls into an empty queue, takes 4.7 us (forward) and 10.4 (backward) into given outputs.
//
// The library's entry points come in as addresses (`bind`), so that this module works with whichever build of the
// library the Python side has loaded.  Functions return the result tensors, or the library's status code as an int
// when it is not TVM_ATTN_OK; the Python side turns that into an exception.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <cstring>
#include <stdexcept>

#include "tvm_attn.h"

namespace {

decltype(&tvm_attn_jvp_fwd) p_fwd = nullptr;
decltype(&tvm_attn_jvp_bwd) p_bwd = nullptr;
decltype(&tvm_attn_jvp_bwd_noalloc) p_bwd_noalloc = nullptr;
decltype(&tvm_attn_jvp_workspace_bytes) p_ws = nullptr;
decltype(&tvm_qk_rmsnorm_jvp_fwd) p_norm_fwd = nullptr;
decltype(&tvm_qk_rmsnorm_jvp_bwd) p_norm_bwd = nullptr;
decltype(&tvm_qk_rmsnorm_jvp_workspace_bytes) p_norm_ws = nullptr;

struct ValueError : std::runtime_error { using std::runtime_error::runtime_error; };

const at::Tensor& tensor(PyObject* o) {
    if (!THPVariable_Check(o)) throw ValueError("expected a torch.Tensor");
    return THPVariable_Unpack(o);
}
// An absent cotangent or an unwanted output (None) is an undefined tensor.
at::Tensor optional_tensor(PyObject* o) { return o == Py_None ? at::Tensor() : tensor(o); }
void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }

// Every tensor of one side shares shape, strides, dtype and device with the side's first tensor.
void check_side(const at::Tensor& ref, const at::Tensor* const* ts, int n) {
    for (int i = 0; i < n; ++i) {
        const at::Tensor& t = *ts[i];
        if (!t.defined()) continue;
        if (t.sizes() != ref.sizes() || t.scalar_type() != ref.scalar_type() || t.device() != ref.device() || t.strides() != ref.strides())
            throw ValueError("all tensors of one side must share shape, strides, dtype and device");
    }
    if (!ref.is_cuda()) throw ValueError("tensors must be CUDA tensors");
}

// {row, head, batch} element strides of a (B, H, rows, d) tensor; zeros for the packed layout.
void side_strides(const at::Tensor& t, int64_t (&st)[3]) {
    if (t.stride(3) != 1 && t.size(3) != 1) throw ValueError("the d elements of a row must be contiguous");
    if (t.is_contiguous()) { st[0] = st[1] = st[2] = 0; return; }
    st[0] = t.stride(2); st[1] = t.stride(1); st[2] = t.stride(0);
}

// Parameters from a query-side tensor q (B, H, M, d) and a key-side tensor k (B, H, N, d).
tvm_attn_params params(const at::Tensor& q, const at::Tensor& k, double scale, uint32_t flags) {
    if (q.dim() != 4) throw ValueError("expected (B, H, rows, d) tensors");
    tvm_attn_params p;
    std::memset(&p, 0, sizeof p);
    if (q.scalar_type() == at::kBFloat16) p.dtype = TVM_ATTN_BF16;
    else if (q.scalar_type() == at::kFloat) p.dtype = TVM_ATTN_FP32;
    else throw ValueError("tensors must be bfloat16 or float32");
    if (k.dim() != 4 || k.size(0) != q.size(0) || k.size(1) != q.size(1) || k.size(3) != q.size(3))
        throw ValueError("query-side and key-side tensors must agree in B, H and d");
    const int64_t B = q.size(0), H = q.size(1), M = q.size(2), N = k.size(2), d = q.size(3);
    if (B > INT32_MAX || H > INT32_MAX || M > INT32_MAX || N > INT32_MAX || d > INT32_MAX) throw ValueError("dimensions must fit 32 bits");
    p.B = (int32_t)B; p.H = (int32_t)H; p.N = (int32_t)N; p.d = (int32_t)d;
    p.M = M == N ? 0 : (int32_t)M;
    p.scale = (float)scale;
    p.flags = flags;
    side_strides(q, p.q_strides);
    side_strides(k, p.k_strides);
    return p;
}

// A new tensor with the shape and the strides of t.
at::Tensor like(const at::Tensor& t) { return at::Tensor(at::detail::empty_strided_cuda(t.sizes(), t.strides(), t.scalar_type(), t.device())); }
at::Tensor packed(at::IntArrayRef sizes, at::ScalarType type, const at::Device& dev) {
    return at::Tensor(at::detail::empty_cuda(sizes, type, dev, std::nullopt));
}

// The stream of a call: the caller's, or PyTorch's current one.
c10::cuda::CUDAStream stream_of(PyObject* o, const at::Device& dev) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream(dev.index());
    return c10::cuda::getStreamFromExternal((cudaStream_t)PyLong_AsVoidPtr(o), dev.index());
}
// Memory allocated here belongs to the current stream.  Where the call runs on another, the allocator has to know: freed, by this
// module (the workspace) or by the caller, it is not given out again before that stream is done with it.  Without a stream
// of the caller's there is nothing to tell (the allocator would look each block up: 0.7 us of the smallest step's 22.5).
void used_on(const at::Tensor* ts, int n, PyObject* callers, c10::cuda::CUDAStream st) {
    if (callers == Py_None) return;
    for (int i = 0; i < n; ++i)
        if (ts[i].defined()) c10::cuda::CUDACachingAllocator::recordStream(ts[i].storage().data_ptr(), st);
}

PyObject* tuple_of(at::Tensor* ts, int n) {
    PyObject* r = PyTuple_New(n);
    if (!r) return nullptr;
    for (int i = 0; i < n; ++i) {
        PyObject* o = THPVariable_Wrap(std::move(ts[i]));
        if (!o) { Py_DECREF(r); return nullptr; }
        PyTuple_SET_ITEM(r, i, o);
    }
    return r;
}
PyObject* same(PyObject* o) { Py_INCREF(o); return o; }

template <typename F>
PyObject* guarded(Py_ssize_t got, Py_ssize_t want, F&& f) {
    if (got != want) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }
    if (!p_fwd) { PyErr_SetString(PyExc_RuntimeError, "the library is not bound"); return nullptr; }
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const ValueError& e) {
        PyErr_SetString(PyExc_ValueError, e.what());
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

template <typename F>
int without_gil(F&& f) {
    PyThreadState* save = PyEval_SaveThread();
    const int rc = f();
    PyEval_RestoreThread(save);
    return rc;
}

// What float(o) and int(o) give, the latter's low 32 bits as flags.
double number(PyObject* o) {
    THPObjectPtr f(PyNumber_Float(o));
    if (!f) throw python_error();
    return PyFloat_AS_DOUBLE(f.get());
}
uint32_t flag_bits(PyObject* o) {
    THPObjectPtr i(PyNumber_Long(o));
    if (!i) throw python_error();
    return (uint32_t)PyLong_AsUnsignedLongLongMask(i.get());
}
// The n entries of `out` as optional tensors.  Returns the list or tuple that they were read from: an iterator has nothing
// left to give after that, so results are made from what is returned here, never from `o` again.  `indexable`: the caller
// gets `o` itself back, so an iterator is refused.
THPObjectPtr entries(PyObject* o, int n, at::Tensor* to, bool indexable) {
    if (indexable && !PySequence_Check(o) && !PyMapping_Check(o)) {   // (a tensor of stacked outputs is a mapping)
        PyErr_Format(PyExc_TypeError, "'%.200s' object is not subscriptable: `out` must be a sequence of tensors", Py_TYPE(o)->tp_name);
        throw python_error();
    }
    THPObjectPtr s(PySequence_Fast(o, "`out` must be a sequence of tensors"));
    if (!s) throw python_error();
    if (PySequence_Fast_GET_SIZE(s.get()) != n) throw ValueError("`out` must hold one entry per output");
    for (int i = 0; i < n; ++i) to[i] = optional_tensor(PySequence_Fast_GET_ITEM(s.get(), i));
    return s;
}

// fwd(Q, K, V, tQ, tK, tV, scale, flags, out | None, stream | None)
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&]() -> PyObject* {
        const at::Tensor &Q = tensor(a[0]), &K = tensor(a[1]), &V = tensor(a[2]), &tQ = tensor(a[3]), &tK = tensor(a[4]), &tV = tensor(a[5]);
        const bool given = a[8] != Py_None;
        at::Tensor o[4];
        THPObjectPtr outs;
        if (given) outs = entries(a[8], 4, o, false);
        const at::Tensor* qs[] = {&tQ, &o[0], &o[1]};
        const at::Tensor* ks[] = {&V, &tK, &tV};
        check_side(Q, qs, 3);
        check_side(K, ks, 3);
        const tvm_attn_params p = params(Q, K, number(a[6]), flag_bits(a[7]));
        if (!given) {
            o[0] = like(Q); o[1] = like(Q);
            o[2] = packed(Q.sizes().slice(0, 3), at::kFloat, Q.device());
            o[3] = packed(Q.sizes().slice(0, 3), at::kFloat, Q.device());
        }
        const c10::cuda::CUDAGuard guard(Q.device());
        const c10::cuda::CUDAStream st = stream_of(a[9], Q.device());
        if (!given) used_on(o, 4, a[9], st);
        const int rc = without_gil([&] {
            return p_fwd(&p, ptr(Q), ptr(K), ptr(V), ptr(tQ), ptr(tK), ptr(tV), ptr(o[0]), ptr(o[1]), (float*)ptr(o[2]), (float*)ptr(o[3]),
                         nullptr, 0, st.stream());
        });
        if (rc != TVM_ATTN_OK) return PyLong_FromLong(rc);
        return given ? PySequence_Tuple(outs.get()) : tuple_of(o, 4);
    });
}

// bwd(Q, K, V, tQ, tK, tV, O, tO, lse, mu, dO | None, dtO | None, scale, flags, out | None, workspace | None, stream | None,
// noalloc): with noalloc, `out` is required and the workspace is the library's own.
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 18, [&]() -> PyObject* {
        const at::Tensor &Q = tensor(a[0]), &K = tensor(a[1]), &V = tensor(a[2]), &tQ = tensor(a[3]), &tK = tensor(a[4]), &tV = tensor(a[5]);
        const at::Tensor &O = tensor(a[6]), &tO = tensor(a[7]), &lse = tensor(a[8]), &mu = tensor(a[9]);
        const at::Tensor dO = optional_tensor(a[10]), dtO = optional_tensor(a[11]);
        const tvm_attn_params p = params(Q, K, number(a[12]), flag_bits(a[13]));
        const bool given = a[14] != Py_None, noalloc = a[17] == Py_True;
        at::Tensor o[6];
        THPObjectPtr outs;
        if (given) outs = entries(a[14], 6, o, true);
        else if (noalloc) throw ValueError("`out` must hold the six gradients");
        const at::Tensor* qs[] = {&tQ, &O, &tO, &dO, &dtO, &o[0], &o[3]};
        const at::Tensor* ks[] = {&V, &tK, &tV, &o[1], &o[2], &o[4], &o[5]};
        check_side(Q, qs, 7);
        check_side(K, ks, 7);
        if (!given)
            for (int i = 0; i < 6; ++i) o[i] = like(i % 3 == 0 ? Q : K);
        at::Tensor ws = noalloc ? at::Tensor() : optional_tensor(a[15]);
        const bool own_ws = !noalloc && !ws.defined();
        if (own_ws) {
            const int64_t need = (int64_t)p_ws(&p, 1);
            ws = packed({need > 16 ? need : 16}, at::kByte, Q.device());
        }
        const c10::cuda::CUDAGuard guard(Q.device());
        const c10::cuda::CUDAStream st = stream_of(a[16], Q.device());
        if (!given) used_on(o, 6, a[16], st);
        if (own_ws) used_on(&ws, 1, a[16], st);
        const int rc = without_gil([&] {
            if (noalloc)
                return p_bwd_noalloc(&p, ptr(Q), ptr(K), ptr(V), ptr(tQ), ptr(tK), ptr(tV), ptr(O), ptr(tO), (float*)ptr(lse), (float*)ptr(mu),
                                     ptr(dO), ptr(dtO), ptr(o[0]), ptr(o[1]), ptr(o[2]), ptr(o[3]), ptr(o[4]), ptr(o[5]), st.stream());
            return p_bwd(&p, ptr(Q), ptr(K), ptr(V), ptr(tQ), ptr(tK), ptr(tV), ptr(O), ptr(tO), (float*)ptr(lse), (float*)ptr(mu), ptr(dO),
                         ptr(dtO), ptr(o[0]), ptr(o[1]), ptr(o[2]), ptr(o[3]), ptr(o[4]), ptr(o[5]), ptr(ws), (size_t)ws.numel(), st.stream());
        });
        if (rc != TVM_ATTN_OK) return PyLong_FromLong(rc);
        return given ? (noalloc ? PySequence_Tuple(outs.get()) : same(a[14])) : tuple_of(o, 6);
    });
}

void check_scale(const at::Tensor& g, const at::Tensor& ref) {
    if (g.scalar_type() != at::kFloat || g.dim() != 1 || g.numel() != ref.size(-1) || g.device() != ref.device() || !g.is_contiguous())
        throw ValueError("a scale must be a contiguous float32 CUDA vector of d elements");
}

// norm_fwd(Q, tQ, K, tK, gQ, gK, eps, stream | None)
PyObject* norm_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 8, [&]() -> PyObject* {
        const at::Tensor &Q = tensor(a[0]), &tQ = tensor(a[1]), &K = tensor(a[2]), &tK = tensor(a[3]), &gQ = tensor(a[4]), &gK = tensor(a[5]);
        const at::Tensor *qs[] = {&tQ}, *ks[] = {&tK};
        check_side(Q, qs, 1);
        check_side(K, ks, 1);
        check_scale(gQ, Q);
        check_scale(gK, Q);
        const tvm_attn_params p = params(Q, K, 0.0, 0);
        at::Tensor o[4] = {like(Q), like(Q), like(K), like(K)};
        const c10::cuda::CUDAGuard guard(Q.device());
        const float eps = (float)number(a[6]);
        const c10::cuda::CUDAStream st = stream_of(a[7], Q.device());
        used_on(o, 4, a[7], st);
        const int rc = without_gil([&] {
            return p_norm_fwd(&p, eps, ptr(Q), ptr(tQ), ptr(K), ptr(tK), (float*)ptr(gQ), (float*)ptr(gK), ptr(o[0]), ptr(o[1]), ptr(o[2]), ptr(o[3]), st.stream());
        });
        return rc != TVM_ATTN_OK ? PyLong_FromLong(rc) : tuple_of(o, 4);
    });
}

// norm_bwd(Q, tQ, K, tK, gQ, gK, dQn, dtQn, dKn, dtKn, eps, workspace | None, stream | None)
PyObject* norm_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 13, [&]() -> PyObject* {
        const at::Tensor &Q = tensor(a[0]), &tQ = tensor(a[1]), &K = tensor(a[2]), &tK = tensor(a[3]), &gQ = tensor(a[4]), &gK = tensor(a[5]);
        const at::Tensor &dQn = tensor(a[6]), &dtQn = tensor(a[7]), &dKn = tensor(a[8]), &dtKn = tensor(a[9]);
        const at::Tensor *qs[] = {&tQ, &dQn, &dtQn}, *ks[] = {&tK, &dKn, &dtKn};
        check_side(Q, qs, 3);
        check_side(K, ks, 3);
        check_scale(gQ, Q);
        check_scale(gK, Q);
        const tvm_attn_params p = params(Q, K, 0.0, 0);
        at::Tensor ws = optional_tensor(a[11]);
        const bool own_ws = !ws.defined();
        if (own_ws) {
            const int64_t need = (int64_t)p_norm_ws(&p);
            ws = packed({need > 16 ? need : 16}, at::kByte, Q.device());
        }
        at::Tensor o[6] = {like(Q), like(Q), like(K), like(K), like(gQ), like(gK)};
        const c10::cuda::CUDAGuard guard(Q.device());
        const float eps = (float)number(a[10]);
        const c10::cuda::CUDAStream st = stream_of(a[12], Q.device());
        used_on(o, 6, a[12], st);
        if (own_ws) used_on(&ws, 1, a[12], st);
        const int rc = without_gil([&] {
            return p_norm_bwd(&p, eps, ptr(Q), ptr(tQ), ptr(K), ptr(tK), (float*)ptr(gQ), (float*)ptr(gK), ptr(dQn), ptr(dtQn), ptr(dKn), ptr(dtKn),
                              ptr(o[0]), ptr(o[1]), ptr(o[2]), ptr(o[3]), (float*)ptr(o[4]), (float*)ptr(o[5]), ptr(ws), (size_t)ws.numel(), st.stream());
        });
        return rc != TVM_ATTN_OK ? PyLong_FromLong(rc) : tuple_of(o, 6);
    });
}

// bind(addresses of tvm_attn_jvp_fwd, _bwd, _bwd_noalloc, _workspace_bytes, tvm_qk_rmsnorm_jvp_fwd, _bwd, _workspace_bytes)
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 7) { PyErr_SetString(PyExc_TypeError, "seven addresses are needed"); return nullptr; }
    void* f[7];
    for (int i = 0; i < 7; ++i) {
        f[i] = PyLong_AsVoidPtr(a[i]);
        if (!f[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "a null address");
            return nullptr;
        }
    }
    p_fwd = (decltype(p_fwd))f[0]; p_bwd = (decltype(p_bwd))f[1]; p_bwd_noalloc = (decltype(p_bwd_noalloc))f[2]; p_ws = (decltype(p_ws))f[3];
    p_norm_fwd = (decltype(p_norm_fwd))f[4]; p_norm_bwd = (decltype(p_norm_bwd))f[5]; p_norm_ws = (decltype(p_norm_ws))f[6];
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"bind", (PyCFunction)(void*)bind, METH_FASTCALL, nullptr},
                         {"fwd", (PyCFunction)(void*)fwd, METH_FASTCALL, nullptr},
                         {"bwd", (PyCFunction)(void*)bwd, METH_FASTCALL, nullptr},
                         {"norm_fwd", (PyCFunction)(void*)norm_fwd, METH_FASTCALL, nullptr},
                         {"norm_bwd", (PyCFunction)(void*)norm_bwd, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tvm_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tvm_binding() { return PyModule_Create(&module); }
