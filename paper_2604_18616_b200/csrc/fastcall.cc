// The ordinary case of the binding's calls, in C++: plain CUDA tensors, results allocated here, the current stream.
//
// A small call is bound by the host.  In Python its checks, two allocations, the marshalling of 14 arguments through ctypes
// and the launch take longer than the kernel (a call of 128 tokens 10.6 us there, 5.6 here; split-KV 11.0 and 5.5, a product
// of 128 x 128 x 256 7.6 and 4.1, calls back to back).  Each function returns None, having done nothing, when anything
// about the call is out of the ordinary (types, shapes, strides, devices, dispatch modes): the Python wrapper then takes its
// own way, which knows every check and message.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>

#include <climits>
#include <cstdint>

namespace {

typedef int (*AttnFn)(const void *, const void *, const void *, void *, float *, int, int, int, int, int, int, int, float, void *);
typedef int (*SplitFn)(const void *, const void *, const void *, void *, float *, int, int, int, int, int, int, int, float, int,
                       void *, size_t, void *);
typedef int (*GemmFn)(const void *, const void *, void *, int, int, int, void *);

AttnFn attn_fn = nullptr;
SplitFn splitkv_fn = nullptr;
GemmFn gemm_fn[2] = {nullptr, nullptr};  // tn, nn

PyObject *bind(PyObject *, PyObject *args) {
    unsigned long long a, s, t, n;
    if (!PyArg_ParseTuple(args, "KKKK", &a, &s, &t, &n)) return nullptr;
    attn_fn = reinterpret_cast<AttnFn>(static_cast<uintptr_t>(a));
    splitkv_fn = reinterpret_cast<SplitFn>(static_cast<uintptr_t>(s));
    gemm_fn[0] = reinterpret_cast<GemmFn>(static_cast<uintptr_t>(t));
    gemm_fn[1] = reinterpret_cast<GemmFn>(static_cast<uintptr_t>(n));
    Py_RETURN_NONE;
}

// A plain contiguous bf16 tensor on a CUDA device, with `dims` dimensions that fit an int.
const at::Tensor *plain(PyObject *obj, int dims) {
    if (!THPVariable_CheckExact(obj)) return nullptr;
    const at::Tensor &t = THPVariable_Unpack(obj);
    if (!t.defined() || !t.is_cuda() || t.scalar_type() != at::kBFloat16 || t.dim() != dims || t.layout() != at::kStrided ||
        !t.has_storage() || !t.is_contiguous())
        return nullptr;
    for (int i = 0; i < dims; ++i)
        if (t.size(i) > INT_MAX) return nullptr;
    return &t;
}

bool modes_active() {
    return c10::impl::TorchDispatchModeTLS::any_modes_set() || at::impl::PythonTorchFunctionTLS::stack_len() > 0;
}

// The scale argument: None stands for D ** -0.5.  False: not a plain number.
bool read_scale(PyObject *obj, int64_t D, float &scale) {
    if (obj == Py_None) {
        PyObject *d = PyLong_FromLongLong(D), *e = PyFloat_FromDouble(-0.5);
        PyObject *r = (d && e) ? PyNumber_Power(d, e, Py_None) : nullptr;  // what the Python wrapper computes, to the bit
        const bool ok = r && PyFloat_CheckExact(r);
        if (ok) scale = static_cast<float>(PyFloat_AS_DOUBLE(r));
        Py_XDECREF(d);
        Py_XDECREF(e);
        Py_XDECREF(r);
        PyErr_Clear();
        return ok;
    }
    if (!PyFloat_CheckExact(obj)) return false;
    scale = static_cast<float>(PyFloat_AS_DOUBLE(obj));
    return true;
}

struct Qkv {
    const at::Tensor *q, *k, *v;
    int B, H, Hkv, Sq, Sk, D, device;
};
bool read_qkv(PyObject *const *args, Qkv &x) {
    x.q = plain(args[0], 4);
    x.k = x.q ? plain(args[1], 4) : nullptr;
    x.v = x.k ? plain(args[2], 4) : nullptr;
    if (!x.v) return false;
    x.device = x.q->get_device();
    if (x.device != c10::cuda::current_device() || x.k->get_device() != x.device || x.v->get_device() != x.device) return false;
    const auto qs = x.q->sizes(), ks = x.k->sizes();
    if (x.v->sizes() != ks || ks[0] != qs[0] || ks[3] != qs[3]) return false;
    x.B = int(qs[0]);
    x.H = int(qs[1]);
    x.Sq = int(qs[2]);
    x.D = int(qs[3]);
    x.Hkv = int(ks[1]);
    x.Sk = int(ks[2]);
    return true;
}

// The result, or the library's status where that is not AVE_OK.
PyObject *status_or(int st, PyObject *result) {
    if (st == 0 || !result) return result;
    Py_DECREF(result);
    return PyLong_FromLong(st);
}

PyObject *pair_of(at::Tensor &&a, at::Tensor &&b) {
    PyObject *x = THPVariable_Wrap(std::move(a));
    PyObject *y = x ? THPVariable_Wrap(std::move(b)) : nullptr;
    PyObject *r = y ? PyTuple_New(2) : nullptr;
    if (!r) {
        Py_XDECREF(x);
        Py_XDECREF(y);
        return nullptr;
    }
    PyTuple_SET_ITEM(r, 0, x);
    PyTuple_SET_ITEM(r, 1, y);
    return r;
}

// (q, k, v, causal, scale) -> (o, lse), or the library's status as an int, or None
PyObject *attn_fwd(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Qkv x;
    float scale;
    if (n != 5 || !attn_fn || modes_active() || !read_qkv(args, x) || !read_scale(args[4], x.D, scale)) Py_RETURN_NONE;
    const int causal = PyObject_IsTrue(args[3]);
    if (causal < 0) return nullptr;
    at::Tensor o = at::empty_like(*x.q);
    at::Tensor lse = at::empty({x.B, x.H, x.Sq}, x.q->options().dtype(at::kFloat));
    const void *q = x.q->data_ptr(), *k = x.k->data_ptr(), *v = x.v->data_ptr();
    void *op = o.data_ptr();
    float *lp = static_cast<float *>(lse.data_ptr());
    void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(x.device)).stream();
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = attn_fn(q, k, v, op, lp, x.B, x.H, x.Hkv, x.Sq, x.Sk, x.D, causal, scale, stream);
    Py_END_ALLOW_THREADS
    return status_or(st, pair_of(std::move(o), std::move(lse)));
    END_HANDLE_TH_ERRORS
}

// (q, k, v, n_splits, workspace, causal, scale) likewise
PyObject *attn_fwd_splitkv(PyObject *, PyObject *const *args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Qkv x;
    float scale;
    if (n != 7 || !splitkv_fn || modes_active() || !read_qkv(args, x) || !read_scale(args[6], x.D, scale)) Py_RETURN_NONE;
    if (!PyLong_CheckExact(args[3]) || !THPVariable_CheckExact(args[4])) Py_RETURN_NONE;
    int overflow = 0;
    const long splits = PyLong_AsLongAndOverflow(args[3], &overflow);
    const at::Tensor &ws = THPVariable_Unpack(args[4]);
    if (overflow || splits > INT_MAX || splits < INT_MIN || !ws.defined() || !ws.is_cuda() || ws.get_device() != x.device ||
        ws.scalar_type() != at::kByte || !ws.has_storage())
        Py_RETURN_NONE;
    const int causal = PyObject_IsTrue(args[5]);
    if (causal < 0) return nullptr;
    at::Tensor o = at::empty_like(*x.q);
    at::Tensor lse = at::empty({x.B, x.H, x.Sq}, x.q->options().dtype(at::kFloat));
    const void *q = x.q->data_ptr(), *k = x.k->data_ptr(), *v = x.v->data_ptr();
    void *op = o.data_ptr(), *wp = ws.data_ptr();
    float *lp = static_cast<float *>(lse.data_ptr());
    const size_t bytes = static_cast<size_t>(ws.numel());
    void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(x.device)).stream();
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = splitkv_fn(q, k, v, op, lp, x.B, x.H, x.Hkv, x.Sq, x.Sk, x.D, causal, scale, int(splits), wp, bytes, stream);
    Py_END_ALLOW_THREADS
    return status_or(st, pair_of(std::move(o), std::move(lse)));
    END_HANDLE_TH_ERRORS
}

// (a, b) -> c likewise
PyObject *gemm(PyObject *const *args, Py_ssize_t n, int nn) {
    HANDLE_TH_ERRORS
    if (n != 2 || !gemm_fn[nn] || modes_active()) Py_RETURN_NONE;
    const at::Tensor *a = plain(args[0], 2), *b = a ? plain(args[1], 2) : nullptr;
    if (!b || b->size(nn ? 0 : 1) != a->size(1)) Py_RETURN_NONE;
    const int device = a->get_device();
    if (device != c10::cuda::current_device() || b->get_device() != device) Py_RETURN_NONE;
    const int M = int(a->size(0)), K = int(a->size(1)), N = int(b->size(nn ? 1 : 0));
    at::Tensor c = at::empty({M, N}, a->options());
    const void *ap = a->data_ptr(), *bp = b->data_ptr();
    void *cp = c.data_ptr();
    void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device)).stream();
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = gemm_fn[nn](ap, bp, cp, M, N, K, stream);
    Py_END_ALLOW_THREADS
    return status_or(st, THPVariable_Wrap(std::move(c)));
    END_HANDLE_TH_ERRORS
}
PyObject *gemm_tn(PyObject *, PyObject *const *args, Py_ssize_t n) { return gemm(args, n, 0); }
PyObject *gemm_nn(PyObject *, PyObject *const *args, Py_ssize_t n) { return gemm(args, n, 1); }

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, nullptr},
                         {"attn_fwd", FAST(attn_fwd)},
                         {"attn_fwd_splitkv", FAST(attn_fwd_splitkv)},
                         {"gemm_tn", FAST(gemm_tn)},
                         {"gemm_nn", FAST(gemm_nn)},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&module); }
