// Native marshalling of the torch binding (gka.py): tensors in, one C-ABI call, tensors out.  It only checks and fills the
// descriptor; the library itself (libgka.so) knows no torch types.
//
// A call from Python spends its time before the first launch: with the checks and the descriptor in Python a decode step
// took 17 us of host time and a forward 33 to 40, more than the kernels of a small call.  Every function takes its
// arguments by position and returns the result, the library's status (an int) if the call failed, or None if an argument
// does not fit as it is; the Python wrapper then says what is wrong, or converts it and calls once more.
#define PY_SSIZE_T_CLEAN
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/gka.h"

namespace {

using at::Tensor;

struct Bad {};      // thrown where an argument does not fit

const Tensor *tensor(PyObject *o) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) throw Bad();
    return &THPVariable_Unpack(o);
}
const Tensor &need(PyObject *o) {
    const Tensor *t = tensor(o);
    if (!t) throw Bad();
    return *t;
}
long long integer(PyObject *o) {
    if (!PyLong_Check(o)) throw Bad();
    int over = 0;
    const long long v = PyLong_AsLongLongAndOverflow(o, &over);
    if (over) throw Bad();
    return v;
}
int small_integer(PyObject *o) {
    const long long v = integer(o);
    if (v < INT_MIN || v > INT_MAX) throw Bad();
    return (int)v;
}
void *address(PyObject *o) { return o == Py_None ? nullptr : reinterpret_cast<void *>(static_cast<uintptr_t>(integer(o))); }

// q and the tensors of its type and shape; the per-token scalars beside them
struct Tokens {
    const Tensor &q;
    bool cuda;
    explicit Tokens(PyObject *o, int dim, bool on_cuda = true) : q(need(o)), cuda(on_cuda) {
        if (q.dim() != dim || (q.scalar_type() != at::kFloat && q.scalar_type() != at::kBFloat16)) throw Bad();
        place(q);
    }
    void place(const Tensor &t) const {
        if (t.is_cuda() != cuda || !t.is_contiguous()) throw Bad();
    }
    void *vector(PyObject *o, bool optional = false) const {
        const Tensor *t = tensor(o);
        if (!t && optional) return nullptr;
        if (!t || t->scalar_type() != q.scalar_type() || t->sizes() != q.sizes()) throw Bad();
        place(*t);
        return t->data_ptr();
    }
    const float *scalar(PyObject *o, bool optional = false) const {
        const Tensor *t = tensor(o);
        if (!t && optional) return nullptr;
        if (!t || t->scalar_type() != at::kFloat || t->sizes() != q.sizes().slice(0, q.dim() - 1)) throw Bad();
        place(*t);
        return static_cast<const float *>(t->data_ptr());
    }
    float *state(PyObject *o, int64_t n, int64_t heads, int64_t d, bool optional = false) const {
        const Tensor *t = tensor(o);
        if (!t && optional) return nullptr;
        if (!t || t->scalar_type() != at::kFloat || t->dim() != 3 || t->size(0) != n || t->size(1) != heads || t->size(2) != 2 * d * d)
            throw Bad();
        place(*t);
        return static_cast<float *>(t->data_ptr());
    }
};
int *status_word(PyObject *o) {
    const Tensor *t = tensor(o);
    if (!t) return nullptr;
    if (t->scalar_type() != at::kInt || t->dim() != 1 || t->size(0) != 1 || !t->is_cuda()) throw Bad();
    return static_cast<int *>(t->data_ptr());
}
const Tensor &bytes(PyObject *o) {
    const Tensor &t = need(o);
    if (t.scalar_type() != at::kByte || !t.is_cuda() || !t.is_contiguous()) throw Bad();
    return t;
}

gka_desc describe(const Tensor &q, int64_t B, int64_t T, int precision, long long flags, PyObject *stream, int device) {
    gka_desc d = {};
    const int64_t heads = q.size(q.dim() - 2), dim = q.size(q.dim() - 1);
    if (B > INT_MAX || T > INT_MAX || heads > INT_MAX || dim > INT_MAX || flags < 0 || flags > UINT_MAX) throw Bad();
    d.B = (int)B;
    d.T = (int)T;
    d.heads = (int)heads;
    d.d_k = d.d_v = (int)dim;
    d.io_dtype = q.scalar_type() == at::kFloat ? GKA_F32 : GKA_BF16;
    d.precision = precision;
    d.flags = (unsigned)flags;
    d.stream = stream == Py_None ? static_cast<void *>(c10::cuda::getCurrentCUDAStream(device).stream()) : address(stream);
    return d;
}
// Where the caller names a stream, what a call allocates (scratch above all, which is given back when the call returns, with its
// kernels still to run) belongs to that stream: a block of the current stream's pool could go to other work of the current
// stream at once.
struct OnStream {
    c10::cuda::OptionalCUDAStreamGuard guard;
    OnStream(PyObject *stream, const gka_desc &d, int device) {
        if (stream == Py_None) return;
        const cudaStream_t s = static_cast<cudaStream_t>(d.stream);
        guard.reset_stream(s == nullptr || s == cudaStreamLegacy ? c10::cuda::getDefaultCUDAStream(device)
                                                                 : c10::cuda::getStreamFromExternal(s, device));
    }
};
void events(gka_desc &d, PyObject *o) {
    if (o == Py_None) return;
    if (!PyTuple_Check(o) || PyTuple_GET_SIZE(o) != 2) throw Bad();
    d.profile_start = address(PyTuple_GET_ITEM(o, 0));
    d.profile_stop = address(PyTuple_GET_ITEM(o, 1));
}
// The workspace given by the caller, or one of this call
Tensor workspace(gka_desc &d, PyObject *o, int chunk, const Tensor &q) {
    Tensor w;
    if (o == Py_None) {
        const size_t n = gka_fwd_workspace_bytes(&d, chunk);
        if (!n) throw Bad();
        w = at::empty({(int64_t)n}, q.options().dtype(at::kByte));
    } else {
        w = bytes(o);
    }
    d.workspace = w.data_ptr();
    d.workspace_bytes = (size_t)w.numel();
    return w;
}
Tensor like(PyObject *given, const Tensor &model) { return given == Py_None ? at::empty_like(model) : THPVariable_Unpack(given); }

template <typename F> PyObject *guarded(Py_ssize_t n, Py_ssize_t want, F f) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
        return nullptr;
    }
    try {
        return f();
    } catch (const Bad &) {
        Py_RETURN_NONE;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename F> int unlocked(F f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return rc;
}

// state, q, k, v, gate, lam, n_iter, out, flags, device_status, stream, profile_events, beta, alpha
template <int DIM> PyObject *decode(PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 14, [&]() -> PyObject * {
        const Tokens tk(a[1], DIM);
        const int64_t N = tk.q.size(0), T = DIM == 4 ? tk.q.size(1) : 1, heads = tk.q.size(DIM - 2), dim = tk.q.size(DIM - 1);
        void *const k = tk.vector(a[2]), *const v = tk.vector(a[3]);
        const float *const gate = tk.scalar(a[4]), *const lam = tk.scalar(a[5]);
        float *const state = tk.state(a[0], N, heads, dim);
        const int n_iter = small_integer(a[6]);
        tk.vector(a[7], true);
        gka_desc d = describe(tk.q, N, T, GKA_PREC_NATIVE, integer(a[8]), a[10], tk.q.get_device());
        d.device_status = status_word(a[9]);
        events(d, a[11]);
        d.beta = tk.scalar(a[12], true);
        d.alpha = tk.scalar(a[13], true);
        const OnStream on(a[10], d, tk.q.get_device());
        Tensor out = like(a[7], tk.q);
        const int rc = unlocked([&] {
            return DIM == 4 ? gka_decode_tokens(&d, state, tk.q.data_ptr(), k, v, gate, lam, n_iter, out.data_ptr())
                            : gka_decode_step(&d, state, tk.q.data_ptr(), k, v, gate, lam, n_iter, out.data_ptr());
        });
        return rc == GKA_OK ? THPVariable_Wrap(std::move(out)) : PyLong_FromLong(rc);
    });
}
PyObject *decode_step(PyObject *, PyObject *const *a, Py_ssize_t n) { return decode<3>(a, n); }
PyObject *decode_tokens(PyObject *, PyObject *const *a, Py_ssize_t n) { return decode<4>(a, n); }

// q, k, v, gate, lam, n_iter, chunk, out, state_out, state_in, workspace, precision, flags, fro_out, device_status, stream,
// profile_events, beta, alpha
PyObject *fwd_chunked(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 19, [&]() -> PyObject * {
        const Tokens tk(a[0], 4);
        const int64_t B = tk.q.size(0), T = tk.q.size(1), heads = tk.q.size(2), dim = tk.q.size(3);
        void *const k = tk.vector(a[1]), *const v = tk.vector(a[2]);
        const float *const gate = tk.scalar(a[3]), *const lam = tk.scalar(a[4]);
        const int n_iter = small_integer(a[5]), chunk = small_integer(a[6]);
        tk.vector(a[7], true);
        tk.state(a[8], B, heads, dim, true);
        gka_desc d = describe(tk.q, B, T, small_integer(a[11]), integer(a[12]), a[15], tk.q.get_device());
        d.state_in = tk.state(a[9], B, heads, dim, true);
        d.fro_out = const_cast<float *>(tk.scalar(a[13], true));
        d.device_status = status_word(a[14]);
        events(d, a[16]);
        d.beta = tk.scalar(a[17], true);
        d.alpha = tk.scalar(a[18], true);
        const OnStream on(a[15], d, tk.q.get_device());
        const Tensor ws = workspace(d, a[10], chunk, tk.q);
        Tensor out = like(a[7], tk.q);
        Tensor state_out = a[8] == Py_None ? at::empty({B, heads, 2 * dim * dim}, tk.q.options().dtype(at::kFloat)) : THPVariable_Unpack(a[8]);
        const int rc = unlocked([&] {
            return gka_fwd_chunked(&d, tk.q.data_ptr(), k, v, gate, lam, n_iter, chunk, out.data_ptr(), static_cast<float *>(state_out.data_ptr()));
        });
        if (rc != GKA_OK) return PyLong_FromLong(rc);
        PyObject *const r = PyTuple_New(2);
        PyTuple_SET_ITEM(r, 0, THPVariable_Wrap(std::move(out)));
        PyTuple_SET_ITEM(r, 1, THPVariable_Wrap(std::move(state_out)));
        return r;
    });
}

// rhs, k, gate, lam, n_iter, chunk, out, state_in, workspace, precision, flags, device_status, stream, beta
PyObject *solve_chunked(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 14, [&]() -> PyObject * {
        const Tokens tk(a[0], 4);
        const int64_t B = tk.q.size(0), T = tk.q.size(1), heads = tk.q.size(2), dim = tk.q.size(3);
        void *const k = tk.vector(a[1]);
        const float *const gate = tk.scalar(a[2]), *const lam = tk.scalar(a[3]);
        const int n_iter = small_integer(a[4]), chunk = small_integer(a[5]);
        tk.vector(a[6], true);
        gka_desc d = describe(tk.q, B, T, small_integer(a[9]), integer(a[10]), a[12], tk.q.get_device());
        d.state_in = tk.state(a[7], B, heads, dim, true);
        d.device_status = status_word(a[11]);
        d.beta = tk.scalar(a[13], true);
        const OnStream on(a[12], d, tk.q.get_device());
        const Tensor ws = workspace(d, a[8], chunk, tk.q);
        Tensor out = like(a[6], tk.q);
        const int rc = unlocked([&] { return gka_solve_chunked(&d, tk.q.data_ptr(), k, gate, lam, n_iter, chunk, out.data_ptr()); });
        return rc == GKA_OK ? THPVariable_Wrap(std::move(out)) : PyLong_FromLong(rc);
    });
}

// q, k, v, gate, lam, n_iter, chunk, out, state_out, staging, workspace, precision, flags, stream, device_status
PyObject *fwd_chunked_host(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded(n, 15, [&]() -> PyObject * {
        const Tokens tk(a[0], 4, false);
        const int64_t B = tk.q.size(0), T = tk.q.size(1), heads = tk.q.size(2), dim = tk.q.size(3);
        void *const k = tk.vector(a[1]), *const v = tk.vector(a[2]), *const out = tk.vector(a[7]);
        const float *const gate = tk.scalar(a[3]), *const lam = tk.scalar(a[4]);
        const int n_iter = small_integer(a[5]), chunk = small_integer(a[6]);
        float *const state_out = tk.state(a[8], B, heads, dim, true);
        const Tensor &staging = bytes(a[9]), &ws = bytes(a[10]);
        gka_desc d = describe(tk.q, B, T, small_integer(a[11]), integer(a[12]), a[13], staging.get_device());
        if ((size_t)staging.numel() < gka_fwd_host_staging_bytes(&d)) throw Bad();
        d.device_status = status_word(a[14]);
        d.workspace = ws.data_ptr();
        d.workspace_bytes = (size_t)ws.numel();
        const int rc = unlocked([&] {
            return gka_fwd_chunked_host(&d, staging.data_ptr(), tk.q.data_ptr(), k, v, gate, lam, n_iter, chunk, out, state_out);
        });
        return PyLong_FromLong(rc);
    });
}

PyMethodDef methods[] = {
    {"decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL, nullptr},
    {"decode_tokens", (PyCFunction)(void (*)(void))decode_tokens, METH_FASTCALL, nullptr},
    {"fwd_chunked", (PyCFunction)(void (*)(void))fwd_chunked, METH_FASTCALL, nullptr},
    {"solve_chunked", (PyCFunction)(void (*)(void))solve_chunked, METH_FASTCALL, nullptr},
    {"fwd_chunked_host", (PyCFunction)(void (*)(void))fwd_chunked_host, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_gka_torch", "Native marshalling of the torch binding", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__gka_torch(void) { return PyModule_Create(&module); }
