// The per-call path of the Python binding (attention forward, backward, cell mean): argument checks, output
// allocation and the call into libmate, in one native function each.  A call costs the host 4.5 us (forward,
// cell mean: two allocations, one launch) or 7.5 us (backward: three allocations, two launches); the same steps
// through ctypes and torch's Python layer took 20 to 30 us, more than the kernels of a small table.
//
// The library is not linked: api.py loads it (MATE_LIB may name another build) and hands over the addresses.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cmath>
#include <optional>

#include "mate.h"

namespace {

struct Library {
    decltype(&mate_attn_workspace_bytes) workspace_bytes = nullptr;
    decltype(&mate_attn_fwd) fwd = nullptr;
    decltype(&mate_attn_bwd) bwd = nullptr;
    decltype(&mate_cell_mean) cell_mean = nullptr;
} lib;
PyObject *mate_error = nullptr;  // exception class, called with (status, where)

// What a call needs to know of a plan; lives in a capsule of the Python object.
struct PlanInfo {
    const mate_plan_t *handle;
    int64_t B, N, H, T;  // T: total tokens of a packed plan, -1 otherwise
    int64_t n_rows, n_cols;  // ids per view (cell mean)
    c10::DeviceIndex device;
    at::Tensor ws[2];    // workspaces of forward and backward, kept from call to call
    c10::StreamId ws_stream[2];  // the streams they were allocated on
};
const char kCapsule[] = "mate_plan_info";

struct Raised {};  // a Python exception is set

// Other Python threads run while a call may wait: the allocator for memory to become free, a launch for room in
// the queue, the first use of a plan on another stream for its upload.
struct NoGil {
    PyThreadState *state = PyEval_SaveThread();
    NoGil() = default;
    NoGil(const NoGil &) = delete;
    ~NoGil() { PyEval_RestoreThread(state); }
};

[[noreturn]] void fail(PyObject *type, const char *msg) {
    PyErr_SetString(type, msg);
    throw Raised();
}
[[noreturn]] void fail_named(PyObject *type, const char *format, const char *name) {
    PyErr_Format(type, format, name);
    throw Raised();
}
void check(int status, const char *where) {
    if (status == MATE_OK) return;
    PyObject *e = PyObject_CallFunction(mate_error, "is", status, where);
    if (e) {
        PyErr_SetObject(mate_error, e);
        Py_DECREF(e);
    }
    throw Raised();
}

const at::Tensor &tensor(PyObject *o, const char *name) {
    if (!THPVariable_Check(o)) fail_named(PyExc_ValueError, "%s must be a contiguous CUDA tensor", name);
    return THPVariable_Unpack(o);
}
void *dev(const at::Tensor &t, const char *name) {
    if (!t.is_cuda() || !t.is_contiguous()) fail_named(PyExc_ValueError, "%s must be a contiguous CUDA tensor", name);
    return t.data_ptr();
}
int dtype_code(const at::Tensor &t) {
    if (t.scalar_type() == at::kBFloat16) return MATE_BF16;
    if (t.scalar_type() == at::kFloat) return MATE_F32;
    PyErr_Format(PyExc_TypeError, "libmate takes bfloat16 or float32 tensors, got %s", c10::toString(t.scalar_type()));
    throw Raised();
}
PlanInfo &plan_info(PyObject *o) {
    void *p = PyCapsule_GetPointer(o, kCapsule);
    if (!p) throw Raised();
    return *static_cast<PlanInfo *>(p);
}
// Checks a tensor's shape against the plan; returns d.
int64_t split(const PlanInfo &pi, const at::Tensor &q) {
    if (pi.T >= 0) {
        if (q.dim() != 3 || q.size(0) != pi.H || q.size(1) != pi.T) fail(PyExc_ValueError, "a packed plan takes [H, T, d] tensors");
        return q.size(2);
    }
    if (q.dim() != 4 || q.size(0) != pi.B || q.size(1) != pi.H || q.size(2) != pi.N)
        fail(PyExc_ValueError, "tensor shapes do not match the plan");
    return q.size(3);
}
float scale_of(PyObject *o, int64_t d) {
    if (o == Py_None) return (float)(1.0 / std::sqrt((double)d));
    const double s = PyFloat_AsDouble(o);
    if (s == -1.0 && PyErr_Occurred()) throw Raised();
    return (float)s;
}
unsigned flags_of(PyObject *o) {
    const unsigned long f = PyLong_AsUnsignedLongMask(o);
    if (PyErr_Occurred()) throw Raised();
    return (unsigned)f;
}
at::Tensor empty(c10::IntArrayRef size, at::ScalarType type, c10::Device device) {
    return at::Tensor(at::detail::empty_cuda(size, type, device, std::nullopt));
}

// A tensor that is read or written as `n` elements of a type has that type, and at least as many.
void holds(const at::Tensor &t, at::ScalarType type, int64_t n, const char *name) {
    if (t.scalar_type() == type && t.numel() >= n) return;
    PyErr_Format(PyExc_ValueError, "%s must be a %s tensor of %lld elements", name, c10::toString(type), (long long)n);
    throw Raised();
}

// The caller's workspace, or the plan's own (allocated at the first call, kept afterwards).
struct Workspace {
    void *ptr = nullptr;
    size_t bytes = 0;
    at::Tensor keep;  // the plan's own: another thread may put a larger one in its place during the call
    Workspace(PyObject *given, PlanInfo &pi, int which, size_t need, const c10::cuda::CUDAStream &stream) {
        if (given != Py_None) {
            const at::Tensor &t = tensor(given, "workspace");
            ptr = t.data_ptr();
            bytes = (size_t)t.numel();
        } else if (need > 0) {
            keep = pi.ws[which];
            if (!keep.defined() || (size_t)keep.numel() < need) {
                {
                    const NoGil no_gil;
                    keep = empty({(int64_t)need}, at::kByte, c10::Device(c10::kCUDA, pi.device));
                }
                pi.ws[which] = keep;
                pi.ws_stream[which] = stream.id();
            } else if (stream.id() != pi.ws_stream[which]) {
                keep.record_stream(stream);  // not to be handed out again before this call's kernels are done
            }
            ptr = keep.data_ptr();
            bytes = (size_t)keep.numel();
        }
    }
};

template <typename F>
PyObject *guarded(F &&f) {
    try {
        return f();
    } catch (const Raised &) {
        return nullptr;
    } catch (const std::exception &e) {
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}

// attn_fwd(info, Q, K, V, scale, impl, out, lse, workspace) -> (O, LSE)
PyObject *attn_fwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        if (n != 9) fail(PyExc_TypeError, "attn_fwd takes 9 arguments");
        PlanInfo &pi = plan_info(a[0]);
        const at::Tensor &Q = tensor(a[1], "Q"), &K = tensor(a[2], "K"), &V = tensor(a[3], "V");
        const int64_t d = split(pi, Q);
        if (K.sizes() != Q.sizes() || V.sizes() != Q.sizes()) fail(PyExc_ValueError, "tensor shapes do not match the plan");
        const int dt = dtype_code(Q);
        for (const at::Tensor *t : {&K, &V})
            if (t->scalar_type() != Q.scalar_type()) fail(PyExc_ValueError, "K and V must match Q in dtype");
        at::Tensor O = a[6] == Py_None ? at::Tensor() : tensor(a[6], "O");
        at::Tensor LSE = a[7] == Py_None ? at::Tensor() : tensor(a[7], "LSE");
        if (O.defined()) holds(O, Q.scalar_type(), Q.numel(), "O");
        if (LSE.defined()) holds(LSE, at::kFloat, d > 0 ? Q.numel() / d : 0, "LSE");
        const float scale = scale_of(a[4], d);
        const unsigned impl = flags_of(a[5]);
        void *q = dev(Q, "Q"), *k = dev(K, "K"), *v = dev(V, "V");
        const c10::cuda::OptionalCUDAGuard guard(Q.device().index() != c10::cuda::current_device()
                                                     ? std::optional<c10::Device>(Q.device())
                                                     : std::nullopt);
        void *o = O.defined() ? dev(O, "O") : nullptr, *l = LSE.defined() ? dev(LSE, "LSE") : nullptr;
        size_t need = 0;
        check(lib.workspace_bytes(pi.handle, (int)d, dt, impl, &need, nullptr), "mate_attn_workspace_bytes");
        const c10::cuda::CUDAStream stream = c10::cuda::getCurrentCUDAStream(Q.device().index());
        const Workspace ws(a[8], pi, 0, need, stream);
        const mate_plan_t *plan = pi.handle;
        int status;
        {
            const NoGil no_gil;
            if (!o) O = empty(Q.sizes(), Q.scalar_type(), Q.device()), o = O.data_ptr();
            if (!l) LSE = empty(Q.sizes().slice(0, Q.dim() - 1), at::kFloat, Q.device()), l = LSE.data_ptr();
            status = lib.fwd(plan, q, k, v, (int)d, dt, scale, o, (float *)l, ws.ptr, ws.bytes, impl, stream.stream());
        }
        check(status, "mate_attn_fwd");
        PyObject *po = a[6] == Py_None ? THPVariable_Wrap(O) : Py_NewRef(a[6]);
        PyObject *pl = a[7] == Py_None ? THPVariable_Wrap(LSE) : Py_NewRef(a[7]);
        PyObject *r = po && pl ? PyTuple_Pack(2, po, pl) : nullptr;
        Py_XDECREF(po);
        Py_XDECREF(pl);
        return r;
    });
}

// attn_bwd(info, Q, K, V, O, LSE, dO, scale, impl, workspace) -> (dQ, dK, dV)
PyObject *attn_bwd(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        if (n != 10) fail(PyExc_TypeError, "attn_bwd takes 10 arguments");
        PlanInfo &pi = plan_info(a[0]);
        static const char *const names[] = {"Q", "K", "V", "O", "LSE", "dO"};
        const at::Tensor *t[6];
        for (int i = 0; i < 6; ++i) t[i] = &tensor(a[1 + i], names[i]);
        const at::Tensor &Q = *t[0];
        const int64_t d = split(pi, Q);
        for (int i : {1, 2, 3, 5})
            if (t[i]->sizes() != Q.sizes() || t[i]->scalar_type() != Q.scalar_type())
                fail(PyExc_ValueError, "K, V, O, dO must match Q in shape and dtype");
        const int dt = dtype_code(Q);
        holds(*t[4], at::kFloat, d > 0 ? Q.numel() / d : 0, "LSE");
        const float scale = scale_of(a[7], d);
        const unsigned impl = flags_of(a[8]);
        void *ptr[6];
        for (int i = 0; i < 6; ++i) ptr[i] = dev(*t[i], names[i]);
        const c10::cuda::OptionalCUDAGuard guard(Q.device().index() != c10::cuda::current_device()
                                                     ? std::optional<c10::Device>(Q.device())
                                                     : std::nullopt);
        size_t need = 0;
        check(lib.workspace_bytes(pi.handle, (int)d, dt, impl, nullptr, &need), "mate_attn_workspace_bytes");
        const c10::cuda::CUDAStream stream = c10::cuda::getCurrentCUDAStream(Q.device().index());
        const Workspace ws(a[9], pi, 1, need, stream);
        const mate_plan_t *plan = pi.handle;
        at::Tensor g[3];
        int status;
        {
            const NoGil no_gil;
            for (at::Tensor &x : g) x = empty(Q.sizes(), Q.scalar_type(), Q.device());
            status = lib.bwd(plan, ptr[0], ptr[1], ptr[2], ptr[3], (const float *)ptr[4], ptr[5], (int)d, dt, scale, g[0].data_ptr(),
                             g[1].data_ptr(), g[2].data_ptr(), ws.ptr, ws.bytes, impl, stream.stream());
        }
        check(status, "mate_attn_bwd");
        PyObject *r = PyTuple_New(3);
        for (int i = 0; r && i < 3; ++i) {
            PyObject *o = THPVariable_Wrap(g[i]);
            if (!o) {
                Py_DECREF(r);
                return nullptr;
            }
            PyTuple_SET_ITEM(r, i, o);
        }
        return r;
    });
}

// cell_mean(info, logits, col_ids, want_count, mean or None, count or None) -> (mean, count or None)
PyObject *cell_mean(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        if (n != 6) fail(PyExc_TypeError, "cell_mean takes 6 arguments");
        PlanInfo &pi = plan_info(a[0]);
        const at::Tensor &x = tensor(a[1], "logits"), &ids = tensor(a[2], "col_ids");
        const auto fits = [&](const at::Tensor &t) { return t.dim() == 2 && t.size(0) == pi.B && t.size(1) == pi.N; };
        if (x.scalar_type() != at::kFloat || !fits(x)) fail(PyExc_ValueError, "logits must be a float32 [B, N] tensor");
        if (ids.scalar_type() != at::kInt || !fits(ids))
            fail(PyExc_ValueError, "col_ids must be the int32 [B, N] tensor given to mate_plan");
        const bool given = a[4] != Py_None;  // (mean, count) tensors of an earlier call, written in place
        const bool want = given ? a[5] != Py_None : PyObject_IsTrue(a[3]) == 1;
        at::Tensor mean = given ? tensor(a[4], "mean") : at::Tensor(), count = given && want ? tensor(a[5], "count") : at::Tensor();
        if (given) holds(mean, at::kFloat, pi.B * pi.n_rows * pi.n_cols, "mean");
        if (given && want) holds(count, at::kInt, pi.B * pi.n_rows * pi.n_cols, "count");
        void *px = dev(x, "logits"), *pc = dev(ids, "col_ids");
        const c10::cuda::OptionalCUDAGuard guard(x.device().index() != c10::cuda::current_device()
                                                     ? std::optional<c10::Device>(x.device())
                                                     : std::nullopt);
        const int64_t shape[3] = {pi.B, pi.n_rows, pi.n_cols};
        void *pm_out = given ? dev(mean, "mean") : nullptr, *pn_out = given && want ? dev(count, "count") : nullptr;
        const mate_plan_t *plan = pi.handle;
        int status;
        {
            const NoGil no_gil;
            if (!given) mean = empty(shape, at::kFloat, x.device()), pm_out = mean.data_ptr();
            if (!given && want) count = empty(shape, at::kInt, x.device()), pn_out = count.data_ptr();
            status = lib.cell_mean(plan, (const float *)px, (const int32_t *)pc, (float *)pm_out, (int32_t *)pn_out,
                                   c10::cuda::getCurrentCUDAStream(x.device().index()).stream());
        }
        check(status, "mate_cell_mean");
        PyObject *pm = given ? Py_NewRef(a[4]) : THPVariable_Wrap(mean);
        PyObject *po = !want ? Py_NewRef(Py_None) : given ? Py_NewRef(a[5]) : THPVariable_Wrap(count);
        PyObject *r = pm && po ? PyTuple_Pack(2, pm, po) : nullptr;
        Py_XDECREF(pm);
        Py_XDECREF(po);
        return r;
    });
}

// plan_info(handle, B, N, H, T, n_rows, n_cols, device) -> capsule
PyObject *new_plan_info(PyObject *, PyObject *args) {
    unsigned long long h;
    long long B, N, H, T, nr, nc;
    int device;
    if (!PyArg_ParseTuple(args, "KLLLLLLi", &h, &B, &N, &H, &T, &nr, &nc, &device)) return nullptr;
    PlanInfo *pi = new PlanInfo{reinterpret_cast<const mate_plan_t *>(h), B, N, H, T, nr, nc, (c10::DeviceIndex)device, {}, {}};
    return PyCapsule_New(pi, kCapsule, [](PyObject *c) { delete static_cast<PlanInfo *>(PyCapsule_GetPointer(c, kCapsule)); });
}
// drop(info): the plan has been destroyed; later calls report a null plan
PyObject *drop(PyObject *, PyObject *o) {
    return guarded([&]() -> PyObject * {
        PlanInfo &pi = plan_info(o);
        pi.handle = nullptr;
        for (at::Tensor &w : pi.ws) w = at::Tensor();
        Py_RETURN_NONE;
    });
}
// bind(workspace_bytes, fwd, bwd, cell_mean, error class): addresses of the library's entry points
PyObject *bind(PyObject *, PyObject *args) {
    unsigned long long w, f, b, c;
    PyObject *e;
    if (!PyArg_ParseTuple(args, "KKKKO", &w, &f, &b, &c, &e)) return nullptr;
    lib.workspace_bytes = reinterpret_cast<decltype(lib.workspace_bytes)>(w);
    lib.fwd = reinterpret_cast<decltype(lib.fwd)>(f);
    lib.bwd = reinterpret_cast<decltype(lib.bwd)>(b);
    lib.cell_mean = reinterpret_cast<decltype(lib.cell_mean)>(c);
    Py_XSETREF(mate_error, Py_NewRef(e));
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"attn_fwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(attn_fwd)), METH_FASTCALL, nullptr},
    {"attn_bwd", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(attn_bwd)), METH_FASTCALL, nullptr},
    {"cell_mean", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(cell_mean)), METH_FASTCALL, nullptr},
    {"plan_info", new_plan_info, METH_VARARGS, nullptr},
    {"drop", drop, METH_O, nullptr},
    {"bind", bind, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
