// Native argument marshalling of the Python binding (mbscan.py).
//
// A Python-level call spends 12-20 us on checking ten tensors (type, dtype,
// shape, strides, device) and filling the argument struct, several times what
// the small calls take on the GPU. These functions make the same checks on the
// tensors' C++ objects and call the C ABI. Each returns the mb_status, or -1 if
// anything is not as the plain path wants it (a tensor subclass, a wrong dtype,
// shape, stride or device, no storage, no CUDA device, ...): the caller then
// takes the plain path, which raises the error or handles the rest. Nothing is
// kept from one call for the next.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "mbscan.h"

namespace {

// The C ABI's entry points, from the library that mbscan.py has loaded (init).
struct Api {
    decltype(&mb_scan_prefill) prefill;
    decltype(&mb_scan_verify) verify;
    decltype(&mb_scan_verify_resume) verify_resume;
    decltype(&mb_scan_prefill_ckpt) prefill_ckpt;
    decltype(&mb_step) step;
    decltype(&mb_step_resume) step_resume;
    decltype(&mb_rollback) rollback;
    decltype(&mb_accept_topk) accept_topk;
    decltype(&mb_rmsnorm) rmsnorm;
    decltype(&mb_conv1d_step) conv1d_step;
    decltype(&mb_conv_xproj) conv_xproj;
} api;

// One call's tensors and whether all of them are as they should be.
struct Call {
    PyObject *const *v;
    bool ok = true;
    c10::Device dev{c10::kCPU};
    bool have_dev = false;

    const at::Tensor *get(int i) {   // null for None
        if (v[i] == Py_None) return nullptr;
        if (!THPVariable_CheckExact(v[i])) {
            ok = false;
            return nullptr;
        }
        return &THPVariable_Unpack(v[i]);
    }
    void *ptr(const at::Tensor *t) { return t && ok ? t->data_ptr() : nullptr; }
    // contiguous, of this dtype and shape, on the call's device (that of its first tensor, a CUDA device)
    void *need(int i, at::ScalarType ty, c10::IntArrayRef dims, bool any_shape = false) {
        const at::Tensor *t = get(i);
        if (!t || !ok) return nullptr;
        if (t->scalar_type() != ty || (!any_shape && t->sizes() != dims) || !t->is_contiguous() || !on(*t)) ok = false;
        return ptr(t);
    }
    // the same, and not None
    void *must(int i, at::ScalarType ty, c10::IntArrayRef dims, bool any_shape = false) {
        if (v[i] == Py_None) ok = false;
        return need(i, ty, dims, any_shape);
    }
    bool on(const at::Tensor &t) {
        if (!have_dev) {
            dev = t.device();
            have_dev = true;
        }
        return t.device() == dev && dev.is_cuda();
    }
    // row stride of a [batch, L, width] tensor: contiguous, or a column block of wider rows
    int64_t row_stride(const at::Tensor *t, int64_t batch, int64_t L, int64_t width, at::ScalarType ty) {
        if (!t || t->scalar_type() != ty || t->sizes() != c10::IntArrayRef({batch, L, width}) || !on(*t)) {
            ok = false;
            return 0;
        }
        if (t->is_contiguous()) return width;
        const auto st = t->strides();
        if (st[2] != 1 || (L > 1 && st[0] != L * st[1]) || st[1] < width) {
            ok = false;
            return 0;
        }
        return L > 1 || batch == 1 ? st[1] : st[0];
    }
};

constexpr at::ScalarType kF32 = at::kFloat;

bool dtype_of(const at::Tensor *t, int32_t &dt) {
    if (!t) return false;
    if (t->scalar_type() == at::kFloat) dt = MB_F32;
    else if (t->scalar_type() == at::kBFloat16) dt = MB_BF16;
    else return false;
    return true;
}

// v[0..9]: x, dt, B, C, A, y, z, D, dt_bias, h0
bool fill(Call &c, mb_scan_args &a) {
    a = mb_scan_args{};
    const at::Tensor *x = c.get(0), *A = c.get(4), *B = c.get(2), *C = c.get(3);
    if (!c.ok || !x || !A || !B || !C || x->dim() != 3 || A->dim() != 2 || !dtype_of(x, a.dtype)) return false;
    c.on(*x);
    const at::ScalarType ty = x->scalar_type();
    const int64_t b = x->size(0), L = x->size(1), D = x->size(2), N = A->size(1);
    a.batch = b; a.seqlen = L; a.d_inner = D; a.d_state = N;
    const int64_t tok[3] = {b, L, D};
    a.x = c.must(0, ty, tok);
    a.dt = c.must(1, ty, tok);
    a.y = c.must(5, ty, tok);
    a.z = c.need(6, ty, tok);
    const int64_t S = c.row_stride(B, b, L, N, ty), S2 = c.row_stride(C, b, L, N, ty);
    if (S != S2 || S > INT32_MAX) c.ok = false;
    a.bc_stride = S == N ? 0 : (int32_t)S;
    a.B = c.ptr(B);
    a.C = c.ptr(C);
    a.A = static_cast<const float *>(c.must(4, kF32, {D, N}));
    a.D = static_cast<const float *>(c.need(7, kF32, {D}));
    a.dt_bias = static_cast<const float *>(c.need(8, kF32, {D}));
    a.h0 = static_cast<const float *>(c.need(9, kF32, {b, D, N}));
    return c.ok;
}

// A workspace tensor: uint8, contiguous; bytes in `n`
void *workspace(Call &c, int i, size_t &n, bool may_be_none) {
    n = 0;
    if (c.v[i] == Py_None) {
        if (!may_be_none) c.ok = false;
        return nullptr;
    }
    void *p = c.need(i, at::kByte, {}, true);
    if (c.ok) n = (size_t)c.get(i)->numel();
    return p;
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

template <typename F>
PyObject *guarded(Py_ssize_t have, Py_ssize_t want, F &&f) {
    if (have != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, have);
        return nullptr;
    }
    long rc = -1;
    try {
        rc = f();
    } catch (...) {   // e.g. a tensor without storage: the plain path reports it
        rc = -1;
    }
    return PyLong_FromLong(rc);
}

// Run a C ABI call without the interpreter lock (as ctypes does).
template <typename F>
long call(F &&f) {
    void *s = stream();
    long rc;
    Py_BEGIN_ALLOW_THREADS
    rc = (long)f(s);
    Py_END_ALLOW_THREADS
    return rc;
}

#define ARGS PyObject *, PyObject *const *v, Py_ssize_t n

// x, dt, B, C, A, y, z, D, dt_bias, None, state, ws
PyObject *step(ARGS) {
    return guarded(n, 12, [&]() -> long {
        Call c{v};
        mb_scan_args a;
        if (!fill(c, a)) return -1;
        float *state = static_cast<float *>(c.must(10, kF32, {a.batch, a.d_inner, a.d_state}));
        size_t wb;
        void *ws = workspace(c, 11, wb, true);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.step(&a, state, ws, wb, s); });
    });
}

// x, dt, B, C, A, y, z, D, dt_bias, h0, h_all, accept, state, ws
PyObject *step_resume(ARGS) {
    return guarded(n, 14, [&]() -> long {
        Call c{v};
        mb_scan_args a;
        if (!fill(c, a)) return -1;
        const at::Tensor *h = c.get(10);
        if (!h || h->dim() != 4) return -1;
        const int64_t k = h->size(1);
        const float *h_all = static_cast<const float *>(c.must(10, kF32, {a.batch, k, a.d_inner, a.d_state}));
        const int32_t *acc = static_cast<const int32_t *>(c.must(11, at::kInt, {a.batch}));
        float *state = static_cast<float *>(c.must(12, kF32, {a.batch, a.d_inner, a.d_state}));
        size_t wb;
        void *ws = workspace(c, 13, wb, true);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.step_resume(&a, h_all, acc, k, state, ws, wb, s); });
    });
}

// x, dt, B, C, A, y, z, D, dt_bias, h0, h_last, ws
PyObject *prefill(ARGS) {
    return guarded(n, 12, [&]() -> long {
        Call c{v};
        mb_scan_args a;
        if (!fill(c, a)) return -1;
        float *h_last = static_cast<float *>(c.need(10, kF32, {a.batch, a.d_inner, a.d_state}));
        size_t wb;
        void *ws = workspace(c, 11, wb, false);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.prefill(&a, h_last, ws, wb, s); });
    });
}

// x, dt, B, C, A, y, z, D, dt_bias, h0, h_last, h_ckpt, ws
PyObject *prefill_ckpt(ARGS) {
    return guarded(n, 13, [&]() -> long {
        Call c{v};
        mb_scan_args a;
        if (!fill(c, a)) return -1;
        float *h_last = static_cast<float *>(c.need(10, kF32, {a.batch, a.d_inner, a.d_state}));
        const int64_t nch = (a.seqlen + MB_CKPT_STEPS - 1) / MB_CKPT_STEPS;
        float *ck = static_cast<float *>(c.must(11, kF32, {a.batch, nch, a.d_inner, a.d_state}));
        size_t wb;
        void *ws = workspace(c, 12, wb, false);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.prefill_ckpt(&a, h_last, ck, ws, wb, s); });
    });
}

// x, dt, B, C, A, y, z, D, dt_bias, h0, h_all, ws
PyObject *verify(ARGS) {
    return guarded(n, 12, [&]() -> long {
        Call c{v};
        mb_scan_args a;
        if (!fill(c, a)) return -1;
        float *h_all = static_cast<float *>(c.must(10, kF32, {a.batch, a.seqlen, a.d_inner, a.d_state}));
        size_t wb;
        void *ws = workspace(c, 11, wb, false);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.verify(&a, h_all, ws, wb, s); });
    });
}

// x, dt, B, C, A, y, z, D, dt_bias, h0, h_all, h_all_prev, accept, ws
PyObject *verify_resume(ARGS) {
    return guarded(n, 14, [&]() -> long {
        Call c{v};
        mb_scan_args a;
        if (!fill(c, a)) return -1;
        float *h_all = static_cast<float *>(c.must(10, kF32, {a.batch, a.seqlen, a.d_inner, a.d_state}));
        const at::Tensor *h = c.get(11);
        if (!h || h->dim() != 4) return -1;
        const int64_t k = h->size(1);
        const float *prev = static_cast<const float *>(c.must(11, kF32, {a.batch, k, a.d_inner, a.d_state}));
        const int32_t *acc = static_cast<const int32_t *>(c.must(12, at::kInt, {a.batch}));
        size_t wb;
        void *ws = workspace(c, 13, wb, false);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.verify_resume(&a, prev, acc, k, h_all, ws, wb, s); });
    });
}

// h0, h_all, accept, h_out, ws
PyObject *rollback(ARGS) {
    return guarded(n, 5, [&]() -> long {
        Call c{v};
        const at::Tensor *h = c.get(1);
        if (!h || h->dim() != 4) return -1;
        c.on(*h);
        const int64_t b = h->size(0), k = h->size(1), D = h->size(2), N = h->size(3);
        const float *h_all = static_cast<const float *>(c.must(1, kF32, {b, k, D, N}));
        const float *h0 = static_cast<const float *>(c.need(0, kF32, {b, D, N}));
        const int32_t *acc = static_cast<const int32_t *>(c.must(2, at::kInt, {b}));
        float *out = static_cast<float *>(c.must(3, kF32, {b, D, N}));
        size_t wb;
        void *ws = workspace(c, 4, wb, true);
        if (!c.ok) return -1;
        return call([&](void *s) { return api.rollback(h0, h_all, acc, out, b, k, D, N, ws, s); });
    });
}

// logits, drafted, accept, beta
PyObject *accept_topk(ARGS) {
    return guarded(n, 4, [&]() -> long {
        Call c{v};
        const at::Tensor *t = c.get(0);
        int32_t dt;
        if (!t || t->dim() != 3 || t->size(2) != 256 || !dtype_of(t, dt) || !PyLong_CheckExact(v[3])) return -1;
        int over = 0;
        const long beta = PyLong_AsLongAndOverflow(v[3], &over);
        if (over || beta < INT32_MIN || beta > INT32_MAX) return -1;
        const int64_t b = t->size(0), k = t->size(1);
        const void *logits = c.must(0, t->scalar_type(), {b, k, 256});
        const uint8_t *drafted = static_cast<const uint8_t *>(c.must(1, at::kByte, {b, k}));
        int32_t *acc = static_cast<int32_t *>(c.must(2, at::kInt, {b}));
        if (!c.ok) return -1;
        return call([&](void *s) { return api.accept_topk(logits, dt, drafted, b, k, (int32_t)beta, acc, s); });
    });
}

// residual, w, out, add, eps
PyObject *rmsnorm(ARGS) {
    return guarded(n, 5, [&]() -> long {
        Call c{v};
        const at::Tensor *r = c.get(0), *o = c.get(2);
        int32_t dt;
        if (!r || r->dim() != 2 || !dtype_of(o, dt) || !PyFloat_CheckExact(v[4])) return -1;
        c.on(*r);
        const int64_t b = r->size(0), w = r->size(1);
        float *res = static_cast<float *>(c.must(0, kF32, {b, w}));
        const float *wt = static_cast<const float *>(c.must(1, kF32, {w}));
        void *out = c.must(2, o->scalar_type(), {b, w});
        const void *add = c.need(3, o->scalar_type(), {b, w});
        if (!c.ok) return -1;
        const float eps = (float)PyFloat_AS_DOUBLE(v[4]);
        return call([&](void *s) { return api.rmsnorm(add, res, wt, eps, out, b, w, dt, s); });
    });
}

// x, state, w, out, bias
PyObject *conv1d_step(ARGS) {
    return guarded(n, 5, [&]() -> long {
        Call c{v};
        const at::Tensor *x = c.get(0);
        int32_t dt;
        if (!x || x->dim() != 2 || !dtype_of(x, dt)) return -1;
        c.on(*x);
        const at::ScalarType ty = x->scalar_type();
        const int64_t b = x->size(0), w = x->size(1);
        const void *xp = c.must(0, ty, {b, w});
        void *st = c.must(1, ty, {b, 3, w});
        const float *wt = static_cast<const float *>(c.must(2, kF32, {w, 4}));
        void *out = c.must(3, ty, {b, w});
        const float *bias = static_cast<const float *>(c.need(4, kF32, {w}));
        if (!c.ok) return -1;
        return call([&](void *s) { return api.conv1d_step(xp, st, wt, bias, out, b, w, dt, s); });
    });
}

// x, state, w, W, xc, out, ws, bias
PyObject *conv_xproj(ARGS) {
    return guarded(n, 8, [&]() -> long {
        Call c{v};
        const at::Tensor *x = c.get(0), *W = c.get(3);
        if (!x || x->dim() != 2 || !W || W->dim() != 2 || W->size(0) > INT32_MAX) return -1;
        c.on(*x);
        constexpr at::ScalarType bf = at::kBFloat16;
        const int64_t b = x->size(0), w = x->size(1), no = W->size(0);
        const void *xp = c.must(0, bf, {b, w});
        void *st = c.must(1, bf, {b, 3, w});
        const float *wt = static_cast<const float *>(c.must(2, kF32, {w, 4}));
        const void *Wp = c.must(3, bf, {no, w});
        void *xc = c.must(4, bf, {b, w}), *out = c.must(5, bf, {b, no});
        size_t wb;
        void *ws = workspace(c, 6, wb, false);
        const float *bias = static_cast<const float *>(c.need(7, kF32, {w}));
        if (!c.ok) return -1;
        return call([&](void *s) {
            return api.conv_xproj(xp, st, wt, bias, Wp, xc, out, b, w, (int32_t)no, MB_BF16, ws, wb, s);
        });
    });
}

// init(addresses of the entry points, in Api's order)
PyObject *init(ARGS) {
    constexpr Py_ssize_t kN = sizeof(Api) / sizeof(void *);
    if (n != kN) {
        PyErr_Format(PyExc_TypeError, "expected %zd addresses, got %zd", kN, n);
        return nullptr;
    }
    void *p[kN];
    for (Py_ssize_t i = 0; i < kN; ++i) {
        p[i] = PyLong_AsVoidPtr(v[i]);
        if (PyErr_Occurred()) return nullptr;
    }
    static_assert(sizeof(p) == sizeof(api), "one address per entry point");
    std::memcpy(&api, p, sizeof(api));
    Py_RETURN_NONE;
}

#define DEF(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {DEF(init),     DEF(step),          DEF(step_resume), DEF(prefill), DEF(prefill_ckpt),
                         DEF(verify),   DEF(verify_resume), DEF(rollback),    DEF(accept_topk), DEF(rmsnorm),
                         DEF(conv1d_step), DEF(conv_xproj), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mbcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mbcall(void) { return PyModule_Create(&module); }
