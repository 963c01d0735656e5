// binding.cpp -- the Python binding's argument marshalling in native code.
//
// A call through ctypes spends 8-10 us on checking tensors attribute by
// attribute, building structures and asking torch for the stream, against 2.6 us
// in the library (validation, tensor maps, launch); a linear layer on a few
// hundred tokens is bound by that.  Each function here takes the arguments of
// the Python function of the same name, all positional, checks the tensors as
// the Python code does and calls the library: 11.7 -> 3.5 us for
// puro_fp8_quantize, 13.6 -> 3.8 us for puro_fp8_linear_fprop.
//
// Only the ordinary case is handled: plain torch.Tensor objects with storage,
// on CUDA, contiguous, of the expected dtype and not empty, and plain integers
// and floats.  For anything else the function returns None and does nothing,
// and the caller takes its general path, which raises the error or handles the
// case.  Otherwise the result is the library's status code.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "puro_fp8.h"

namespace {

PyObject *operand_type = nullptr;  // the binding's FP8Operand class

// The library's entry points, handed over by the binding (set_library): the
// same library its ctypes calls go to, also where a process holds two copies of
// the package.  Linked by name, the second copy's module got the first one's.
#define PURO_ENTRIES(X)                \
    X(puro_fp8_amax)                   \
    X(puro_fp8_quantize)               \
    X(puro_fp8_quantize_rmsnorm)       \
    X(puro_fp8_quantize_swiglu)        \
    X(puro_fp8_quantize_weights)       \
    X(puro_fp8_linear_fprop)           \
    X(puro_fp8_linear_dgrad)           \
    X(puro_fp8_linear_wgrad)           \
    X(puro_fp8_linear_wgrad_main_grad) \
    X(puro_fp8_linear_backward)        \
    X(puro_fp8_linear_dgrad_quantize)  \
    X(puro_bf16_linear_fprop)          \
    X(puro_bf16_linear_dgrad)          \
    X(puro_bf16_linear_wgrad)
struct Library {
#define PURO_FIELD(name) decltype(&::name) name;
    PURO_ENTRIES(PURO_FIELD)
#undef PURO_FIELD
};
Library lib{};
bool have_library = false;

// `ok` is cleared when an argument is not of the ordinary kind: the call is left to Python.
struct Args {
    PyObject *const *v;
    bool ok = true;

    const at::Tensor *plain(PyObject *o) {
        if (!THPVariable_CheckExact(o)) return nullptr;
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.defined() || !t.has_storage() || !t.is_cuda() || t.numel() == 0) return nullptr;
        return &t;
    }
    // Device pointer of a contiguous tensor of dtype dt or dt2.
    void *ptr_of(PyObject *o, at::ScalarType dt, at::ScalarType dt2) {
        const at::Tensor *t = plain(o);
        if (!t || !t->is_contiguous() || (t->scalar_type() != dt && t->scalar_type() != dt2)) return fail();
        return t->data_ptr();
    }
    void *ptr(int i, at::ScalarType dt) { return ptr_of(v[i], dt, dt); }
    void *opt(int i, at::ScalarType dt) { return v[i] == Py_None ? nullptr : ptr_of(v[i], dt, dt); }
    void *bits(int i) { return ptr_of(v[i], at::kInt, at::kUInt32); }
    void *opt_bits(int i) { return v[i] == Py_None ? nullptr : bits(i); }
    int32_t *status(int i) { return static_cast<int32_t *>(opt(i, at::kInt)); }
    // Scratch of any dtype, and its bytes.
    void *scratch(int i, size_t *bytes) {
        *bytes = 0;
        if (v[i] == Py_None) return nullptr;
        const at::Tensor *t = plain(v[i]);
        if (!t || !t->is_contiguous()) return fail();
        *bytes = t->nbytes();
        return t->data_ptr();
    }
    // Rows and columns of a 2-D tensor.
    void shape(int i, int64_t *rows, int64_t *cols) {
        *rows = *cols = 0;
        if (!ok) return;
        const at::Tensor &t = THPVariable_Unpack(v[i]);
        if (t.dim() != 2) {
            ok = false;
            return;
        }
        *rows = t.size(0);
        *cols = t.size(1);
    }
    int64_t integer_of(PyObject *o) {
        if (!PyLong_CheckExact(o)) return fail(), 0;
        int over = 0;
        const long long x = PyLong_AsLongLongAndOverflow(o, &over);
        if (over) return fail(), 0;
        return x;
    }
    int64_t i64(int i) { return integer_of(v[i]); }
    int32_t i32(int i) {
        const int64_t x = integer_of(v[i]);
        if (x < INT32_MIN || x > INT32_MAX) return fail(), 0;
        return static_cast<int32_t>(x);
    }
    float f32(int i) {
        if (!PyFloat_CheckExact(v[i])) return fail(), 0.0f;
        return static_cast<float>(PyFloat_AS_DOUBLE(v[i]));
    }
    void *stream(int i) {
        if (!ok) return nullptr;
        if (v[i] == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        return fail();  // a Stream object or a raw handle
    }
    // An FP8Operand: its codes, scales and enums.
    void operand(int i, puro_fp8_tensor_t *t) {
        *t = puro_fp8_tensor_t{};
        if (reinterpret_cast<PyObject *>(Py_TYPE(v[i])) != operand_type) ok = false;
        static PyObject *names[5] = {
            PyUnicode_InternFromString("data"), PyUnicode_InternFromString("scale"), PyUnicode_InternFromString("fmt"),
            PyUnicode_InternFromString("scaling"), PyUnicode_InternFromString("role")};
        PyObject *f[5] = {};
        for (int k = 0; k < 5 && ok; ++k) {
            f[k] = PyObject_GetAttr(v[i], names[k]);
            if (!f[k]) {
                PyErr_Clear();
                ok = false;
            }
        }
        if (ok) {
            t->data = static_cast<const uint8_t *>(ptr_of(f[0], at::kByte, at::kByte));
            const at::Tensor *s = plain(f[1]);
            if (!s || !s->is_contiguous()) fail();
            if (ok) {
                const at::Tensor &d = THPVariable_Unpack(f[0]);
                if (d.dim() == 2) {
                    t->rows = d.size(0);
                    t->red = d.size(1);
                } else {
                    ok = false;
                }
                t->scale = s->data_ptr();
            }
            const int64_t e[3] = {integer_of(f[2]), integer_of(f[3]), integer_of(f[4])};
            for (int64_t x : e)
                if (x < INT32_MIN || x > INT32_MAX) ok = false;
            t->fmt = static_cast<int32_t>(e[0]);
            t->scaling = static_cast<int32_t>(e[1]);
            t->role = static_cast<int32_t>(e[2]);
        }
        for (PyObject *o : f) Py_XDECREF(o);  // the operand keeps its tensors
    }
    std::nullptr_t fail() {
        ok = false;
        return nullptr;
    }
};

// Runs `call` without the GIL when every argument was ordinary.  It touches no
// tensor and must not throw: every pointer and size is taken before.
template <class F>
PyObject *finish(const Args &a, F call) {
    if (!a.ok) Py_RETURN_NONE;
    puro_status_t st;
    Py_BEGIN_ALLOW_THREADS;
    st = call();
    Py_END_ALLOW_THREADS;
    return PyLong_FromLong(st);
}

#define PURO_NATIVE(name, nargs)                                                               \
    PyObject *name(PyObject *, PyObject *const *argv, Py_ssize_t n) {                          \
        if (n != (nargs) || !have_library) Py_RETURN_NONE;                                     \
        Args a{argv};                                                                          \
        try {                                                                                  \
            return name##_call(a);                                                             \
        } catch (const std::exception &) { /* e.g. a tensor whose memory cannot be accessed */ \
            Py_RETURN_NONE;                                                                    \
        }                                                                                      \
    }

constexpr at::ScalarType kBF16 = at::kBFloat16, kU8 = at::kByte, kF32 = at::kFloat;

uint8_t *u8(void *p) { return static_cast<uint8_t *>(p); }

// (x, amax_bits, stream)
PyObject *amax_call(Args &a) {
    const void *x = a.ptr(0, kBF16);
    uint32_t *bits = static_cast<uint32_t *>(a.bits(1));
    int64_t r, c;
    a.shape(0, &r, &c);
    void *s = a.stream(2);
    return finish(a, [&] { return lib.puro_fp8_amax(x, r, c, bits, s); });
}
PURO_NATIVE(amax, 3)

// (x, fmt, scaling, role, amax_bits, q, scale, q_t, scale_t, dev_status, stream)
PyObject *quantize_call(Args &a) {
    const void *x = a.ptr(0, kBF16);
    int64_t r, c;
    a.shape(0, &r, &c);
    const int32_t fmt = a.i32(1), scaling = a.i32(2), role = a.i32(3);
    const at::ScalarType sdt = scaling == PURO_SCALE_BLOCK ? kU8 : kF32;
    const uint32_t *bits = static_cast<const uint32_t *>(a.opt_bits(4));
    uint8_t *q = u8(a.opt(5, kU8)), *qt = u8(a.opt(7, kU8));
    void *sc = a.opt(6, sdt), *sct = a.opt(8, sdt);
    int32_t *st = a.status(9);
    void *s = a.stream(10);
    return finish(a, [&] { return lib.puro_fp8_quantize(x, r, c, fmt, scaling, role, bits, q, sc, qt, sct, st, s); });
}
PURO_NATIVE(quantize, 11)

// (h, gamma, eps, fmt, rstd, y, q, scale, q_t, scale_t, dev_status, stream)
PyObject *quantize_rmsnorm_call(Args &a) {
    const void *h = a.ptr(0, kBF16), *gamma = a.opt(1, kBF16);
    int64_t r, c;
    a.shape(0, &r, &c);
    const float eps = a.f32(2);
    const int32_t fmt = a.i32(3);
    float *rstd = static_cast<float *>(a.opt(4, kF32));
    void *y = a.opt(5, kBF16), *sc = a.opt(7, kU8), *sct = a.opt(9, kU8);
    uint8_t *q = u8(a.opt(6, kU8)), *qt = u8(a.opt(8, kU8));
    int32_t *st = a.status(10);
    void *s = a.stream(11);
    return finish(a, [&] { return lib.puro_fp8_quantize_rmsnorm(h, r, c, gamma, eps, fmt, rstd, y, q, sc, qt, sct, st, s); });
}
PURO_NATIVE(quantize_rmsnorm, 12)

// (gate, up, fmt, y, q, scale, q_t, scale_t, dev_status, stream): gate and up
// share their shape and row stride, with unit column stride
PyObject *quantize_swiglu_call(Args &a) {
    const at::Tensor *g = a.plain(a.v[0]), *u = a.plain(a.v[1]);
    if (!g || !u || g->scalar_type() != kBF16 || u->scalar_type() != kBF16 || g->dim() != 2 || u->dim() != 2 ||
        g->sizes() != u->sizes() || g->size(0) < 2 || g->stride(1) != 1 || u->stride(1) != 1 ||
        g->stride(0) != u->stride(0))
        Py_RETURN_NONE;
    const void *gp = g->data_ptr(), *up = u->data_ptr();
    const int64_t r = g->size(0), c = g->size(1), ld = g->stride(0);
    const int32_t fmt = a.i32(2);
    void *y = a.opt(3, kBF16), *sc = a.opt(5, kU8), *sct = a.opt(7, kU8);
    uint8_t *q = u8(a.opt(4, kU8)), *qt = u8(a.opt(6, kU8));
    int32_t *st = a.status(8);
    void *s = a.stream(9);
    return finish(a, [&] { return lib.puro_fp8_quantize_swiglu(gp, up, r, c, ld, fmt, y, q, sc, qt, sct, st, s); });
}
PURO_NATIVE(quantize_swiglu, 10)

// (address of the table, count, fmt, dev_status, stream)
PyObject *quantize_weights_call(Args &a) {
    const int64_t table = a.i64(0);
    const int32_t count = a.i32(1), fmt = a.i32(2);
    int32_t *st = a.status(3);
    void *s = a.stream(4);
    return finish(a, [&] {
        return lib.puro_fp8_quantize_weights(reinterpret_cast<const puro_fp8_weight_t *>(table), count, fmt, st, s);
    });
}
PURO_NATIVE(quantize_weights, 5)

// (a, b, out, workspace, dev_status, stream)
template <class Fn>
PyObject *gemm(Args &a, Fn fn, at::ScalarType out_dtype) {
    puro_fp8_tensor_t x, w;
    a.operand(0, &x);
    a.operand(1, &w);
    void *out = a.opt(2, out_dtype);
    size_t bytes;
    void *ws = a.scratch(3, &bytes);
    int32_t *st = a.status(4);
    void *s = a.stream(5);
    return finish(a, [&] { return fn(&x, &w, out, ws, bytes, st, s); });
}
PyObject *linear_fprop_call(Args &a) { return gemm(a, lib.puro_fp8_linear_fprop, kBF16); }
PyObject *linear_dgrad_call(Args &a) { return gemm(a, lib.puro_fp8_linear_dgrad, kBF16); }
PyObject *linear_wgrad_call(Args &a) { return gemm(a, lib.puro_fp8_linear_wgrad, kBF16); }
PyObject *linear_wgrad_main_grad_call(Args &a) {
    return gemm(a,
                [](const puro_fp8_tensor_t *x, const puro_fp8_tensor_t *w, void *out, void *ws, size_t bytes, int32_t *st,
                   void *s) {
                    return lib.puro_fp8_linear_wgrad_main_grad(x, w, static_cast<float *>(out), ws, bytes, st, s);
                },
                kF32);
}
PURO_NATIVE(linear_fprop, 6)
PURO_NATIVE(linear_dgrad, 6)
PURO_NATIVE(linear_wgrad, 6)
PURO_NATIVE(linear_wgrad_main_grad, 6)

// (dy, w_t, dx, dy_t, x_t, dw, workspace, dev_status, stream)
PyObject *linear_backward_call(Args &a) {
    puro_fp8_tensor_t dy, wt, dyt, xt;
    a.operand(0, &dy);
    a.operand(1, &wt);
    void *dx = a.opt(2, kBF16);
    a.operand(3, &dyt);
    a.operand(4, &xt);
    void *dw = a.opt(5, kBF16);
    size_t bytes;
    void *ws = a.scratch(6, &bytes);
    int32_t *st = a.status(7);
    void *s = a.stream(8);
    return finish(a, [&] { return lib.puro_fp8_linear_backward(&dy, &wt, dx, &dyt, &xt, dw, ws, bytes, st, s); });
}
PURO_NATIVE(linear_backward, 9)

// (dy, w_t, fmt, dx, dxq, dxq_scale, dxq_t, dxq_t_scale, dev_status, stream)
PyObject *linear_dgrad_quantize_call(Args &a) {
    puro_fp8_tensor_t dy, wt;
    a.operand(0, &dy);
    a.operand(1, &wt);
    const int32_t fmt = a.i32(2);
    void *dx = a.opt(3, kBF16), *sc = a.opt(5, kU8), *sct = a.opt(7, kU8);
    uint8_t *q = u8(a.opt(4, kU8)), *qt = u8(a.opt(6, kU8));
    int32_t *st = a.status(8);
    void *s = a.stream(9);
    return finish(a, [&] { return lib.puro_fp8_linear_dgrad_quantize(&dy, &wt, fmt, dx, q, sc, qt, sct, st, s); });
}
PURO_NATIVE(linear_dgrad_quantize, 10)

// (a, b, out, M, N, K, dev_status, stream)
template <class Fn>
PyObject *bf16(Args &a, Fn fn) {
    const void *x = a.opt(0, kBF16), *w = a.opt(1, kBF16);
    void *out = a.opt(2, kBF16);
    const int64_t M = a.i64(3), N = a.i64(4), K = a.i64(5);
    int32_t *st = a.status(6);
    void *s = a.stream(7);
    return finish(a, [&] { return fn(x, w, out, M, N, K, st, s); });
}
PyObject *bf16_fprop_call(Args &a) { return bf16(a, lib.puro_bf16_linear_fprop); }
PyObject *bf16_dgrad_call(Args &a) { return bf16(a, lib.puro_bf16_linear_dgrad); }
PyObject *bf16_wgrad_call(Args &a) { return bf16(a, lib.puro_bf16_linear_wgrad); }
PURO_NATIVE(bf16_fprop, 8)
PURO_NATIVE(bf16_dgrad, 8)
PURO_NATIVE(bf16_wgrad, 8)

// (the FP8Operand class)
PyObject *set_operand_type(PyObject *, PyObject *const *argv, Py_ssize_t n) {
    if (n != 1) {
        PyErr_SetString(PyExc_TypeError, "set_operand_type takes one class");
        return nullptr;
    }
    Py_INCREF(argv[0]);
    Py_XDECREF(operand_type);
    operand_type = argv[0];
    Py_RETURN_NONE;
}

// (name -> address of each entry point)
PyObject *set_library(PyObject *, PyObject *const *argv, Py_ssize_t n) {
    if (n != 1 || !PyDict_Check(argv[0])) {
        PyErr_SetString(PyExc_TypeError, "set_library takes one dict");
        return nullptr;
    }
    Library l{};
#define PURO_TAKE(name)                                                                    \
    {                                                                                      \
        PyObject *o = PyDict_GetItemString(argv[0], #name);                                \
        void *p = o ? PyLong_AsVoidPtr(o) : nullptr;                                       \
        if (!p) {                                                                          \
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no address of " #name); \
            return nullptr;                                                                \
        }                                                                                  \
        l.name = reinterpret_cast<decltype(l.name)>(p);                                    \
    }
    PURO_ENTRIES(PURO_TAKE)
#undef PURO_TAKE
    lib = l;
    have_library = true;
    Py_RETURN_NONE;
}

#define PURO_METHOD(py, fn) {py, reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(fn)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PURO_METHOD("set_operand_type", set_operand_type),
                         PURO_METHOD("set_library", set_library),
                         PURO_METHOD("puro_fp8_amax", amax),
                         PURO_METHOD("puro_fp8_quantize", quantize),
                         PURO_METHOD("puro_fp8_quantize_rmsnorm", quantize_rmsnorm),
                         PURO_METHOD("puro_fp8_quantize_swiglu", quantize_swiglu),
                         PURO_METHOD("puro_fp8_quantize_weights", quantize_weights),
                         PURO_METHOD("puro_fp8_linear_fprop", linear_fprop),
                         PURO_METHOD("puro_fp8_linear_dgrad", linear_dgrad),
                         PURO_METHOD("puro_fp8_linear_wgrad", linear_wgrad),
                         PURO_METHOD("puro_fp8_linear_wgrad_main_grad", linear_wgrad_main_grad),
                         PURO_METHOD("puro_fp8_linear_backward", linear_backward),
                         PURO_METHOD("puro_fp8_linear_dgrad_quantize", linear_dgrad_quantize),
                         PURO_METHOD("puro_bf16_linear_fprop", bf16_fprop),
                         PURO_METHOD("puro_bf16_linear_dgrad", bf16_dgrad),
                         PURO_METHOD("puro_bf16_linear_wgrad", bf16_wgrad),
                         {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", "Native argument marshalling of the Python binding.", -1, methods};

}  // namespace

// (native_for: the torch and the interpreter it was compiled for)
PyMODINIT_FUNC PyInit__native() {
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "native_for", PURO_NATIVE_FOR) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
