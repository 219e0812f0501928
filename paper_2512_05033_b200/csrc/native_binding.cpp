// The per-call part of the Python binding: checks the tensors, fills the parameter record and calls the C ABI.
//
// A decode token is one call per layer, and the calls of a small model take less time on the device than Python needs
// to marshal them: through ctypes a decode_step call cost 11.4 us of host time (attribute look-ups on nine tensors, a
// structure, twelve converted arguments), against 9-14 us on the device; here 4.3 us (chunk attention 14.7 -> 5.8, the router
// head 8.9 -> 2.3, a cache write 10.8 -> 2.5).  The functions of the library come
// from the handle the Python side has opened (the ordinary or the bounds-check build), so this module links neither.
//
// Every function takes positional arguments, the context handle first, and returns the arb_status; a tensor that is not a
// contiguous CUDA tensor raises ValueError, one of the wrong type TypeError.
#include <Python.h>
#include <dlfcn.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/arb.h"

namespace {

struct Raised {};   // a Python error is set

#define ARB_FUNCTIONS(X)                                                                                              \
    X(arb_attn) X(arb_attn_host) X(arb_attn_host_begin) X(arb_attn_host_wait) X(arb_decode_step) X(arb_decode_step_e4m3)  \
    X(arb_decode_step_i4) X(arb_kv_append) X(arb_kv_append_e4m3) X(arb_kv_append_i4) X(arb_attn_decode_e4m3)               \
    X(arb_attn_e4m3) X(arb_route) X(arb_rollback) X(arb_policy) X(arb_route_classes) X(arb_spearman) X(arb_phase_lens)     \
    X(arb_phase_lens_tokens)

struct Library {
#define X(f) decltype(&::f) f = nullptr;
    ARB_FUNCTIONS(X)
#undef X
} lib;

[[noreturn]] void fail(PyObject *kind, const char *format, const char *a, const char *b = "", const char *c = "") {
    PyErr_Format(kind, format, a, b, c);
    throw Raised();
}

const char *dtype_name(at::ScalarType t) { return torch::getTHPDtype(t)->name; }

const at::Tensor &tensor(PyObject *o, const char *name) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "%s must be a tensor", name);
    return THPVariable_Unpack(o);
}

// address of a contiguous CUDA tensor
void *dev(const at::Tensor &t, const char *name) {
    if (!t.is_cuda() || !t.is_contiguous()) fail(PyExc_ValueError, "%s must be a contiguous CUDA tensor", name);
    return t.data_ptr();
}
void *dev(const at::Tensor &t, const char *name, at::ScalarType want) {
    void *p = dev(t, name);
    if (t.scalar_type() != want) fail(PyExc_TypeError, "%s must be torch.%s, got torch.%s", name, dtype_name(want), dtype_name(t.scalar_type()));
    return p;
}
void *dev(PyObject *o, const char *name, at::ScalarType want) { return dev(tensor(o, name), name, want); }
void *dev_or_null(PyObject *o, const char *name, at::ScalarType want) { return o == Py_None ? nullptr : dev(o, name, want); }

// address of a contiguous host tensor
void *host(const at::Tensor &t) {
    if (t.is_cuda() || !t.is_contiguous()) fail(PyExc_ValueError, "%s", "host tensors must be contiguous CPU tensors");
    return t.data_ptr();
}
void *host(PyObject *o) { return host(tensor(o, "host tensor")); }

int dtype_code(const at::Tensor &t) {
    if (t.scalar_type() == at::kFloat) return ARB_F32;
    if (t.scalar_type() == at::kBFloat16) return ARB_BF16;
    fail(PyExc_TypeError, "arb takes fp32 or bf16 tensors, got torch.%s", dtype_name(t.scalar_type()));
}

int size_of(const at::Tensor &t, int dim, const char *name) {
    if (dim >= t.dim()) fail(PyExc_ValueError, "%s has too few dimensions", name);
    return (int)t.size(dim);
}

// The sizes of a tensor mean what they should only at the right rank: a pool of all layers, or a batch of rows with a
// dimension of its own, would be read with the wrong ones.
const at::Tensor &of_rank(const at::Tensor &t, int rank, const char *name) {
    if (t.dim() != rank) {
        PyErr_Format(PyExc_ValueError, "%s must have %d dimensions, got %d", name, rank, (int)t.dim());
        throw Raised();
    }
    return t;
}

// a number, taken as a C field takes it
int integer(PyObject *o) {
    if (PyFloat_Check(o)) fail(PyExc_TypeError, "%s", "int expected instead of float");
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw Raised();
    return (int)v;
}
float real(PyObject *o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw Raised();
    return (float)v;
}
// ... and as int() and float() take it
int to_int(PyObject *o) {
    if (PyLong_Check(o)) return integer(o);
    PyObject *n = PyNumber_Long(o);
    if (n == nullptr) throw Raised();
    const unsigned long v = PyLong_AsUnsignedLongMask(n);
    Py_DECREF(n);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw Raised();
    return (int)v;
}
float to_float(PyObject *o) {
    if (PyFloat_Check(o)) return real(o);
    PyObject *n = PyNumber_Float(o);
    if (n == nullptr) throw Raised();
    const double v = PyFloat_AS_DOUBLE(n);
    Py_DECREF(n);
    return (float)v;
}
template <typename T>
T *pointer(PyObject *o) {
    if (o == Py_None) return nullptr;
    void *p = PyLong_AsVoidPtr(o);
    if (p == nullptr && PyErr_Occurred()) throw Raised();
    return static_cast<T *>(p);
}
arb_ctx *context(PyObject *o) { return pointer<arb_ctx>(o); }

// None: torch's current stream; else an object with a cuda_stream attribute
arb_stream_t stream_of(PyObject *o) {
    if (o == Py_None) return at::cuda::getCurrentCUDAStream().stream();
    PyObject *v = PyObject_GetAttrString(o, "cuda_stream");
    if (v == nullptr) throw Raised();
    void *p = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    if (p == nullptr && PyErr_Occurred()) throw Raised();
    return static_cast<arb_stream_t>(p);
}

arb_attn_params from_record(PyObject *record) {   // the caller's own AttnParams
    arb_attn_params p;
    Py_buffer view;
    if (PyObject_GetBuffer(record, &view, PyBUF_SIMPLE) != 0) throw Raised();
    const bool fits = view.len == (Py_ssize_t)sizeof(p);
    if (fits) memcpy(&p, view.buf, sizeof(p));
    PyBuffer_Release(&view);
    if (!fits) fail(PyExc_TypeError, "%s", "params must be an AttnParams");
    return p;
}

arb_attn_params params_for(const at::Tensor &q, const at::Tensor &pool, const at::Tensor &table, int max_q_len, PyObject *scale,
                           int flags, PyObject *record, bool exact_q = true) {
    if (record != Py_None) return from_record(record);   // the tensors' shapes are the caller's business then
    if (exact_q) of_rank(q, 3, "q");
    size_of(q, 2, "q");
    of_rank(pool, 4, "the pool");
    of_rank(table, 2, "block_table");
    return {dtype_code(q), (int)table.size(0), (int)q.size(1), (int)pool.size(1), (int)q.size(2), (int)pool.size(2), (int)pool.size(0),
            (int)table.size(1), (int)q.size(0), max_q_len, real(scale), (uint32_t)flags};
}
// code_pack: dimensions per element of a pool row
arb_attn_params params_for_append(int dtype, const at::Tensor &pool, const at::Tensor &table, int code_pack) {
    of_rank(pool, 4, "the pool");
    of_rank(table, 2, "block_table");
    const int hkv = (int)pool.size(1);
    return {dtype, (int)table.size(0), hkv, hkv, code_pack * (int)pool.size(3), (int)pool.size(2), (int)pool.size(0),
            (int)table.size(1), 0, 0, 0.0f, 0u};
}

// Runs `body` (arguments checked, the call made without the GIL) and turns its status into a Python int.
template <typename Body>
PyObject *guarded(Py_ssize_t nargs, Py_ssize_t want, Body body) {
    if (nargs != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
        return nullptr;
    }
    if (lib.arb_attn == nullptr) {
        PyErr_SetString(PyExc_RuntimeError, "bind() has not been called");
        return nullptr;
    }
    try {
        return PyLong_FromLong((long)body());
    } catch (const Raised &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename Call>
arb_status without_gil(Call call) {
    arb_status st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    return st;
}

constexpr auto kI32 = at::kInt;
constexpr auto kU8 = at::kByte;
constexpr auto kBf16 = at::kBFloat16;
#define I32(x) static_cast<int32_t *>(x)
#define U8(x) static_cast<uint8_t *>(x)
#define F32(x) static_cast<float *>(x)
#define METHOD(name) PyObject *name(PyObject *, PyObject *const *a, Py_ssize_t n)

// (h, q, k_pages, v_pages, block_table, seq_lens, q_lens, max_q_len, out, softmax_scale, stream, params)
METHOD(attn) {
    return guarded(n, 12, [&] {
        const at::Tensor &q = tensor(a[1], "q"), &kp = tensor(a[2], "k_pages"), &bt = tensor(a[4], "block_table");
        const arb_attn_params p = params_for(q, kp, bt, integer(a[7]), a[9], 0, a[11]);
        arb_ctx *h = context(a[0]);
        void *qp = dev(q, "q"), *k = dev(kp, "k_pages", q.scalar_type()), *v = dev(a[3], "v_pages", q.scalar_type());
        void *t = dev(bt, "block_table", kI32), *sl = dev(a[5], "seq_lens", kI32), *ql = dev(a[6], "q_lens", kI32);
        void *out = dev(a[8], "out", q.scalar_type());
        arb_stream_t s = stream_of(a[10]);
        return without_gil([&] { return lib.arb_attn(h, &p, qp, k, v, I32(t), I32(sl), I32(ql), out, s); });
    });
}

// (h, q, k_pages, v_pages, block_table, seq_lens, q_lens, max_q_len, out, softmax_scale, flags, stream, begin): q, table, lengths, out on the host
METHOD(attn_host) {
    return guarded(n, 13, [&] {
        const at::Tensor &q = tensor(a[1], "q_host"), &kp = tensor(a[2], "k_pages"), &bt = tensor(a[4], "block_table_host");
        void *qp = host(q), *t = host(bt), *sl = host(a[5]), *ql = host(a[6]), *out = host(a[8]);
        const arb_attn_params p = params_for(q, kp, bt, integer(a[7]), a[9], integer(a[10]), Py_None);
        arb_ctx *h = context(a[0]);
        void *k = dev(kp, "k_pages"), *v = dev(tensor(a[3], "v_pages"), "v_pages");
        arb_stream_t s = stream_of(a[11]);
        auto call = integer(a[12]) ? lib.arb_attn_host_begin : lib.arb_attn_host;
        return without_gil([&] { return call(h, &p, qp, k, v, I32(t), I32(sl), I32(ql), out, s); });
    });
}

// (h)
METHOD(attn_host_wait) {
    return guarded(n, 1, [&] {
        arb_ctx *h = context(a[0]);
        return without_gil([&] { return lib.arb_attn_host_wait(h); });
    });
}

// (h, q, k_new, v_new, k_pages, v_pages, block_table, seq_lens, q_lens, out, softmax_scale, stream, params)
METHOD(decode_step) {
    return guarded(n, 13, [&] {
        const at::Tensor &q = tensor(a[1], "q"), &kp = tensor(a[4], "k_pages"), &bt = tensor(a[6], "block_table");
        const arb_attn_params p = params_for(q, kp, bt, 1, a[10], 0, a[12]);
        arb_ctx *h = context(a[0]);
        const auto dt = q.scalar_type();
        void *qp = dev(q, "q"), *kn = dev(a[2], "k_new", dt), *vn = dev(a[3], "v_new", dt), *k = dev(kp, "k_pages", dt);
        void *v = dev(a[5], "v_pages", dt), *t = dev(bt, "block_table", kI32), *sl = dev(a[7], "seq_lens", kI32);
        void *ql = dev(a[8], "q_lens", kI32), *out = dev(a[9], "out", dt);
        arb_stream_t s = stream_of(a[11]);
        return without_gil([&] { return lib.arb_decode_step(h, &p, qp, kn, vn, k, v, I32(t), I32(sl), I32(ql), out, s); });
    });
}

// (h, q, k_new, v_new, k_codes, v_codes, k_scale, v_scale, k_inv_scale, v_inv_scale, block_table, seq_lens, q_lens, out, softmax_scale, stream, params)
METHOD(decode_step_e4m3) {
    return guarded(n, 17, [&] {
        const at::Tensor &q = tensor(a[1], "q"), &kp = tensor(a[4], "k_codes"), &bt = tensor(a[10], "block_table");
        const arb_attn_params p = params_for(q, kp, bt, 1, a[14], 0, a[16]);
        arb_ctx *h = context(a[0]);
        void *qp = dev(q, "q", kBf16), *kn = dev(a[2], "k_new", kBf16), *vn = dev(a[3], "v_new", kBf16);
        void *k = dev(kp, "k_codes", kU8), *v = dev(a[5], "v_codes", kU8), *t = dev(bt, "block_table", kI32);
        void *sl = dev(a[11], "seq_lens", kI32), *ql = dev(a[12], "q_lens", kI32), *out = dev(a[13], "out", kBf16);
        const float ks = to_float(a[6]), vs = to_float(a[7]), ki = to_float(a[8]), vi = to_float(a[9]);
        arb_stream_t s = stream_of(a[15]);
        return without_gil([&] {
            return lib.arb_decode_step_e4m3(h, &p, qp, kn, vn, U8(k), U8(v), ks, vs, ki, vi, I32(t), I32(sl), I32(ql), out, s);
        });
    });
}

// (h, q, k_new, v_new, k_codes, v_codes, k_scales, v_scales, block_table, seq_lens, q_lens, out, softmax_scale, stream, params)
METHOD(decode_step_i4) {
    return guarded(n, 15, [&] {
        const at::Tensor &q = tensor(a[1], "q"), &kp = tensor(a[4], "k_codes"), &bt = tensor(a[8], "block_table");
        const arb_attn_params p = params_for(q, kp, bt, 1, a[12], 0, a[14], false);
        arb_ctx *h = context(a[0]);
        void *qp = dev(q, "q", kBf16), *kn = dev(a[2], "k_new", kBf16), *vn = dev(a[3], "v_new", kBf16);
        void *k = dev(kp, "k_codes", kU8), *v = dev(a[5], "v_codes", kU8);
        void *ks = dev(a[6], "k_scales", at::kFloat), *vs = dev(a[7], "v_scales", at::kFloat), *t = dev(bt, "block_table", kI32);
        void *sl = dev(a[9], "seq_lens", kI32), *ql = dev(a[10], "q_lens", kI32), *out = dev(a[11], "out", kBf16);
        arb_stream_t s = stream_of(a[13]);
        return without_gil([&] {
            return lib.arb_decode_step_i4(h, &p, qp, kn, vn, U8(k), U8(v), F32(ks), F32(vs), I32(t), I32(sl), I32(ql), out, s);
        });
    });
}

// (h, k_new, v_new, block_table, seq_lens, new_lens, k_pages, v_pages, update_lens, stream)
METHOD(kv_append) {
    return guarded(n, 10, [&] {
        const at::Tensor &kn = tensor(a[1], "k_new"), &bt = tensor(a[3], "block_table"), &kp = tensor(a[6], "k_pages");
        const auto dt = kp.scalar_type();
        const arb_attn_params p = params_for_append(dtype_code(kp), kp, bt, 1);
        arb_ctx *h = context(a[0]);
        void *k = dev(kn, "k_new", dt), *v = dev(a[2], "v_new", dt), *t = dev(bt, "block_table", kI32);
        void *sl = dev(a[4], "seq_lens", kI32), *nl = dev(a[5], "new_lens", kI32), *ko = dev(kp, "k_pages"), *vo = dev(a[7], "v_pages", dt);
        const int total = size_of(kn, 0, "k_new"), update = integer(a[8]);
        arb_stream_t s = stream_of(a[9]);
        return without_gil([&] { return lib.arb_kv_append(h, &p, total, k, v, I32(t), I32(sl), I32(nl), update, ko, vo, s); });
    });
}

// (h, k_new, v_new, k_inv_scale, v_inv_scale, block_table, seq_lens, new_lens, k_codes, v_codes, update_lens, stream)
METHOD(kv_append_e4m3) {
    return guarded(n, 12, [&] {
        const at::Tensor &kn = tensor(a[1], "k_new"), &bt = tensor(a[5], "block_table"), &kp = tensor(a[8], "k_codes");
        const arb_attn_params p = params_for_append(dtype_code(kn), kp, bt, 1);
        arb_ctx *h = context(a[0]);
        void *k = dev(kn, "k_new"), *v = dev(a[2], "v_new", kn.scalar_type()), *t = dev(bt, "block_table", kI32);
        void *sl = dev(a[6], "seq_lens", kI32), *nl = dev(a[7], "new_lens", kI32), *ko = dev(kp, "k_codes", kU8), *vo = dev(a[9], "v_codes", kU8);
        const float ki = to_float(a[3]), vi = to_float(a[4]);
        const int total = size_of(kn, 0, "k_new"), update = integer(a[10]);
        arb_stream_t s = stream_of(a[11]);
        return without_gil([&] { return lib.arb_kv_append_e4m3(h, &p, total, k, v, ki, vi, I32(t), I32(sl), I32(nl), update, U8(ko), U8(vo), s); });
    });
}

// (h, k_new, v_new, block_table, seq_lens, new_lens, k_codes, v_codes, k_scales, v_scales, update_lens, stream)
METHOD(kv_append_i4) {
    return guarded(n, 12, [&] {
        const at::Tensor &kn = tensor(a[1], "k_new"), &bt = tensor(a[3], "block_table"), &kp = tensor(a[6], "k_codes");
        const arb_attn_params p = params_for_append(dtype_code(kn), kp, bt, 2);
        arb_ctx *h = context(a[0]);
        void *k = dev(kn, "k_new", kBf16), *v = dev(a[2], "v_new", kBf16), *t = dev(bt, "block_table", kI32);
        void *sl = dev(a[4], "seq_lens", kI32), *nl = dev(a[5], "new_lens", kI32), *ko = dev(kp, "k_codes", kU8), *vo = dev(a[7], "v_codes", kU8);
        void *ks = dev(a[8], "k_scales", at::kFloat), *vs = dev(a[9], "v_scales", at::kFloat);
        const int total = size_of(kn, 0, "k_new"), update = integer(a[10]);
        arb_stream_t s = stream_of(a[11]);
        return without_gil([&] {
            return lib.arb_kv_append_i4(h, &p, total, k, v, I32(t), I32(sl), I32(nl), update, U8(ko), U8(vo), F32(ks), F32(vs), s);
        });
    });
}

// (h, q, k_codes, v_codes, k_scale, v_scale, block_table, seq_lens, q_lens, max_q_len, out, softmax_scale, flags, stream, params, decode_only)
METHOD(attn_e4m3) {
    return guarded(n, 16, [&] {
        const at::Tensor &q = tensor(a[1], "q"), &kp = tensor(a[2], "k_codes"), &bt = tensor(a[6], "block_table");
        const arb_attn_params p = params_for(q, kp, bt, integer(a[9]), a[11], integer(a[12]), a[14]);
        arb_ctx *h = context(a[0]);
        void *qp = dev(q, "q", kBf16), *k = dev(kp, "k_codes", kU8), *v = dev(a[3], "v_codes", kU8), *t = dev(bt, "block_table", kI32);
        void *sl = dev(a[7], "seq_lens", kI32), *ql = dev(a[8], "q_lens", kI32), *out = dev(a[10], "out", kBf16);
        const float ks = to_float(a[4]), vs = to_float(a[5]);
        arb_stream_t s = stream_of(a[13]);
        auto call = integer(a[15]) ? lib.arb_attn_decode_e4m3 : lib.arb_attn_e4m3;
        return without_gil([&] { return call(h, &p, qp, U8(k), U8(v), ks, vs, I32(t), I32(sl), I32(ql), out, s); });
    });
}

// (h, hidden, w, b, tau, scores, decisions, stream)
METHOD(route) {
    return guarded(n, 8, [&] {
        const at::Tensor &x = of_rank(tensor(a[1], "hidden"), 2, "hidden");
        const int dt = dtype_code(x), steps = size_of(x, 0, "hidden"), dim = size_of(x, 1, "hidden");
        arb_ctx *h = context(a[0]);
        void *hp = dev(x, "hidden"), *w = dev(a[2], "w", x.scalar_type());
        void *sc = dev(a[5], "scores", at::kFloat), *de = dev(a[6], "decisions", kU8);
        const float b = to_float(a[3]), tau = to_float(a[4]);
        arb_stream_t s = stream_of(a[7]);
        return without_gil([&] { return lib.arb_route(h, dt, steps, dim, hp, w, b, tau, F32(sc), U8(de), s); });
    });
}

// (h, mode, hidden, w, biases (tuple of floats), tau, probs, scores, decisions, stream)
METHOD(route_classes) {
    return guarded(n, 10, [&] {
        const at::Tensor &x = of_rank(tensor(a[2], "hidden"), 2, "hidden");
        const int dt = dtype_code(x), steps = size_of(x, 0, "hidden"), dim = size_of(x, 1, "hidden"), mode = integer(a[1]);
        if (!PyTuple_Check(a[4])) fail(PyExc_TypeError, "%s", "b must be a tuple of floats");
        const int classes = (int)PyTuple_GET_SIZE(a[4]);
        float bias[ARB_MAX_CLASSES] = {};
        for (int c = 0; c < classes && c < ARB_MAX_CLASSES; ++c) bias[c] = real(PyTuple_GET_ITEM(a[4], c));
        arb_ctx *h = context(a[0]);
        void *hp = dev(x, "hidden"), *w = dev(a[3], "w", x.scalar_type()), *pr = dev(a[6], "probs", at::kFloat);
        void *sc = dev(a[7], "scores", at::kFloat), *de = dev(a[8], "decisions", kU8);
        const float tau = to_float(a[5]);
        arb_stream_t s = stream_of(a[9]);
        return without_gil([&] {
            return lib.arb_route_classes(h, dt, mode, steps, dim, classes, hp, w, bias, tau, F32(pr), F32(sc), U8(de), s);
        });
    });
}

// (h, seq_lens, step_lens, decisions, stream)
METHOD(rollback) {
    return guarded(n, 5, [&] {
        const at::Tensor &sl = tensor(a[1], "seq_lens");
        const int batch = size_of(sl, 0, "seq_lens");
        arb_ctx *h = context(a[0]);
        void *l = dev(sl, "seq_lens", kI32), *st = dev(a[2], "step_lens", kI32), *de = dev_or_null(a[3], "decisions", kU8);
        arb_stream_t s = stream_of(a[4]);
        return without_gil([&] { return lib.arb_rollback(h, batch, I32(l), I32(st), U8(de), s); });
    });
}

// (h, step_lens, decisions, want, t, out, stream)
METHOD(phase_lens) {
    return guarded(n, 7, [&] {
        const at::Tensor &st = tensor(a[1], "step_lens");
        const int batch = size_of(st, 0, "step_lens"), want = to_int(a[3]), t = to_int(a[4]);
        arb_ctx *h = context(a[0]);
        void *l = dev(st, "step_lens", kI32), *de = dev_or_null(a[2], "decisions", kU8), *out = dev(a[5], "out", kI32);
        arb_stream_t s = stream_of(a[6]);
        return without_gil([&] { return lib.arb_phase_lens(h, batch, I32(l), U8(de), want, t, I32(out), s); });
    });
}

// (h, step_lens, decisions, want, n_tokens, out, stream)
METHOD(phase_lens_tokens) {
    return guarded(n, 7, [&] {
        const at::Tensor &st = tensor(a[1], "step_lens");
        const int batch = size_of(st, 0, "step_lens"), want = to_int(a[3]), tokens = to_int(a[4]);
        arb_ctx *h = context(a[0]);
        void *l = dev(st, "step_lens", kI32), *de = dev_or_null(a[2], "decisions", kU8), *out = dev(a[5], "out", kI32);
        arb_stream_t s = stream_of(a[6]);
        return without_gil([&] { return lib.arb_phase_lens_tokens(h, batch, I32(l), U8(de), want, tokens, I32(out), s); });
    });
}

// (h, kind, s_d, s_t, tau, budget, decisions, stats, stream)
METHOD(policy) {
    return guarded(n, 9, [&] {
        const at::Tensor &sd = tensor(a[2], "s_d");
        const int kind = integer(a[1]), steps = size_of(sd, 0, "s_d"), budget = to_int(a[5]);
        arb_ctx *h = context(a[0]);
        void *d = dev(sd, "s_d", at::kFloat), *t = dev_or_null(a[3], "s_t", at::kFloat), *de = dev(a[6], "decisions", kU8);
        void *st = dev_or_null(a[7], "stats", at::kDouble);
        const float tau = to_float(a[4]);
        arb_stream_t s = stream_of(a[8]);
        return without_gil([&] {
            return lib.arb_policy(h, kind, steps, F32(d), F32(t), tau, budget, U8(de), static_cast<arb_policy_stats *>(st), s);
        });
    });
}

// (h, x, y, rho, stream)
METHOD(spearman) {
    return guarded(n, 5, [&] {
        const at::Tensor &x = tensor(a[1], "x");
        const int count = size_of(x, 0, "x");
        arb_ctx *h = context(a[0]);
        void *xp = dev(x, "x", at::kFloat), *yp = dev(a[2], "y", at::kFloat), *r = dev(a[3], "rho", at::kDouble);
        arb_stream_t s = stream_of(a[4]);
        return without_gil([&] { return lib.arb_spearman(h, count, F32(xp), F32(yp), static_cast<double *>(r), s); });
    });
}

// (handle of the opened library): looks its functions up
PyObject *bind(PyObject *, PyObject *handle) {
    void *h = PyLong_AsVoidPtr(handle);
    if (h == nullptr) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no library handle");
        return nullptr;
    }
    Library found;
#define X(f)                                                                      \
    found.f = reinterpret_cast<decltype(found.f)>(dlsym(h, #f));                  \
    if (found.f == nullptr) {                                                     \
        PyErr_SetString(PyExc_ImportError, "the library does not export " #f);    \
        return nullptr;                                                           \
    }
    ARB_FUNCTIONS(X)
#undef X
    lib = found;
    Py_RETURN_NONE;
}

#define ENTRY(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    ENTRY(attn), ENTRY(attn_host), ENTRY(attn_host_wait), ENTRY(decode_step), ENTRY(decode_step_e4m3), ENTRY(decode_step_i4),
    ENTRY(kv_append), ENTRY(kv_append_e4m3), ENTRY(kv_append_i4), ENTRY(attn_e4m3), ENTRY(route), ENTRY(route_classes),
    ENTRY(rollback), ENTRY(phase_lens), ENTRY(phase_lens_tokens), ENTRY(policy), ENTRY(spearman),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
