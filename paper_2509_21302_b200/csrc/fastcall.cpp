// The call path from Python into libqvggt, for the calls a program makes per layer: forward passes and preparation.
//
// Through ctypes a call costs 8.5 us on the host, 2.4 of it the launch itself: tensor attributes read one by one from Python, the
// stream object, ctypes' argument conversion.  At a frame or less that is more than the work on the GPU.  Here the arguments go
// from the tensors to the C entry points directly (2.7 us a call in all).
//
// A function returns what its namesake in binding.py returns, or None when an argument is not plainly what the call expects or
// the library returned a status: binding.py then takes its own path, which checks, converts and reports.  (The two views of a handle
// have no other path and raise.)  Nothing here keeps state.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <ATen/ops/from_blob.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/qvggt.h"

namespace {

using at::ScalarType;
using at::Tensor;

// Positional arguments of one call.  `ok` turns false at the first one that this path does not take.
struct Args {
    PyObject *const *a;
    Py_ssize_t n, i = 0;
    bool ok = true;

    PyObject *next() { return (i < n) ? a[i++] : (ok = false, Py_None); }
    const qvggt_weights_t *handle()
    {
        PyObject *o = next();
        void *p = PyLong_Check(o) ? PyLong_AsVoidPtr(o) : nullptr;
        if (!p) ok = false;
        if (PyErr_Occurred()) PyErr_Clear();
        return static_cast<const qvggt_weights_t *>(p);
    }
    long long integer()
    {
        PyObject *o = next();
        const long long v = PyLong_Check(o) ? PyLong_AsLongLong(o) : (ok = false, 0);
        if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
        return v;
    }
    double real()
    {
        PyObject *o = next();
        const double v = (PyFloat_Check(o) || PyLong_Check(o)) ? PyFloat_AsDouble(o) : (ok = false, 0.0);
        if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
        return v;
    }
    // A CUDA tensor (which device it is on is the caller's affair, as on the other route), or an undefined one for None where `optional`.
    const Tensor &tensor(bool optional = false)
    {
        static const Tensor none;
        PyObject *o = next();
        if (o == Py_None && optional) return none;
        if (!THPVariable_Check(o)) { ok = false; return none; }
        const Tensor &t = THPVariable_Unpack(o);
        if (!t.is_cuda() || t.layout() != at::kStrided) ok = false;
        return t;
    }
    // Activation rows: bf16 [M, K], unit stride along K.
    const Tensor &rows(int64_t K)
    {
        const Tensor &t = tensor();
        if (ok && !(t.dim() == 2 && t.element_size() == 2 && t.size(1) == K && t.stride(1) == 1)) ok = false;
        return t;
    }
    // A contiguous tensor of the given type and shape.
    const Tensor &exact(ScalarType type, int64_t d0, int64_t d1, bool optional = false)
    {
        const Tensor &t = tensor(optional);
        if (ok && t.defined()) {
            const bool shape = d1 < 0 ? (t.dim() == 1 && t.size(0) == d0) : (t.dim() == 2 && t.size(0) == d0 && t.size(1) == d1);
            if (t.scalar_type() != type || !shape || !t.is_contiguous()) ok = false;
        }
        return t;
    }
    // A contiguous tensor of the given type with at least n elements.
    const Tensor &at_least(ScalarType type, int64_t n_min)
    {
        const Tensor &t = tensor();
        if (ok && !(t.scalar_type() == type && t.numel() >= n_min && t.is_contiguous())) ok = false;
        return t;
    }
    bool done() const { return ok && i == n; }
};

int64_t pitch(const Tensor &t) { return t.size(0) > 1 ? t.stride(0) : t.size(1); }

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// f() touches no tensor and no Python object: a tensor's data_ptr() may throw, or call back into Python.
template <class F>
int without_gil(F f)
{
    struct Released {
        PyThreadState *s = PyEval_SaveThread();
        ~Released() { PyEval_RestoreThread(s); }
    } released;
    return f();
}

PyObject *wrap(const Tensor &given, const Tensor &made, PyObject *obj)
{
    if (given.defined()) { Py_INCREF(obj); return obj; }
    return THPVariable_Wrap(made);
}

#define QVGGT_GUARD_BEGIN try {
#define QVGGT_GUARD_END                                     \
    }                                                       \
    catch (const std::exception &) { Py_RETURN_NONE; }

// Quantize calls: f(handle, X, ldx, M, Xq, a_scale, stream); `X` and what precedes the outputs have been read from `in`.
template <class F>
PyObject *quantize(Args &in, const Tensor &X, ScalarType code, int64_t row_codes, int64_t row_scales, F f)
{
    if (!in.ok) Py_RETURN_NONE;
    const int64_t M = X.size(0);
    PyObject *oq = in.next(), *oa = in.next();
    in.i -= 2;
    const Tensor &xq = in.exact(code, M, row_codes, true), &as = in.exact(at::kFloat, M, row_scales, true);
    if (!in.done() || M > INT32_MAX) Py_RETURN_NONE;
    const Tensor made_q = xq.defined() ? Tensor() : at::empty({M, row_codes}, X.options().dtype(code));
    const Tensor made_a = as.defined() ? Tensor() : (row_scales < 0 ? at::empty({M}, X.options().dtype(at::kFloat)) : at::empty({M, row_scales}, X.options().dtype(at::kFloat)));
    const void *x = X.data_ptr();
    void *q = (xq.defined() ? xq : made_q).data_ptr();
    float *a = static_cast<float *>((as.defined() ? as : made_a).data_ptr());
    void *st = stream();
    const int64_t ldx = pitch(X);
    if (without_gil([&] { return f(x, ldx, (int)M, q, a, st); }) != QVGGT_OK) Py_RETURN_NONE;
    return PyTuple_Pack(2, wrap(xq, made_q, oq), wrap(as, made_a, oa));
}

// PyTuple_Pack adds references of its own: give back the ones wrap() made.
PyObject *release_items(PyObject *t)
{
    if (t && PyTuple_Check(t))
        for (Py_ssize_t i = 0; i < PyTuple_GET_SIZE(t); ++i) Py_DECREF(PyTuple_GET_ITEM(t, i));
    return t;
}

// GEMM calls: f(codes, a_scale, M, Y, ldy, stream); reads Y (optional) and returns it.
template <class F>
PyObject *linear(Args &in, const Tensor &xq, const Tensor &as, int64_t N, F f)
{
    if (!in.ok) Py_RETURN_NONE;
    const int64_t M = xq.size(0);
    PyObject *oy = in.next();
    --in.i;
    const Tensor &y = in.tensor(true);
    if (!in.done() || M > INT32_MAX) Py_RETURN_NONE;
    if (y.defined() && !(y.dim() == 2 && y.element_size() == 2 && y.size(0) == M && y.size(1) == N && y.stride(1) == 1)) Py_RETURN_NONE;
    const Tensor made = y.defined() ? Tensor() : at::empty({M, N}, xq.options().dtype(at::kBFloat16));
    const Tensor &Y = y.defined() ? y : made;
    const void *q = xq.data_ptr();
    const float *a = static_cast<const float *>(as.data_ptr());
    void *out = Y.data_ptr(), *st = stream();
    const int64_t ldy = pitch(Y);
    if (without_gil([&] { return f(q, a, (int)M, out, ldy, st); }) != QVGGT_OK) Py_RETURN_NONE;
    return wrap(y, made, oy);
}

using U8 = unsigned char;
using S8 = signed char;

// (handle, K, X, group, Xq, a_scale)
PyObject *rotate_smooth_quantize(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t K = in.integer();
    const Tensor &X = in.rows(K);
    const int64_t group = in.integer();
    if (group != 0 && group != 128) Py_RETURN_NONE;
    return release_items(quantize(in, X, at::kByte, K / 2, group ? K / 128 : -1, [&](const void *x, int64_t ldx, int M, void *q, float *a, void *st) {
        return qvggt_rotate_smooth_quantize(h, x, ldx, M, (int)group, static_cast<U8 *>(q), a, st);
    }));
    QVGGT_GUARD_END
}

// (handle, K, X, Xq8, a_scale)
template <int (*FN)(const qvggt_weights_t *, const void *, long long, int, S8 *, float *, void *), bool GROUPED>
PyObject *quantize_c8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t K = in.integer();
    const Tensor &X = in.rows(K);
    return release_items(quantize(in, X, at::kChar, K, GROUPED ? K / 128 : -1, [&](const void *x, int64_t ldx, int M, void *q, float *a, void *st) {
        return FN(h, x, ldx, M, static_cast<S8 *>(q), a, st);
    }));
    QVGGT_GUARD_END
}

// (handle, K, X, c8, Xq, a_scale)
PyObject *rotate_smooth_quantize_tc(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t K = in.integer();
    const Tensor &X = in.rows(K);
    const bool c8 = in.integer() != 0;
    return release_items(quantize(in, X, c8 ? at::kChar : at::kByte, c8 ? K : K / 2, -1, [&](const void *x, int64_t ldx, int M, void *q, float *a, void *st) {
        return c8 ? qvggt_rotate_smooth_quantize_tc_c8(h, x, ldx, M, static_cast<S8 *>(q), a, nullptr, st)
                  : qvggt_rotate_smooth_quantize_tc(h, x, ldx, M, static_cast<U8 *>(q), a, nullptr, st);
    }));
    QVGGT_GUARD_END
}

// (handle, K, X, delta, Xq8, a_scale)
PyObject *rotate_smooth_quantize_static_c8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t K = in.integer();
    const Tensor &X = in.rows(K);
    const Tensor &delta = in.at_least(at::kFloat, 1);
    if (!in.ok || delta.numel() != 1) Py_RETURN_NONE;
    const auto *d = static_cast<const float *>(delta.data_ptr());
    return release_items(quantize(in, X, at::kChar, K, -1, [&](const void *x, int64_t ldx, int M, void *q, float *a, void *st) {
        return qvggt_rotate_smooth_quantize_static_c8(h, x, ldx, M, d, static_cast<S8 *>(q), a, st);
    }));
    QVGGT_GUARD_END
}

// (handle, K, X, gamma, beta, eps, Xq8, a_scale)
PyObject *layernorm_rotate_smooth_quantize_c8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t K = in.integer();
    const Tensor &X = in.rows(K);
    const Tensor &gamma = in.exact(at::kFloat, K, -1), &beta = in.exact(at::kFloat, K, -1);
    const float eps = (float)in.real();
    if (!in.ok) Py_RETURN_NONE;
    const auto *gp = static_cast<const float *>(gamma.data_ptr()), *bp = static_cast<const float *>(beta.data_ptr());
    return release_items(quantize(in, X, at::kChar, K, -1, [&](const void *x, int64_t ldx, int M, void *q, float *a, void *st) {
        return qvggt_layernorm_rotate_smooth_quantize_c8(h, x, ldx, M, gp, bp, eps, static_cast<S8 *>(q), a, st);
    }));
    QVGGT_GUARD_END
}

// (handle, N, K, X, w_scratch, Xq8, a_scale)
PyObject *rotate_smooth_quantize_c8_expand(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t N = in.integer(), K = in.integer();
    const Tensor &X = in.rows(K);
    const Tensor &scratch = in.at_least(at::kChar, N * K);
    if (!in.ok) Py_RETURN_NONE;
    S8 *w = static_cast<S8 *>(scratch.data_ptr());
    return release_items(quantize(in, X, at::kChar, K, -1, [&](const void *x, int64_t ldx, int M, void *q, float *a, void *st) {
        return qvggt_rotate_smooth_quantize_c8_expand(h, x, ldx, M, static_cast<S8 *>(q), a, w, st);
    }));
    QVGGT_GUARD_END
}

// (handle, N, K, Xq, a_scale, group, Y)
PyObject *w4a4_linear(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t N = in.integer(), K = in.integer();
    const Tensor &xq = in.at_least(at::kByte, 0);
    if (!in.ok || xq.dim() != 2 || xq.size(1) != K / 2) Py_RETURN_NONE;
    const Tensor &as = in.at_least(at::kFloat, 0);
    const int64_t group = in.integer();
    if (!in.ok || (group != 0 && group != 128) || as.numel() < xq.size(0) * (group ? K / 128 : 1)) Py_RETURN_NONE;
    return linear(in, xq, as, N, [&](const void *q, const float *a, int M, void *y, int64_t ldy, void *st) {
        return qvggt_w4a4_linear(h, static_cast<const U8 *>(q), a, M, (int)group, y, ldy, nullptr, st);
    });
    QVGGT_GUARD_END
}

// (handle, N, K, Xq8, a_scale, Y)
template <int (*FN)(const qvggt_weights_t *, const S8 *, const float *, int, void *, long long, int *, void *), bool GROUPED>
PyObject *linear_c8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t N = in.integer(), K = in.integer();
    const Tensor &xq = in.at_least(at::kChar, 0);
    if (!in.ok || xq.dim() != 2 || xq.size(1) != K) Py_RETURN_NONE;
    const Tensor &as = GROUPED ? in.exact(at::kFloat, xq.size(0), K / 128) : in.at_least(at::kFloat, xq.size(0));
    return linear(in, xq, as, N, [&](const void *q, const float *a, int M, void *y, int64_t ldy, void *st) {
        return FN(h, static_cast<const S8 *>(q), a, M, y, ldy, nullptr, st);
    });
    QVGGT_GUARD_END
}

// (handle, N, K, Xq8, a_scale, w_scratch, Y)
template <bool EXPANDED>
PyObject *linear_scratch(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    auto *h = in.handle();
    const int64_t N = in.integer(), K = in.integer();
    const Tensor &xq = in.at_least(at::kChar, 0);
    if (!in.ok || xq.dim() != 2 || xq.size(1) != K) Py_RETURN_NONE;
    const Tensor &as = in.at_least(at::kFloat, xq.size(0));
    const Tensor &scratch = in.at_least(at::kChar, N * K);
    if (!in.ok) Py_RETURN_NONE;
    S8 *w = static_cast<S8 *>(scratch.data_ptr());
    return linear(in, xq, as, N, [&](const void *q, const float *a, int M, void *y, int64_t ldy, void *st) {
        return EXPANDED ? qvggt_w4a4_linear_c8_expanded(h, static_cast<const S8 *>(q), a, M, y, ldy, w, nullptr, st)
                        : qvggt_w4a4_linear_c8_packed_weights(h, static_cast<const S8 *>(q), a, M, y, ldy, w, nullptr, st);
    });
    QVGGT_GUARD_END
}

// (X_calib, W, alpha, lo, hi) -> c
PyObject *calibrate_smooth(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    const Tensor &X = in.tensor(), &W = in.tensor();
    const float alpha = (float)in.real(), lo = (float)in.real(), hi = (float)in.real();
    if (!in.done() || X.dim() != 2 || W.dim() != 2 || X.element_size() != 2 || W.element_size() != 2 || !X.is_contiguous() || !W.is_contiguous() ||
        X.size(1) != W.size(1) || X.size(0) > INT32_MAX || W.size(0) > INT32_MAX || W.size(1) > INT32_MAX)
        Py_RETURN_NONE;
    const int64_t K = W.size(1);
    const Tensor scratch = at::empty({2 * K}, W.options().dtype(at::kFloat)), c = at::empty({K}, W.options().dtype(at::kFloat));
    const void *x = X.data_ptr(), *w = W.data_ptr();
    float *s = static_cast<float *>(scratch.data_ptr()), *out = static_cast<float *>(c.data_ptr());
    void *st = stream();
    const int Mc = (int)X.size(0), N = (int)W.size(0);
    if (without_gil([&] { return qvggt_calibrate_smooth(x, Mc, w, N, (int)K, alpha, lo, hi, s, out, st); }) != QVGGT_OK) Py_RETURN_NONE;
    return THPVariable_Wrap(c);
    QVGGT_GUARD_END
}

// (W, bias, smooth_c, sign_v, flags) -> handle as an integer
PyObject *prepare_weights(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    QVGGT_GUARD_BEGIN
    Args in{args, n};
    const Tensor &W = in.tensor(), &bias = in.tensor(true), &c = in.tensor(), &v = in.tensor(true);
    const int flags = (int)in.integer();
    if (!in.done() || W.dim() != 2 || W.element_size() != 2 || !W.is_contiguous() || W.size(0) > INT32_MAX || W.size(1) > INT32_MAX) Py_RETURN_NONE;
    const int64_t N = W.size(0), K = W.size(1);
    if (c.scalar_type() != at::kFloat || c.numel() != K || !c.is_contiguous()) Py_RETURN_NONE;
    if (bias.defined() && (bias.element_size() != 2 || bias.numel() != N || !bias.is_contiguous())) Py_RETURN_NONE;
    if (v.defined() && (v.scalar_type() != at::kChar || v.numel() != K || !v.is_contiguous())) Py_RETURN_NONE;
    const void *w = W.data_ptr(), *b = bias.defined() ? bias.data_ptr() : nullptr;
    const float *cp = static_cast<const float *>(c.data_ptr());
    const S8 *vp = v.defined() ? static_cast<const S8 *>(v.data_ptr()) : nullptr;
    void *st = stream();
    qvggt_weights_t *h = nullptr;
    if (without_gil([&] { return qvggt_prepare_weights(w, b, cp, vp, (int)N, (int)K, flags, st, &h); }) != QVGGT_OK) Py_RETURN_NONE;
    return PyLong_FromVoidPtr(h);
    QVGGT_GUARD_END
}

// Copy of a device array as a new tensor on the current device (d1 < 0: one dimension), undefined for a null pointer.  The array lies
// on the device of its handle, which need not be the current one.
Tensor copy_array(const void *p, ScalarType type, int64_t d0, int64_t d1)
{
    if (!p) return Tensor();
    const auto options = at::TensorOptions().dtype(type).device(at::kCUDA);
    void *q = const_cast<void *>(p);
    const Tensor t = d1 < 0 ? at::from_blob(q, {d0}, options) : at::from_blob(q, {d0, d1}, options);
    const at::Device here(at::kCUDA, c10::cuda::getCurrentCUDAStream().device_index());
    return t.device() == here ? t.clone() : t.to(here);
}

PyObject *wrap_or_none(const Tensor &t)
{
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}

// The two views have no other route: what goes wrong in them (out of memory, say) is raised as it is.

// (handle) -> copies (wq, w_scale, amul, bias), None where the handle has no such array
PyObject *weights_view(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    Args in{args, n};
    auto *h = in.handle();
    const U8 *wq = nullptr;
    const float *ws = nullptr, *am = nullptr;
    const void *bias = nullptr;
    int N = 0, K = 0;
    if (!in.done() || qvggt_weights_view(h, &wq, &ws, &am, &bias, &N, &K) != QVGGT_OK) Py_RETURN_NONE;
    const Tensor a = copy_array(wq, at::kByte, N, K / 2), b = copy_array(ws, at::kFloat, N, -1), c = copy_array(am, at::kFloat, K, -1),
                 d = copy_array(bias, at::kBFloat16, N, -1);
    return release_items(PyTuple_Pack(4, wrap_or_none(a), wrap_or_none(b), wrap_or_none(c), wrap_or_none(d)));
    END_HANDLE_TH_ERRORS
}

// (handle, N, K) -> (copy of the codes one per byte or None, code width)
PyObject *weights_view_c8(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    HANDLE_TH_ERRORS
    Args in{args, n};
    auto *h = in.handle();
    const int64_t N = in.integer(), K = in.integer();
    const S8 *wq8 = nullptr;
    int bits = 0;
    if (!in.done() || qvggt_weights_view_c8(h, &wq8, &bits) != QVGGT_OK) Py_RETURN_NONE;
    const Tensor codes = copy_array(wq8, at::kChar, N, K);
    return release_items(PyTuple_Pack(2, wrap_or_none(codes), PyLong_FromLong(bits)));
    END_HANDLE_TH_ERRORS
}

#define FAST(name, fn) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(static_cast<PyObject *(*)(PyObject *, PyObject *const *, Py_ssize_t)>(fn))), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("rotate_smooth_quantize", rotate_smooth_quantize),
    FAST("w4a4_linear", w4a4_linear),
    FAST("rotate_smooth_quantize_c8", (quantize_c8<qvggt_rotate_smooth_quantize_c8, false>)),
    FAST("rotate_smooth_quantize_c8_grouped", (quantize_c8<qvggt_rotate_smooth_quantize_c8_grouped, true>)),
    FAST("gelu_rotate_smooth_quantize_c8", (quantize_c8<qvggt_gelu_rotate_smooth_quantize_c8, false>)),
    FAST("layernorm_rotate_smooth_quantize_c8", layernorm_rotate_smooth_quantize_c8),
    FAST("rotate_smooth_quantize_static_c8", rotate_smooth_quantize_static_c8),
    FAST("rotate_smooth_quantize_tc", rotate_smooth_quantize_tc),
    FAST("rotate_smooth_quantize_c8_expand", rotate_smooth_quantize_c8_expand),
    FAST("w4a4_linear_c8", (linear_c8<qvggt_w4a4_linear_c8, false>)),
    FAST("w4a4_linear_c8_grouped", (linear_c8<qvggt_w4a4_linear_c8_grouped, true>)),
    FAST("w4a4_linear_c8_packed_weights", (linear_scratch<false>)),
    FAST("w4a4_linear_c8_expanded", (linear_scratch<true>)),
    FAST("calibrate_smooth", calibrate_smooth),
    FAST("prepare_weights", prepare_weights),
    FAST("weights_view", weights_view),
    FAST("weights_view_c8", weights_view_c8),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_qvggt_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__qvggt_fastcall() { return PyModule_Create(&module); }
