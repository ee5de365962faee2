// The calls of binding.py without its Python marshalling: each function takes the arguments of the Python function of the
// same name in order (all positional, stream left out), checks them, allocates the outputs that were not given and calls
// the C ABI on torch's current stream.  It does so only for arguments in the ordinary form (exact torch tensors on
// the device, right type, contiguous); anything else gets NotImplemented back, and the Python form of the call, which
// names the fault or takes the unusual argument, runs instead.  A q8_linear in Python cost 8 us per call before the
// first launch, more than the kernels of a small layer take.

#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <limits>

#include "q8.h"

namespace {

// ---- the C ABI, bound to the addresses in the library that binding.py has loaded
#define Q8_CALLS(X)                                                                                                    \
    X(q8_quantize_weight) X(q8_fake_quantize) X(q8_ste_backward) X(q8_calibrate) X(q8_linear)  \
    X(q8_linear_workspace_bytes) X(q8_linear_q) X(q8_linear_requant) X(q8_linear_q_requant) X(q8_linear_dyn)            \
    X(q8_embedding) X(q8_add_layernorm) X(q8_add_layernorm_quant) X(q8_add_layernorm_absmax) X(q8_attention)            \
    X(q8_attention_quant) X(q8_attention_absmax) X(q8_embed_layernorm)
#define Q8_DECLARE(name) decltype(&::name) p_##name = nullptr;
Q8_CALLS(Q8_DECLARE)
PyObject *g_check = nullptr;  // binding._check(status, where): raises

constexpr auto kF32 = at::kFloat;
constexpr auto kI8 = at::kChar;
constexpr auto kI32 = at::kInt;

struct Call {
    bool plain = true;  // every argument so far is in the ordinary form

    const at::Tensor *tensor(PyObject *o)
    {
        if (!THPVariable_CheckExact(o)) {
            plain = false;
            return nullptr;
        }
        return &THPVariable_Unpack(o);
    }
    // pointer of an optional tensor of the given type (nullptr for None)
    template <typename T = void>
    T *ptr(PyObject *o, at::ScalarType type)
    {
        if (o == Py_None) return nullptr;
        const at::Tensor *t = tensor(o);
        if (t == nullptr) return nullptr;
        if (!t->is_cuda() || t->scalar_type() != type || !t->is_contiguous()) {
            plain = false;
            return nullptr;
        }
        return static_cast<T *>(t->data_ptr());
    }
    // the same for a tensor of which `values` values are read
    template <typename T>
    T *covering(PyObject *o, at::ScalarType type, int64_t values)
    {
        T *p = ptr<T>(o, type);
        if (plain && o != Py_None && THPVariable_Unpack(o).numel() < values) plain = false;
        return p;
    }
    void *any_ptr(PyObject *o, size_t *bytes = nullptr)
    {
        const at::Tensor *t = tensor(o);
        if (t == nullptr || !t->is_cuda() || !t->is_contiguous()) {
            plain = false;
            return nullptr;
        }
        if (bytes != nullptr) *bytes = (size_t)t->numel() * t->element_size();
        return t->data_ptr();
    }
    bool matrix(PyObject *o, int64_t *rows, int64_t *cols)
    {
        const at::Tensor *t = tensor(o);
        if (t == nullptr || t->dim() != 2) return plain = false;
        *rows = t->size(0);
        *cols = t->size(1);
        return true;
    }
    int64_t integer(PyObject *o)
    {
        const int64_t v = PyLong_CheckExact(o) ? PyLong_AsLongLong(o) : (plain = false, 0);
        if (v == -1 && PyErr_Occurred()) {
            PyErr_Clear();
            plain = false;
        }
        return v;
    }
    int small(PyObject *o)
    {
        const int64_t v = integer(o);
        if (v < std::numeric_limits<int>::min() || v > std::numeric_limits<int>::max()) plain = false;
        return (int)v;
    }
    float real(PyObject *o)
    {
        if (!PyFloat_CheckExact(o)) return plain = false, 0.0f;
        return (float)PyFloat_AS_DOUBLE(o);
    }
};

void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor device_tensor(at::IntArrayRef shape, at::ScalarType type, PyObject *like)
{
    return at::empty(shape, at::TensorOptions().dtype(type).device(THPVariable_Unpack(like).device()));
}

PyObject *other_form() { return Py_NewRef(Py_NotImplemented); }

bool failed(q8_status st, const char *where)
{
    if (st == Q8_OK) return false;
    PyObject *r = PyObject_CallFunction(g_check, "is", (int)st, where);
    Py_XDECREF(r);
    return true;
}

// Runs a call without the interpreter lock; nullptr (exception set) when it fails.
template <typename F>
bool run(const char *where, F f)
{
    q8_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f(current_stream());
    Py_END_ALLOW_THREADS
    return !failed(st, where);
}

// An output that the caller gave, or a new tensor (of a shape, or like an input).
struct Output {
    PyObject *given;
    at::Tensor made;
    Output(Call &c, PyObject *o, PyObject *like) : given(o)
    {
        if (o == Py_None && c.plain) made = at::empty_like(THPVariable_Unpack(like));
    }
    Output(Call &c, PyObject *o, at::IntArrayRef shape, at::ScalarType type, PyObject *like) : given(o)
    {
        if (o == Py_None && c.plain) made = device_tensor(shape, type, like);
    }
    template <typename T>
    T *ptr(Call &c, at::ScalarType type)
    {
        return given == Py_None ? (made.defined() ? static_cast<T *>(made.data_ptr()) : nullptr) : c.ptr<T>(given, type);
    }
    PyObject *result() { return given == Py_None ? THPVariable_Wrap(made) : Py_NewRef(given); }
};

using Args = PyObject *const *;

// X [M, K] and Wq [N, K] of a layer
bool layer_shape(Call &c, PyObject *X, PyObject *Wq, int64_t *M, int64_t *N, int64_t *K)
{
    int64_t K2 = 0;
    if (!c.matrix(X, M, K) || !c.matrix(Wq, N, &K2) || K2 != *K) c.plain = false;
    return c.plain;
}
struct Workspace {
    at::Tensor made;
    void *ptr = nullptr;
    size_t bytes = 0;
    Workspace(Call &c, PyObject *o, PyObject *X, int64_t M, int64_t N, int64_t K)
    {
        if (!c.plain) return;
        if (o == Py_None) {
            bytes = p_q8_linear_workspace_bytes(M, N, K);
            made = device_tensor({(int64_t)bytes}, at::kByte, X);
            ptr = made.data_ptr();
        } else {
            ptr = c.any_ptr(o, &bytes);
        }
    }
};

// (X, Wq, S_w, S_x, bias, act, Y, workspace, dbg_Xq, dbg_acc)
PyObject *linear(Args a)
{
    Call c;
    int64_t M, N, K;
    if (!layer_shape(c, a[0], a[1], &M, &N, &K)) return other_form();
    auto X = c.ptr<const float>(a[0], kF32);
    auto Wq = c.ptr<const int8_t>(a[1], kI8);
    auto S_w = c.ptr<const float>(a[2], kF32), S_x = c.ptr<const float>(a[3], kF32), bias = c.ptr<const float>(a[4], kF32);
    const int act = c.small(a[5]);
    auto dbg_Xq = c.ptr<int8_t>(a[8], kI8);
    auto dbg_acc = c.ptr<int32_t>(a[9], kI32);
    Output Y(c, a[6], {M, N}, kF32, a[0]);
    auto y = Y.ptr<float>(c, kF32);
    Workspace ws(c, a[7], a[0], M, N, K);
    if (!c.plain) return other_form();
    if (!run("q8_linear", [&](void *s) { return p_q8_linear(X, Wq, S_w, S_x, bias, act, y, M, N, K, ws.ptr, ws.bytes, dbg_Xq, dbg_acc, s); }))
        return nullptr;
    return Y.result();
}

// (Xq, S_x, Wq, S_w, bias, act, Y, dbg_acc, dev_status)
PyObject *linear_q(Args a)
{
    Call c;
    int64_t M, N, K;
    if (!layer_shape(c, a[0], a[2], &M, &N, &K)) return other_form();
    auto Xq = c.ptr<const int8_t>(a[0], kI8), Wq = c.ptr<const int8_t>(a[2], kI8);
    auto S_x = c.ptr<const float>(a[1], kF32), S_w = c.ptr<const float>(a[3], kF32), bias = c.ptr<const float>(a[4], kF32);
    const int act = c.small(a[5]);
    auto dbg_acc = c.ptr<int32_t>(a[7], kI32), status = c.ptr<int32_t>(a[8], kI32);
    Output Y(c, a[6], {M, N}, kF32, a[0]);
    auto y = Y.ptr<float>(c, kF32);
    if (!c.plain) return other_form();
    if (!run("q8_linear_q", [&](void *s) { return p_q8_linear_q(Xq, S_x, Wq, S_w, bias, act, y, M, N, K, dbg_acc, status, s); }))
        return nullptr;
    return Y.result();
}

// (X, Wq, S_w, S_x, bias, act, S_y, Yq, Y, workspace, dbg_Xq, dbg_acc)
PyObject *linear_requant(Args a)
{
    Call c;
    int64_t M, N, K;
    if (!layer_shape(c, a[0], a[1], &M, &N, &K)) return other_form();
    auto X = c.ptr<const float>(a[0], kF32);
    auto Wq = c.ptr<const int8_t>(a[1], kI8);
    auto S_w = c.ptr<const float>(a[2], kF32), S_x = c.ptr<const float>(a[3], kF32), bias = c.ptr<const float>(a[4], kF32),
         S_y = c.ptr<const float>(a[6], kF32);
    const int act = c.small(a[5]);
    auto y = c.ptr<float>(a[8], kF32);
    auto dbg_Xq = c.ptr<int8_t>(a[10], kI8);
    auto dbg_acc = c.ptr<int32_t>(a[11], kI32);
    Output Yq(c, a[7], {M, N}, kI8, a[0]);
    auto yq = Yq.ptr<int8_t>(c, kI8);
    Workspace ws(c, a[9], a[0], M, N, K);
    if (!c.plain) return other_form();
    if (!run("q8_linear_requant", [&](void *s) {
            return p_q8_linear_requant(X, Wq, S_w, S_x, bias, act, S_y, yq, y, M, N, K, ws.ptr, ws.bytes, dbg_Xq, dbg_acc, s);
        }))
        return nullptr;
    return Yq.result();
}

// (Xq, S_x, Wq, S_w, bias, act, S_y, Yq, Y, dbg_acc, dev_status)
PyObject *linear_q_requant(Args a)
{
    Call c;
    int64_t M, N, K;
    if (!layer_shape(c, a[0], a[2], &M, &N, &K)) return other_form();
    auto Xq = c.ptr<const int8_t>(a[0], kI8), Wq = c.ptr<const int8_t>(a[2], kI8);
    auto S_x = c.ptr<const float>(a[1], kF32), S_w = c.ptr<const float>(a[3], kF32), bias = c.ptr<const float>(a[4], kF32),
         S_y = c.ptr<const float>(a[6], kF32);
    const int act = c.small(a[5]);
    auto y = c.ptr<float>(a[8], kF32);
    auto dbg_acc = c.ptr<int32_t>(a[9], kI32), status = c.ptr<int32_t>(a[10], kI32);
    Output Yq(c, a[7], {M, N}, kI8, a[0]);
    auto yq = Yq.ptr<int8_t>(c, kI8);
    if (!c.plain) return other_form();
    if (!run("q8_linear_q_requant", [&](void *s) {
            return p_q8_linear_q_requant(Xq, S_x, Wq, S_w, bias, act, S_y, yq, y, M, N, K, dbg_acc, status, s);
        }))
        return nullptr;
    return Yq.result();
}

// (X, x_absmax, Wq, S_w, bias, act, Y, y_absmax, workspace, dbg_Xq, dbg_acc)
PyObject *linear_dyn(Args a)
{
    Call c;
    int64_t M, N, K;
    if (!layer_shape(c, a[0], a[2], &M, &N, &K)) return other_form();
    auto X = c.ptr<const float>(a[0], kF32);
    auto xw = c.ptr<const uint32_t>(a[1], kI32);
    auto Wq = c.ptr<const int8_t>(a[2], kI8);
    auto S_w = c.ptr<const float>(a[3], kF32), bias = c.ptr<const float>(a[4], kF32);
    const int act = c.small(a[5]);
    auto yw = c.ptr<uint32_t>(a[7], kI32);
    auto dbg_Xq = c.ptr<int8_t>(a[9], kI8);
    auto dbg_acc = c.ptr<int32_t>(a[10], kI32);
    Output Y(c, a[6], {M, N}, kF32, a[0]);
    auto y = Y.ptr<float>(c, kF32);
    Workspace ws(c, a[8], a[0], M, N, K);
    if (!c.plain) return other_form();
    if (!run("q8_linear_dyn", [&](void *s) {
            return p_q8_linear_dyn(X, xw, Wq, S_w, bias, act, y, yw, M, N, K, ws.ptr, ws.bytes, dbg_Xq, dbg_acc, s);
        }))
        return nullptr;
    return Y.result();
}

// (ids, Eq, S_e, out, rows_q, dev_status)
PyObject *embedding(Args a)
{
    Call c;
    int64_t V, H;
    const at::Tensor *t = c.tensor(a[0]);
    if (t == nullptr || !c.matrix(a[1], &V, &H)) return other_form();
    const int64_t T = t->numel();
    auto ids = c.ptr<const int32_t>(a[0], kI32);
    auto Eq = c.ptr<const int8_t>(a[1], kI8);
    auto S_e = c.ptr<const float>(a[2], kF32);
    auto rows_q = c.ptr<int8_t>(a[4], kI8);
    auto status = c.ptr<int32_t>(a[5], kI32);
    Output out(c, a[3], {T, H}, kF32, a[1]);
    auto o = out.ptr<float>(c, kF32);
    if (!c.plain) return other_form();
    if (!run("q8_embedding", [&](void *s) { return p_q8_embedding(ids, T, Eq, S_e, V, H, o, rows_q, status, s); })) return nullptr;
    return out.result();
}

// (x, r1, r2, gamma, beta, eps, out, S_q, out_q, absmax_bits): plain (S_q, absmax_bits None), quantising or folding max|out|
template <int KIND>
PyObject *add_layernorm(Args a)
{
    Call c;
    int64_t rows, H;
    if (!c.matrix(a[0], &rows, &H)) return other_form();
    auto x = c.ptr<const float>(a[0], kF32), r1 = c.covering<const float>(a[1], kF32, rows * H),
         r2 = c.covering<const float>(a[2], kF32, rows * H), gamma = c.covering<const float>(a[3], kF32, H),
         beta = c.covering<const float>(a[4], kF32, H), S_q = c.ptr<const float>(a[7], kF32);
    const float eps = c.real(a[5]);
    auto word = c.ptr<uint32_t>(a[9], kI32);
    if (KIND == 1) {
        auto o = c.ptr<float>(a[6], kF32);
        Output out_q(c, a[8], {rows, H}, kI8, a[0]);
        auto oq = out_q.ptr<int8_t>(c, kI8);
        if (!c.plain) return other_form();
        if (!run("q8_add_layernorm_quant", [&](void *s) { return p_q8_add_layernorm_quant(x, r1, r2, gamma, beta, eps, rows, H, o, S_q, oq, s); }))
            return nullptr;
        return out_q.result();
    }
    Output out(c, a[6], {rows, H}, kF32, a[0]);
    auto o = out.ptr<float>(c, kF32);
    if (!c.plain) return other_form();
    if (!(KIND == 0 ? run("q8_add_layernorm", [&](void *s) { return p_q8_add_layernorm(x, r1, r2, gamma, beta, eps, rows, H, o, s); })
                    : run("q8_add_layernorm_absmax", [&](void *s) {
                          return p_q8_add_layernorm_absmax(x, r1, r2, gamma, beta, eps, rows, H, o, word, s);
                      })))
        return nullptr;
    return out.result();
}

// (qkv, B, S, heads, ctx, S_q, ctx_q, absmax_bits)
template <int KIND>
PyObject *attention(Args a)
{
    Call c;
    int64_t T, W;
    if (!c.matrix(a[0], &T, &W)) return other_form();
    const int64_t B = c.integer(a[1]), S = c.integer(a[2]), heads = c.integer(a[3]);
    if (!c.plain || B < 0 || S < 0 || heads < 0 || heads > 65535 || B > 65535 || S > (int64_t(1) << 31) || B * S != T ||
        heads * 192 != W)
        return other_form();
    const int64_t H = heads * 64;
    auto qkv = c.ptr<const float>(a[0], kF32);
    auto S_q = c.ptr<const float>(a[5], kF32);
    auto word = c.ptr<uint32_t>(a[7], kI32);
    if (KIND == 1) {
        auto ctx = c.ptr<float>(a[4], kF32);
        Output ctx_q(c, a[6], {T, H}, kI8, a[0]);
        auto cq = ctx_q.ptr<int8_t>(c, kI8);
        if (!c.plain) return other_form();
        if (!run("q8_attention_quant", [&](void *s) { return p_q8_attention_quant(qkv, B, S, heads, ctx, S_q, cq, s); })) return nullptr;
        return ctx_q.result();
    }
    Output out(c, a[4], {T, H}, kF32, a[0]);
    auto ctx = out.ptr<float>(c, kF32);
    if (!c.plain) return other_form();
    if (!(KIND == 0 ? run("q8_attention", [&](void *s) { return p_q8_attention(qkv, B, S, heads, ctx, s); })
                    : run("q8_attention_absmax", [&](void *s) { return p_q8_attention_absmax(qkv, B, S, heads, ctx, word, s); })))
        return nullptr;
    return out.result();
}

// (ids, S, word, S_word, pos, S_pos, typ, S_typ, eps, out, S_q, out_q, absmax_bits, dev_status)
PyObject *embed_layernorm(Args a)
{
    Call c;
    int64_t V, H, P, H2, rows, H3;
    const at::Tensor *t = c.tensor(a[0]);
    if (t == nullptr || !c.matrix(a[2], &V, &H) || !c.matrix(a[4], &P, &H2) || !c.matrix(a[6], &rows, &H3) || H2 != H || H3 != H ||
        rows < 1 || (a[9] == Py_None && a[11] == Py_None))
        return other_form();
    const int64_t T = t->numel(), S = c.integer(a[1]);
    auto ids = c.ptr<const int32_t>(a[0], kI32);
    auto word = c.ptr<const int8_t>(a[2], kI8), pos = c.ptr<const int8_t>(a[4], kI8), typ = c.ptr<const int8_t>(a[6], kI8);
    auto S_word = c.ptr<const float>(a[3], kF32), S_pos = c.ptr<const float>(a[5], kF32), S_typ = c.ptr<const float>(a[7], kF32);
    const float eps = c.real(a[8]);
    auto out = c.ptr<float>(a[9], kF32);
    auto S_q = c.ptr<const float>(a[10], kF32);
    auto out_q = c.ptr<int8_t>(a[11], kI8);
    auto peak = c.ptr<uint32_t>(a[12], kI32);
    auto status = c.ptr<int32_t>(a[13], kI32);
    if (!c.plain) return other_form();
    if (!run("q8_embed_layernorm", [&](void *s) {
            return p_q8_embed_layernorm(ids, T, S, word, S_word, V, pos, S_pos, P, typ, S_typ, eps, H, out, S_q, out_q, peak, status, s);
        }))
        return nullptr;
    return Py_NewRef(a[9] != Py_None ? a[9] : a[11]);
}

// (W, Wq, S_w, dev_status) -> (Wq, S_w)
PyObject *quantize_weight(Args a)
{
    Call c;
    int64_t N, K;
    if (!c.matrix(a[0], &N, &K)) return other_form();
    auto W = c.ptr<const float>(a[0], kF32);
    auto status = c.ptr<int32_t>(a[3], kI32);
    Output Wq(c, a[1], {N, K}, kI8, a[0]), S_w(c, a[2], {1}, kF32, a[0]);
    auto wq = Wq.ptr<int8_t>(c, kI8);
    auto sw = S_w.ptr<float>(c, kF32);
    if (!c.plain) return other_form();
    if (!run("q8_quantize_weight", [&](void *s) { return p_q8_quantize_weight(W, N, K, wq, sw, status, s); })) return nullptr;
    PyObject *q = Wq.result(), *w = S_w.result();
    PyObject *r = PyTuple_Pack(2, q, w);
    Py_DECREF(q);
    Py_DECREF(w);
    return r;
}

// (X, decay, state)
PyObject *calibrate(Args a)
{
    Call c;
    const at::Tensor *t = c.tensor(a[0]);
    if (t == nullptr) return other_form();
    const int64_t n = t->numel();
    auto X = c.ptr<const float>(a[0], kF32);
    const float decay = c.real(a[1]);
    void *state = c.any_ptr(a[2]);
    if (!c.plain) return other_form();
    if (!run("q8_calibrate", [&](void *s) { return p_q8_calibrate(X, n, decay, state, s); })) return nullptr;
    Py_RETURN_NONE;
}

// (X, S, Xhat)
PyObject *fake_quantize(Args a)
{
    Call c;
    const at::Tensor *t = c.tensor(a[0]);
    if (t == nullptr) return other_form();
    auto X = c.ptr<const float>(a[0], kF32), S = c.ptr<const float>(a[1], kF32);
    Output out(c, a[2], a[0]);
    auto o = out.ptr<float>(c, kF32);
    const int64_t n = t->numel();
    if (!c.plain) return other_form();
    if (!run("q8_fake_quantize", [&](void *s) { return p_q8_fake_quantize(X, n, S, o, s); })) return nullptr;
    return out.result();
}

// (grad_out, grad_in)
PyObject *ste_backward(Args a)
{
    Call c;
    const at::Tensor *t = c.tensor(a[0]);
    if (t == nullptr) return other_form();
    auto g = c.ptr<const float>(a[0], kF32);
    Output out(c, a[1], a[0]);
    auto o = out.ptr<float>(c, kF32);
    const int64_t n = t->numel();
    if (!c.plain) return other_form();
    if (!run("q8_ste_backward", [&](void *s) { return p_q8_ste_backward(g, n, o, s); })) return nullptr;
    return out.result();
}

// A C++ exception (a tensor without storage, an allocation that fails) leaves the call to its Python form.
template <PyObject *(*F)(Args), int COUNT>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t count)
{
    if (count != COUNT) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", COUNT, count);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const std::exception &) {
        return other_form();
    }
}

// bind(address of each call, _check)
PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t count)
{
    if (count != 2 || !PyDict_Check(args[0])) {
        PyErr_SetString(PyExc_TypeError, "bind(addresses, check)");
        return nullptr;
    }
#define Q8_BIND(name)                                                                          \
    {                                                                                          \
        PyObject *v = PyDict_GetItemString(args[0], #name);                                    \
        void *p = v != nullptr ? PyLong_AsVoidPtr(v) : nullptr;                                \
        if (p == nullptr) {                                                                    \
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_KeyError, #name);                     \
            return nullptr;                                                                    \
        }                                                                                      \
        p_##name = reinterpret_cast<decltype(p_##name)>(p);                                    \
    }
    Q8_CALLS(Q8_BIND)
    Py_XSETREF(g_check, Py_NewRef(args[1]));
    Py_RETURN_NONE;
}

#define Q8_ENTRY(name, function, count) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&entry<function, count>)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&bind)), METH_FASTCALL, nullptr},
    Q8_ENTRY("linear", linear, 10),
    Q8_ENTRY("linear_q", linear_q, 9),
    Q8_ENTRY("linear_requant", linear_requant, 12),
    Q8_ENTRY("linear_q_requant", linear_q_requant, 11),
    Q8_ENTRY("linear_dyn", linear_dyn, 11),
    Q8_ENTRY("embedding", embedding, 6),
    Q8_ENTRY("add_layernorm", add_layernorm<0>, 10),
    Q8_ENTRY("add_layernorm_quant", add_layernorm<1>, 10),
    Q8_ENTRY("add_layernorm_absmax", add_layernorm<2>, 10),
    Q8_ENTRY("attention", attention<0>, 8),
    Q8_ENTRY("attention_quant", attention<1>, 8),
    Q8_ENTRY("attention_absmax", attention<2>, 8),
    Q8_ENTRY("embed_layernorm", embed_layernorm, 14),
    Q8_ENTRY("quantize_weight", quantize_weight, 4),
    Q8_ENTRY("calibrate", calibrate, 3),
    Q8_ENTRY("fake_quantize", fake_quantize, 3),
    Q8_ENTRY("ste_backward", ste_backward, 2),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_q8_native", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

#define Q8_STRING(x) #x
#define Q8_VALUE(x) Q8_STRING(x)
// build.py looks for this in the file, binding.py asks the module: torch's ABI holds for one version
extern "C" __attribute__((visibility("default"), used)) const char q8_native_built_for[] =
    "q8 native for torch " Q8_TORCH_VERSION ", python " Q8_VALUE(PY_MAJOR_VERSION) "." Q8_VALUE(PY_MINOR_VERSION);

PyMODINIT_FUNC PyInit__q8_native()
{
    PyObject *m = PyModule_Create(&kModule);
    if (m != nullptr && PyModule_AddStringConstant(m, "built_for", Q8_TORCH_VERSION) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
