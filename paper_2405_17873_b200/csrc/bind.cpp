// CPython binding of the C ABI's layer calls and tensor helpers (module _mixdq_native).
//
// A layer of a few-step UNet runs for 5 to 10 microseconds on the GPU, and a step has some 800 of them: what a call
// costs on the host is what it costs.  Marshalling the same calls through ctypes from Python (seventeen converted
// arguments, torch.empty, torch.cuda.current_stream, shape and stride look-ups) took 13 to 15 us of host time per
// layer; here the arguments are read from the tensor objects directly.  Nothing else happens in this file: every step
// of the path runs in the library's kernels.
//
// Functions take their arguments by position or by name, exactly like the Python functions whose signatures stand in
// their docstrings.  The global interpreter lock is released around the library call, which may block while the
// launch queue is full.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/mixdq.h"
#include "unlocked.h"

namespace {

PyObject* g_error = nullptr;  // paper_2405_17873_b200.mixdq.MixdqError

struct Failed {};  // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* text)
{
    PyErr_SetString(type, text);
    throw Failed{};
}

void check(int rc, const char* what)
{
    if (rc == MIXDQ_OK) return;
    PyErr_Format(g_error, "%s: %s (%d)", what, mixdq_strerror(rc), rc);
    throw Failed{};
}

// Arguments of one call, matched against a signature: `values[i]` is a borrowed reference or nullptr (default).
constexpr int kMaxArgs = 16;

struct Signature {
    const char* function;
    int required;
    int count;
    const char* names[kMaxArgs];
    PyObject* interned[kMaxArgs];
};

struct Args {
    PyObject* v[kMaxArgs];

    Args(Signature& sig, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames)
    {
        if (nargs > sig.count) {
            PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments", sig.function, sig.count);
            throw Failed{};
        }
        for (Py_ssize_t i = 0; i < nargs; ++i) v[i] = args[i];
        for (int i = static_cast<int>(nargs); i < sig.count; ++i) v[i] = nullptr;
        const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
        for (Py_ssize_t k = 0; k < nkw; ++k) {
            PyObject* key = PyTuple_GET_ITEM(kwnames, k);
            int at = -1;
            for (int i = 0; i < sig.count && at < 0; ++i)
                if (sig.interned[i] == key) at = i;
            for (int i = 0; i < sig.count && at < 0; ++i)
                if (PyUnicode_Compare(sig.interned[i], key) == 0) at = i;
            if (at < 0 || v[at]) {
                PyErr_Format(PyExc_TypeError, at < 0 ? "%s() got an unexpected keyword argument '%U'"
                                                     : "%s() got multiple values for argument '%U'",
                             sig.function, key);
                throw Failed{};
            }
            v[at] = args[nargs + k];
        }
        for (int i = 0; i < sig.required; ++i)
            if (!v[i]) {
                PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", sig.function, sig.names[i]);
                throw Failed{};
            }
    }

    bool given(int i) const { return v[i] && v[i] != Py_None; }

    const at::Tensor& tensor(int i) const
    {
        if (!given(i) || !THPVariable_Check(v[i])) raise(PyExc_TypeError, "a torch.Tensor is expected");
        return THPVariable_Unpack(v[i]);
    }

    // Device address of a tensor argument; nullptr where it is absent or None.
    void* ptr(int i) const { return given(i) ? address(tensor(i)) : nullptr; }
    template <typename T>
    T* as(int i) const
    {
        return static_cast<T*>(ptr(i));
    }

    static void* address(const at::Tensor& t)
    {
        if (!t.is_cuda() || !t.is_contiguous()) raise(PyExc_AssertionError, "device-resident contiguous tensors only");
        return const_cast<void*>(t.const_data_ptr());
    }

    int64_t integer(int i, int64_t otherwise = 0) const
    {
        if (!v[i]) return otherwise;
        const long long x = PyLong_AsLongLong(v[i]);
        if (x == -1 && PyErr_Occurred()) throw Failed{};
        return x;
    }
};

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor new_tensor(at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor& like)
{
    return at::detail::empty_cuda(shape, dtype, like.device(), std::nullopt);
}

// The `out` argument, or a new tensor: a Python object to return and its device address.
struct Output {
    PyObject* object;
    void* address;

    Output(const Args& a, int i, at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor& like)
    {
        if (i >= 0 && a.given(i)) {
            address = a.ptr(i);
            object = Py_NewRef(a.v[i]);
        } else {
            at::Tensor t = new_tensor(shape, dtype, like);
            address = const_cast<void*>(t.const_data_ptr());
            object = THPVariable_Wrap(std::move(t));
            if (!object) throw Failed{};
        }
    }
    ~Output() { Py_XDECREF(object); }
    Output(const Output&) = delete;
    PyObject* release()
    {
        PyObject* o = object;
        object = nullptr;
        return o;
    }
    int64_t stride(int d) const { return THPVariable_Unpack(object).stride(d); }
};

template <typename F>
void call(const char* what, F&& f)
{
    check(unlocked(f), what);
}

void need_dim(const at::Tensor& t, int dim)
{
    if (t.dim() != dim) {
        PyErr_Format(PyExc_ValueError, "a tensor of %d dimensions is expected, got %d", dim, static_cast<int>(t.dim()));
        throw Failed{};
    }
}

size_t bytes_of(const Args& a, int i) { return a.given(i) ? static_cast<size_t>(a.tensor(i).numel()) : 0; }

int64_t conv_out(int64_t size, int64_t stride) { return stride > 0 ? (size - 1) / stride + 1 : size; }

constexpr at::ScalarType kF16 = at::kHalf, kF32 = at::kFloat, kI32 = at::kInt, kU8 = at::kByte, kI8 = at::kChar;

// ---------------------------------------------------------------- weights

PyObject* weight_minmax_params(const Args& a)
{
    const at::Tensor& W = a.tensor(0);
    need_dim(W, 2);
    const int64_t N = W.size(0), K = W.size(1), bits = a.integer(1);
    const int symmetric = PyObject_IsTrue(a.v[2]);
    if (symmetric < 0) throw Failed{};
    Output scale(a, 3, {N}, kF32, W), zero(a, 4, {N}, kI32, W);
    void* st = current_stream();
    const void* w = a.ptr(0);
    call("mixdq_weight_minmax_params", [&] {
        return mixdq_weight_minmax_params(w, N, K, static_cast<int>(bits), symmetric, static_cast<float*>(scale.address),
                                          static_cast<int32_t*>(zero.address), st);
    });
    PyObject* pair = PyTuple_Pack(2, scale.object, zero.object);
    if (!pair) throw Failed{};
    return pair;
}

PyObject* pack_weights(const Args& a)
{
    const at::Tensor& W = a.tensor(0);
    need_dim(W, 2);
    const int64_t N = W.size(0), K = W.size(1);
    const int bits = static_cast<int>(a.integer(1)), layout = static_cast<int>(a.integer(4, MIXDQ_LAYOUT_DEVICE));
    size_t bytes = 0;
    if (!a.given(5)) check(mixdq_packed_bytes(N, K, bits, layout, &bytes), "mixdq_packed_bytes");
    Output out(a, 5, {static_cast<int64_t>(bytes)}, kU8, W);
    void* st = current_stream();
    const void* w = a.ptr(0);
    const float* scale = a.as<float>(2);
    const int32_t* zero = a.as<int32_t>(3);
    call("mixdq_pack_weights", [&] { return mixdq_pack_weights(w, N, K, bits, scale, zero, layout, out.address, st); });
    return out.release();
}

PyObject* weight_code_sums(const Args& a)
{
    const at::Tensor& P = a.tensor(0);
    const int64_t N = a.integer(1), K = a.integer(2), bits = a.integer(3);
    Output out(a, -1, {N}, kI32, P);
    void* st = current_stream();
    const void* p = a.ptr(0);
    call("mixdq_weight_code_sums", [&] {
        return mixdq_weight_code_sums(p, N, K, static_cast<int>(bits), static_cast<int32_t*>(out.address), st);
    });
    return out.release();
}

// ---------------------------------------------------------------- activation ranges

// X as a matrix of its last dimension's rows (a copy only where the tensor is not contiguous and cannot be viewed so).
struct Rows {
    at::Tensor held;
    const void* data;
    int64_t rows, cols;
    explicit Rows(const at::Tensor& X)
    {
        if (X.dim() == 0) raise(PyExc_IndexError, "a tensor of at least one dimension is expected");
        held = X.is_contiguous() ? X : X.reshape({-1, X.size(-1)});
        cols = X.size(-1);
        rows = cols ? held.numel() / cols : 0;
        data = Args::address(held);
    }
};

PyObject* act_absmax(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    Rows x(X);
    const int skip = static_cast<int>(a.integer(1));
    Output out(a, -1, {1}, kF32, X);
    void* st = current_stream();
    call("mixdq_act_absmax", [&] {
        return mixdq_act_absmax(x.data, x.rows, x.cols, x.cols, skip, static_cast<float*>(out.address), st);
    });
    return out.release();
}

PyObject* act_scale_from_absmax(const Args& a)
{
    const at::Tensor& amax = a.tensor(0);
    Output out(a, -1, {1}, kF32, amax);
    void* st = current_stream();
    const float* m = a.as<float>(0);
    call("mixdq_act_scale_from_absmax",
         [&] { return mixdq_act_scale_from_absmax(m, static_cast<float*>(out.address), st); });
    return out.release();
}

PyObject* act_scale(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    Rows x(X);
    const int skip = static_cast<int>(a.integer(1));
    Output out(a, -1, {1}, kF32, X);
    void* st = current_stream();
    call("mixdq_act_scale", [&] {
        return mixdq_act_scale(x.data, x.rows, x.cols, x.cols, skip, static_cast<float*>(out.address), st);
    });
    return out.release();
}

PyObject* act_minmax(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    Rows x(X);
    Output out(a, -1, {2}, kF32, X);
    void* st = current_stream();
    call("mixdq_act_minmax",
         [&] { return mixdq_act_minmax(x.data, x.rows, x.cols, x.cols, static_cast<float*>(out.address), st); });
    return out.release();
}

PyObject* act_asym_params(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    Rows x(X);
    Output scale(a, -1, {1}, kF32, X), zero(a, -1, {1}, kI32, X);
    void* st = current_stream();
    call("mixdq_act_asym_params", [&] {
        return mixdq_act_asym_params(x.data, x.rows, x.cols, x.cols, static_cast<float*>(scale.address),
                                     static_cast<int32_t*>(zero.address), st);
    });
    PyObject* pair = PyTuple_Pack(2, scale.object, zero.object);
    if (!pair) throw Failed{};
    return pair;
}

// ---------------------------------------------------------------- linear layers

PyObject* linear(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t M = X.size(0), K = X.size(1), N = a.integer(2), ldx = X.stride(0);
    const int w_bits = static_cast<int>(a.integer(3)), act_bits = static_cast<int>(a.integer(6, 8));
    Output y(a, 11, {M, N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(8);
    const float *ws = a.as<float>(4), *sx = a.as<float>(7);
    const int32_t* wz = a.as<int32_t>(5);
    void *space = a.ptr(9), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 9);
    int32_t* status = a.as<int32_t>(10);
    call("mixdq_linear", [&] {
        return mixdq_linear(x, M, K, ldx, w, N, w_bits, ws, wz, act_bits, sx, bias, y.address, space, space_bytes, status, st);
    });
    return y.release();
}

PyObject* linear_a8_asym(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t M = X.size(0), K = X.size(1), N = a.integer(2), ldx = X.stride(0);
    const int w_bits = static_cast<int>(a.integer(3));
    Output y(a, 11, {M, N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(8);
    const float *ws = a.as<float>(4), *sx = a.as<float>(6);
    const int32_t *sums = a.as<int32_t>(5), *zx = a.as<int32_t>(7);
    void *space = a.ptr(9), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 9);
    int32_t* status = a.as<int32_t>(10);
    call("mixdq_linear_a8_asym", [&] {
        return mixdq_linear_a8_asym(x, M, K, ldx, w, N, w_bits, ws, sums, sx, zx, bias, y.address, space, space_bytes, status, st);
    });
    return y.release();
}

PyObject* quantize_acts(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t rows = X.size(0), K = X.size(1), ldx = X.stride(0);
    Output out(a, 2, {rows, K}, kI8, X);
    if (X.stride(1) != 1 || !X.is_cuda()) raise(PyExc_AssertionError, "device-resident rows of adjacent elements only");
    const void* x = X.const_data_ptr();  // (the rows themselves may be apart)
    const float* sx = a.as<float>(1);
    void* st = current_stream();
    call("mixdq_quantize_acts", [&] { return mixdq_quantize_acts(x, rows, K, ldx, sx, out.address, st); });
    return out.release();
}

PyObject* linear_q8(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t M = X.size(0), K = X.size(1), N = a.integer(2);
    const int w_bits = static_cast<int>(a.integer(3));
    Output y(a, 8, {M, N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(6);
    const float *ws = a.as<float>(4), *sx = a.as<float>(5);
    int32_t* status = a.as<int32_t>(7);
    void* st = current_stream();
    call("mixdq_linear_q8", [&] { return mixdq_linear_q8(x, M, K, w, N, w_bits, ws, sx, bias, y.address, status, st); });
    return y.release();
}

PyObject* linear_a8_fused_quant(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t M = X.size(0), K = X.size(1), N = a.integer(2), ldx = X.stride(0);
    const int w_bits = static_cast<int>(a.integer(3)), cols = static_cast<int>(a.integer(7, 128));
    Output y(a, 9, {M, N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(6);
    const float *ws = a.as<float>(4), *sx = a.as<float>(5);
    int32_t* status = a.as<int32_t>(8);
    const int64_t ldy = y.stride(0);
    void* st = current_stream();
    call("mixdq_linear_a8_fused_quant", [&] {
        return mixdq_linear_a8_fused_quant(x, M, K, ldx, w, N, w_bits, ws, sx, bias, y.address, ldy, cols, status, st);
    });
    return y.release();
}

PyObject* linear_a8_static_scratch(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t M = X.size(0), K = X.size(1), N = a.integer(2), ldx = X.stride(0);
    const int w_bits = static_cast<int>(a.integer(3));
    Output y(a, 8, {M, N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(6);
    const float *ws = a.as<float>(4), *sx = a.as<float>(5);
    int32_t* status = a.as<int32_t>(7);
    void* st = current_stream();
    call("mixdq_linear_a8_static_scratch", [&] {
        return mixdq_linear_a8_static_scratch(x, M, K, ldx, w, N, w_bits, ws, sx, bias, y.address, status, st);
    });
    return y.release();
}

PyObject* linear_a8_split(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 2);
    const int64_t M = X.size(0), K = X.size(1), at_ = a.integer(1), N = a.integer(4), ldx = X.stride(0);
    const int w_bits = static_cast<int>(a.integer(5));
    Output y(a, 12, {M, N}, kF16, X);
    const void *x = a.ptr(0), *lo = a.ptr(2), *hi = a.ptr(3), *bias = a.ptr(9);
    const float *ws = a.as<float>(6), *s_lo = a.as<float>(7), *s_hi = a.as<float>(8);
    void *space = a.ptr(10), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 10);
    int32_t* status = a.as<int32_t>(11);
    call("mixdq_linear_a8_split", [&] {
        return mixdq_linear_a8_split(x, M, K, ldx, at_, lo, hi, N, w_bits, ws, s_lo, s_hi, bias, y.address, space, space_bytes,
                                     status, st);
    });
    return y.release();
}

PyObject* crossattn_kv(const Args& a)
{
    const at::Tensor& E = a.tensor(0);
    need_dim(E, 3);
    const int64_t B = E.size(0), T = E.size(1), Kt = E.size(2), N = a.integer(2);
    if (T != MIXDQ_TOKENS_PER_PROMPT) raise(PyExc_AssertionError, "77 tokens per prompt are expected");
    const int w_bits = static_cast<int>(a.integer(3));
    Output y(a, 9, {B, T, N}, kF16, E);
    const void *x = a.ptr(0), *w = a.ptr(1), *bos = a.ptr(6);
    const float *ws = a.as<float>(4), *sx = a.as<float>(5);
    void *space = a.ptr(7), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 7);
    int32_t* status = a.as<int32_t>(8);
    call("mixdq_crossattn_kv", [&] {
        return mixdq_crossattn_kv(x, B, Kt, w, N, w_bits, ws, sx, bos, y.address, space, space_bytes, status, st);
    });
    return y.release();
}

// ---------------------------------------------------------------- convolutions

PyObject* conv3x3(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 4);
    const int64_t B = X.size(0), H = X.size(1), W = X.size(2), Cin = X.size(3), N = a.integer(2);
    const int w_bits = static_cast<int>(a.integer(3)), act_bits = static_cast<int>(a.integer(6, 8));
    const int stride = static_cast<int>(a.integer(9, 1));
    Output y(a, 12, {B, conv_out(H, stride), conv_out(W, stride), N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(8);
    const float *ws = a.as<float>(4), *sx = a.as<float>(7);
    const int32_t* wz = a.as<int32_t>(5);
    void *space = a.ptr(10), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 10);
    int32_t* status = a.as<int32_t>(11);
    call("mixdq_conv3x3", [&] {
        return mixdq_conv3x3(x, B, H, W, Cin, w, N, stride, w_bits, ws, wz, act_bits, sx, bias, y.address, space, space_bytes,
                             status, st);
    });
    return y.release();
}

PyObject* conv3x3_a8_asym(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 4);
    const int64_t B = X.size(0), H = X.size(1), W = X.size(2), Cin = X.size(3), N = a.integer(2);
    const int w_bits = static_cast<int>(a.integer(3)), stride = static_cast<int>(a.integer(9, 1));
    Output y(a, 12, {B, conv_out(H, stride), conv_out(W, stride), N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(8);
    const float *ws = a.as<float>(4), *sx = a.as<float>(6);
    const int32_t *sums = a.as<int32_t>(5), *zx = a.as<int32_t>(7);
    void *space = a.ptr(10), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 10);
    int32_t* status = a.as<int32_t>(11);
    call("mixdq_conv3x3_a8_asym", [&] {
        return mixdq_conv3x3_a8_asym(x, B, H, W, Cin, w, N, stride, w_bits, ws, sums, sx, zx, bias, y.address, space, space_bytes,
                                     status, st);
    });
    return y.release();
}

PyObject* conv3x3_q8(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 4);
    const int64_t B = X.size(0), H = X.size(1), W = X.size(2), Cin = X.size(3), N = a.integer(2);
    const int w_bits = static_cast<int>(a.integer(3)), stride = static_cast<int>(a.integer(7, 1));
    Output y(a, 9, {B, conv_out(H, stride), conv_out(W, stride), N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(6);
    const float *ws = a.as<float>(4), *sx = a.as<float>(5);
    int32_t* status = a.as<int32_t>(8);
    void* st = current_stream();
    call("mixdq_conv3x3_q8", [&] {
        return mixdq_conv3x3_q8(x, B, H, W, Cin, w, N, stride, w_bits, ws, sx, bias, y.address, status, st);
    });
    return y.release();
}

PyObject* conv3x3_a8_split(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 4);
    const int64_t B = X.size(0), H = X.size(1), W = X.size(2), Cin = X.size(3), at_ = a.integer(1), N = a.integer(4);
    const int w_bits = static_cast<int>(a.integer(5)), stride = static_cast<int>(a.integer(10, 1));
    Output y(a, 13, {B, conv_out(H, stride), conv_out(W, stride), N}, kF16, X);
    const void *x = a.ptr(0), *lo = a.ptr(2), *hi = a.ptr(3), *bias = a.ptr(9);
    const float *ws = a.as<float>(6), *s_lo = a.as<float>(7), *s_hi = a.as<float>(8);
    void *space = a.ptr(11), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 11);
    int32_t* status = a.as<int32_t>(12);
    call("mixdq_conv3x3_a8_split", [&] {
        return mixdq_conv3x3_a8_split(x, B, H, W, Cin, at_, lo, hi, N, stride, w_bits, ws, s_lo, s_hi, bias, y.address, space,
                                      space_bytes, status, st);
    });
    return y.release();
}

PyObject* conv1x1(const Args& a)
{
    const at::Tensor& X = a.tensor(0);
    need_dim(X, 4);
    const int64_t B = X.size(0), H = X.size(1), W = X.size(2), Cin = X.size(3), N = a.integer(2);
    const int w_bits = static_cast<int>(a.integer(3)), act_bits = static_cast<int>(a.integer(6, 8));
    Output y(a, -1, {B, H, W, N}, kF16, X);
    const void *x = a.ptr(0), *w = a.ptr(1), *bias = a.ptr(8);
    const float *ws = a.as<float>(4), *sx = a.as<float>(7);
    const int32_t* wz = a.as<int32_t>(5);
    void *space = a.ptr(9), *st = current_stream();
    const size_t space_bytes = bytes_of(a, 9);
    int32_t* status = a.as<int32_t>(10);
    call("mixdq_conv1x1", [&] {
        return mixdq_conv1x1(x, B, H, W, Cin, w, N, w_bits, ws, wz, act_bits, sx, bias, y.address, space, space_bytes, status, st);
    });
    return y.release();
}

// ---------------------------------------------------------------- module

template <PyObject* (*F)(const Args&), Signature& S>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames)
{
    try {
        return F(Args(S, args, nargs, kwnames));
    } catch (const Failed&) {
        return nullptr;
    } catch (...) {  // torch's own, e.g. out of memory
        torch::translate_exception_to_python(std::current_exception());
        return nullptr;
    }
}

Signature s_minmax{"weight_minmax_params", 3, 5, {"W", "bits", "symmetric", "scale_out", "zero_out"}};
Signature s_pack{"pack_weights", 3, 6, {"W", "bits", "scale", "zero", "layout", "out"}};
Signature s_sums{"weight_code_sums", 4, 4, {"packed_W", "N", "K", "bits"}};
Signature s_absmax{"act_absmax", 1, 2, {"X", "skip_rows_mod"}};
Signature s_from{"act_scale_from_absmax", 1, 1, {"amax"}};
Signature s_scale{"act_scale", 1, 2, {"X", "skip_rows_mod"}};
Signature s_range{"act_minmax", 1, 1, {"X"}};
Signature s_params{"act_asym_params", 1, 1, {"X"}};
Signature s_linear{"linear", 5, 12, {"X", "packed_W", "N", "w_bits", "w_scale", "w_zero", "act_bits", "act_scale", "bias",
                                     "workspace", "status", "out"}};
Signature s_asym{"linear_a8_asym", 8, 12, {"X", "packed_W", "N", "w_bits", "w_scale", "w_code_sums", "act_scale", "act_zero",
                                           "bias", "workspace", "status", "out"}};
Signature s_quant{"quantize_acts", 2, 3, {"X", "act_scale", "out"}};
Signature s_q8{"linear_q8", 6, 9, {"Xq", "packed_W", "N", "w_bits", "w_scale", "act_scale", "bias", "status", "out"}};
Signature s_fq{"linear_a8_fused_quant", 6, 10, {"X", "packed_W", "N", "w_bits", "w_scale", "act_scale", "bias", "tile_cols",
                                                "status", "out"}};
Signature s_static{"linear_a8_static_scratch", 6, 9, {"X", "packed_W", "N", "w_bits", "w_scale", "act_scale", "bias", "status",
                                                      "out"}};
Signature s_split{"linear_a8_split", 9, 13, {"X", "split_at", "packed_W_lo", "packed_W_hi", "N", "w_bits", "w_scale",
                                             "act_scale_lo", "act_scale_hi", "bias", "workspace", "status", "out"}};
Signature s_kv{"crossattn_kv", 7, 10, {"text_emb", "packed_W", "N", "w_bits", "w_scale", "act_scale", "bos_out", "workspace",
                                       "status", "out"}};
Signature s_conv{"conv3x3", 5, 13, {"X", "packed_W", "Cout", "w_bits", "w_scale", "w_zero", "act_bits", "act_scale", "bias",
                                    "stride", "workspace", "status", "out"}};
Signature s_conv_asym{"conv3x3_a8_asym", 8, 13, {"X", "packed_W", "Cout", "w_bits", "w_scale", "w_code_sums", "act_scale",
                                                 "act_zero", "bias", "stride", "workspace", "status", "out"}};
Signature s_conv_q8{"conv3x3_q8", 6, 10, {"Xq", "packed_W", "Cout", "w_bits", "w_scale", "act_scale", "bias", "stride", "status",
                                          "out"}};
Signature s_conv_split{"conv3x3_a8_split", 9, 14, {"X", "split_at", "packed_W_lo", "packed_W_hi", "Cout", "w_bits", "w_scale",
                                                   "act_scale_lo", "act_scale_hi", "bias", "stride", "workspace", "status",
                                                   "out"}};
Signature s_conv1{"conv1x1", 5, 11, {"X", "packed_W", "Cout", "w_bits", "w_scale", "w_zero", "act_bits", "act_scale", "bias",
                                     "workspace", "status"}};

Signature* const kSignatures[] = {&s_minmax, &s_pack, &s_sums, &s_absmax, &s_from, &s_scale, &s_range, &s_params, &s_linear,
                                  &s_asym, &s_quant, &s_q8, &s_fq, &s_static, &s_split, &s_kv, &s_conv, &s_conv_asym, &s_conv_q8,
                                  &s_conv_split, &s_conv1};

#define MIXDQ_ENTRY(name, sig, text)                                                                                  \
    {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<name, sig>)), METH_FASTCALL | METH_KEYWORDS, \
     #name "($module, " text}

PyMethodDef kMethods[] = {
    MIXDQ_ENTRY(weight_minmax_params, s_minmax, "W, bits, symmetric, scale_out=None, zero_out=None)\n--\n\n"
                "(scale, zero): per-output-channel min-max parameters of W fp16 [N, K]."),
    MIXDQ_ENTRY(pack_weights, s_pack, "W, bits, scale, zero=None, layout=1, out=None)\n--\n\n"
                "Packed codes of W fp16 [N, K]; zero=None: symmetric signed codes."),
    MIXDQ_ENTRY(weight_code_sums, s_sums, "packed_W, N, K, bits)\n--\n\nint32 [N]: sum of every channel's signed codes."),
    MIXDQ_ENTRY(act_absmax, s_absmax, "X, skip_rows_mod=0)\n--\n\nDevice fp32 [1]: max |X| over the rows kept."),
    MIXDQ_ENTRY(act_scale_from_absmax, s_from, "amax)\n--\n\nDevice fp32 [1]: amax / 127 (1 for 0)."),
    MIXDQ_ENTRY(act_scale, s_scale, "X, skip_rows_mod=0)\n--\n\n"
                "Dynamic per-tensor int8 scale max|X| / 127, computed on the device."),
    MIXDQ_ENTRY(act_minmax, s_range, "X)\n--\n\nDevice fp32 [2]: min(min x, 0), max(max x, 0)."),
    MIXDQ_ENTRY(act_asym_params, s_params, "X)\n--\n\n"
                "Asymmetric 8-bit activation parameters (device fp32 scale [1], device int32 zero-point [1])."),
    MIXDQ_ENTRY(linear, s_linear, "X, packed_W, N, w_bits, w_scale, w_zero=None, act_bits=8, act_scale=None, bias=None, "
                "workspace=None, status=None, out=None)\n--\n\nQuantized linear layer (mixdq_linear)."),
    MIXDQ_ENTRY(linear_a8_asym, s_asym, "X, packed_W, N, w_bits, w_scale, w_code_sums, act_scale, act_zero, bias=None, "
                "workspace=None, status=None, out=None)\n--\n\nLinear layer with asymmetric 8-bit activations."),
    MIXDQ_ENTRY(quantize_acts, s_quant, "X, act_scale, out=None)\n--\n\n"
                "int8 codes [rows, K] of X fp16 [rows, K] with the per-tensor scale *act_scale (device)."),
    MIXDQ_ENTRY(linear_q8, s_q8, "Xq, packed_W, N, w_bits, w_scale, act_scale, bias=None, status=None, out=None)\n--\n\n"
                "Linear layer on stored int8 codes."),
    MIXDQ_ENTRY(linear_a8_fused_quant, s_fq, "X, packed_W, N, w_bits, w_scale, act_scale, bias=None, tile_cols=128, "
                "status=None, out=None)\n--\n\n"
                "mixdq_linear (8-bit activations) as one kernel on 128 x tile_cols tiles, whatever the planner would choose."),
    MIXDQ_ENTRY(linear_a8_static_scratch, s_static, "X, packed_W, N, w_bits, w_scale, act_scale, bias=None, status=None, "
                "out=None)\n--\n\n"
                "W8A8 / W4A8 linear whose scratch is the library's built-in array: for callers that cannot allocate\n"
                "device memory.  The output tensor is still the caller's (out, or a fresh one here)."),
    MIXDQ_ENTRY(linear_a8_split, s_split, "X, split_at, packed_W_lo, packed_W_hi, N, w_bits, w_scale, act_scale_lo, "
                "act_scale_hi, bias=None, workspace=None, status=None, out=None)\n--\n\nShortcut-split linear layer."),
    MIXDQ_ENTRY(crossattn_kv, s_kv, "text_emb, packed_W, N, w_bits, w_scale, act_scale, bos_out, workspace=None, status=None, "
                "out=None)\n--\n\nBOS-aware cross-attention K or V projection."),
    MIXDQ_ENTRY(conv3x3, s_conv, "X, packed_W, Cout, w_bits, w_scale, w_zero=None, act_bits=8, act_scale=None, bias=None, "
                "stride=1, workspace=None, status=None, out=None)\n--\n\nQuantized 3x3 convolution, NHWC."),
    MIXDQ_ENTRY(conv3x3_a8_asym, s_conv_asym, "X, packed_W, Cout, w_bits, w_scale, w_code_sums, act_scale, act_zero, "
                "bias=None, stride=1, workspace=None, status=None, out=None)\n--\n\n"
                "3x3 convolution with asymmetric 8-bit activations."),
    MIXDQ_ENTRY(conv3x3_q8, s_conv_q8, "Xq, packed_W, Cout, w_bits, w_scale, act_scale, bias=None, stride=1, status=None, "
                "out=None)\n--\n\n3x3 convolution on a stored int8 image."),
    MIXDQ_ENTRY(conv3x3_a8_split, s_conv_split, "X, split_at, packed_W_lo, packed_W_hi, Cout, w_bits, w_scale, act_scale_lo, "
                "act_scale_hi, bias=None, stride=1, workspace=None, status=None, out=None)\n--\n\n"
                "Shortcut-split 3x3 convolution."),
    MIXDQ_ENTRY(conv1x1, s_conv1, "X, packed_W, Cout, w_bits, w_scale, w_zero=None, act_bits=8, act_scale=None, bias=None, "
                "workspace=None, status=None)\n--\n\n1x1 convolution, NHWC."),
    {nullptr, nullptr, 0, nullptr}};

PyObject* set_error_class(PyObject*, PyObject* cls)
{
    Py_XSETREF(g_error, Py_NewRef(cls));
    Py_RETURN_NONE;
}

PyMethodDef kSetError = {"_set_error_class", set_error_class, METH_O, nullptr};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_mixdq_native", "Native binding of the library's layer calls.", -1, kMethods};

}  // namespace

PyMODINIT_FUNC PyInit__mixdq_native(void)
{
    for (Signature* s : kSignatures)
        for (int i = 0; i < s->count; ++i)
            if (!(s->interned[i] = PyUnicode_InternFromString(s->names[i]))) return nullptr;
    PyObject* m = PyModule_Create(&kModule);
    if (!m) return nullptr;
    g_error = Py_NewRef(PyExc_RuntimeError);
    PyObject* f = PyCFunction_New(&kSetError, nullptr);
    if (!f || PyModule_AddObjectRef(m, "_set_error_class", f) < 0) return nullptr;
    Py_DECREF(f);
    // (build.py looks for the text: a binding made for another torch or Python is out of date whatever its time)
    if (PyModule_AddStringConstant(m, "built_for", MIXDQ_BUILT_FOR) < 0) return nullptr;
    return m;
}
