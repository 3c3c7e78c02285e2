// The part of the Python binding that runs on every call: checks of the tensors, allocation of the outputs
// that the caller did not pass, addresses, torch's current stream, and the call into libgpusq.  No
// arithmetic.  A call costs ~1.5 us of host time on top of the launch (2.1 us) here; the same steps in
// Python through ctypes cost 2 us more for a call that allocates nothing and 5 us for one with two outputs.
// Outputs come from torch's caching allocator without the dispatcher: 0.4 us less for a call with two of them
// (4.7 -> 4.25, of which the launch is 2.1).
// The interpreter's lock is given up once per call, around allocations and library call together: the one may
// go to the driver and synchronise, the other waits when the stream's launch queue is full.
//
// Functions take positional arguments only; binding.py holds the public signatures and their defaults.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <algorithm>
#include <initializer_list>

#include "gpusq.h"

namespace {

PyObject *g_error = nullptr;            // binding.GpusqError
PyObject *g_out_of_memory = nullptr;    // torch.OutOfMemoryError

struct Failed {};                       // a Python exception is set

[[noreturn]] void fail(PyObject *type, const char *fmt, const char *a = "", const char *b = "")
{
    PyErr_Format(type, fmt, a, b);
    throw Failed();
}

const at::Tensor &tensor(PyObject *o, const char *what)
{
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "%s must be a tensor", what);
    return THPVariable_Unpack(o);
}

// a contiguous CUDA tensor of the given type
const at::Tensor &input(PyObject *o, at::ScalarType type, const char *type_name, const char *what)
{
    const at::Tensor &t = tensor(o, what);
    if (!t.is_cuda() || t.scalar_type() != type || !t.is_contiguous())
        fail(PyExc_ValueError, "%s must be a contiguous CUDA tensor of dtype %s", what, type_name);
    return t;
}
#define IN_F32(o, what) input(o, at::kFloat, "torch.float32", what)
#define IN_F16(o, what) input(o, at::kHalf, "torch.float16", what)
#define IN_I8(o, what) input(o, at::kChar, "torch.int8", what)
#define IN_U8(o, what) input(o, at::kByte, "torch.uint8", what)

struct Dims {
    int64_t rows, cols;
};
Dims matrix(const at::Tensor &t, const char *what)
{
    if (t.dim() != 2) fail(PyExc_ValueError, "%s must have two dimensions", what);
    return {t.size(0), t.size(1)};
}
int as_int(int64_t v)
{
    if (v != (int)v) fail(PyExc_OverflowError, "a dimension does not fit 32 bits");
    return (int)v;
}

int int_arg(PyObject *o)
{
    const int v = PyLong_AsInt(o);
    if (v == -1 && PyErr_Occurred()) throw Failed();
    return v;
}

// address of an optional argument (None: null)
void *address(PyObject *o, const char *what) { return o == Py_None ? nullptr : tensor(o, what).data_ptr(); }
template <typename T>
T *address_as(PyObject *o, const char *what) { return static_cast<T *>(address(o, what)); }

// An output: the tensor that the caller passed, or a new one, which make() allocates.
class Out {
public:
    Out(PyObject *given, const at::Tensor &like, at::ScalarType type, std::initializer_list<int64_t> shape, const char *what)
        : given_(given), device_(like.device()), type_(type), dims_(shape.size())
    {
        std::copy(shape.begin(), shape.end(), shape_);
        if (given != Py_None) p_ = tensor(given, what).data_ptr();
    }
    Out(const Out &) = delete;
    // without the interpreter's lock; torch's allocator without its dispatcher in between
    void make()
    {
        if (given_ != Py_None) return;
        made_ = at::Tensor(at::detail::empty_cuda(at::IntArrayRef(shape_, dims_), type_, device_, std::nullopt));
        p_ = made_.data_ptr();
    }
    PyObject *take()
    {
        PyObject *o = given_ != Py_None ? Py_NewRef(given_) : THPVariable_Wrap(std::move(made_));
        if (!o) throw Failed();
        return o;
    }
    template <typename T>
    T *as() const { return static_cast<T *>(p_); }
    void *p() const { return p_; }

private:
    PyObject *given_;
    at::Device device_;
    at::ScalarType type_;
    size_t dims_;
    int64_t shape_[2];
    at::Tensor made_;
    void *p_ = nullptr;
};

PyObject *pair(Out &a, Out &b)
{
    PyObject *t = PyTuple_New(2);
    if (!t) throw Failed();
    try {
        PyTuple_SET_ITEM(t, 0, a.take());
        PyTuple_SET_ITEM(t, 1, b.take());
    } catch (...) {
        Py_DECREF(t);
        throw;
    }
    return t;
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

void check(int status, const char *where)
{
    if (status == GPUSQ_OK) return;
    PyObject *e = PyObject_CallFunction(g_error, "is", status, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    throw Failed();
}

// The interpreter's lock, given up for as long as this object lives.
struct Unlocked {
    PyThreadState *state = PyEval_SaveThread();
    Unlocked() = default;
    Unlocked(const Unlocked &) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};

// Allocates the outputs and calls f(stream), which calls the library and must not touch Python.
template <typename F, typename... O>
void run(const char *where, F f, O &...outs)
{
    int status;
    {
        Unlocked u;
        (outs.make(), ...);
        status = f(stream());
    }
    check(status, where);
}

// C++ exceptions (out of memory, wrong tensor) become Python ones
template <PyObject *(*F)(PyObject *const *)>
PyObject *guarded(PyObject *, PyObject *const *a, Py_ssize_t)
{
    try {
        return F(a);
    } catch (const Failed &) {
    } catch (const c10::OutOfMemoryError &e) {
        PyErr_SetString(g_out_of_memory, e.what_without_backtrace());
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

// ---- weights ----

// W, Wp, mask or None, want_mask
PyObject *prune24(PyObject *const *a)
{
    const at::Tensor &W = IN_F32(a[0], "W");
    const auto [N, K] = matrix(W, "W");
    const int n = as_int(N), k = as_int(K);
    const float *w = W.const_data_ptr<float>();
    Out Wp(a[1], W, at::kFloat, {N, K}, "Wp");
    if (a[3] == Py_True) {
        Out mask(a[2], W, at::kByte, {N, K / 4}, "mask");
        run("gpusq_prune24", [&](void *s) { return gpusq_prune24(w, Wp.as<float>(), mask.as<uint8_t>(), n, k, s); }, Wp, mask);
        return pair(Wp, mask);
    }
    uint8_t *mask = address_as<uint8_t>(a[2], "mask");
    run("gpusq_prune24", [&](void *s) { return gpusq_prune24(w, Wp.as<float>(), mask, n, k, s); }, Wp);
    return Wp.take();
}

// W, want_mask
PyObject *prune48(PyObject *const *a)
{
    const at::Tensor &W = IN_F32(a[0], "W");
    const auto [N, K] = matrix(W, "W");
    const int n = as_int(N), k = as_int(K);
    const float *w = W.const_data_ptr<float>();
    Out Wp(Py_None, W, at::kFloat, {N, K}, "Wp");
    if (a[1] == Py_True) {
        Out mask(Py_None, W, at::kByte, {N, K / 8}, "mask");
        run("gpusq_prune48", [&](void *s) { return gpusq_prune48(w, Wp.as<float>(), mask.as<uint8_t>(), n, k, s); }, Wp, mask);
        return pair(Wp, mask);
    }
    run("gpusq_prune48", [&](void *s) { return gpusq_prune48(w, Wp.as<float>(), nullptr, n, k, s); }, Wp);
    return Wp.take();
}

// Wp, Wq, w_scale
template <int (*Fn)(const float *, int8_t *, float *, int, int, void *)>
PyObject *quantise_weight(PyObject *const *a, const char *where)
{
    const at::Tensor &Wp = IN_F32(a[0], "Wp");
    const auto [N, K] = matrix(Wp, "Wp");
    const int n = as_int(N), k = as_int(K);
    const float *w = Wp.const_data_ptr<float>();
    Out Wq(a[1], Wp, at::kChar, {N, K}, "Wq"), w_scale(a[2], Wp, at::kFloat, {N}, "w_scale");
    run(where, [&](void *s) { return Fn(w, Wq.as<int8_t>(), w_scale.as<float>(), n, k, s); }, Wq, w_scale);
    return pair(Wq, w_scale);
}
PyObject *quant_weight(PyObject *const *a) { return quantise_weight<gpusq_quant_weight>(a, "gpusq_quant_weight"); }
PyObject *quant_weight4(PyObject *const *a) { return quantise_weight<gpusq_quant_weight4>(a, "gpusq_quant_weight4"); }

// Wq, vals, meta
PyObject *compress24(PyObject *const *a)
{
    const at::Tensor &Wq = IN_I8(a[0], "Wq");
    const auto [N, K] = matrix(Wq, "Wq");
    const int n = as_int(N), k = as_int(K);
    const int8_t *w = Wq.const_data_ptr<int8_t>();
    Out vals(a[1], Wq, at::kChar, {N, K / 2}, "vals"), meta(a[2], Wq, at::kByte, {N, K / 8}, "meta");
    run("gpusq_compress24", [&](void *s) { return gpusq_compress24(w, vals.as<int8_t>(), meta.as<uint8_t>(), n, k, s); }, vals, meta);
    return pair(vals, meta);
}

// Wp
PyObject *compress24_f16(PyObject *const *a)
{
    const at::Tensor &Wp = IN_F32(a[0], "Wp");
    const auto [N, K] = matrix(Wp, "Wp");
    const int n = as_int(N), k = as_int(K);
    const float *w = Wp.const_data_ptr<float>();
    Out vals(Py_None, Wp, at::kHalf, {N, K / 2}, "vals"), meta(Py_None, Wp, at::kByte, {N, K / 8}, "meta");
    run("gpusq_compress24_f16", [&](void *s) { return gpusq_compress24_f16(w, vals.p(), meta.as<uint8_t>(), n, k, s); }, vals, meta);
    return pair(vals, meta);
}

// Wq
PyObject *compress48(PyObject *const *a)
{
    const at::Tensor &Wq = IN_I8(a[0], "Wq");
    const auto [N, K] = matrix(Wq, "Wq");
    const int n = as_int(N), k = as_int(K);
    const int8_t *w = Wq.const_data_ptr<int8_t>();
    Out vals4(Py_None, Wq, at::kByte, {N, K / 4}, "vals4"), meta4(Py_None, Wq, at::kByte, {N, K / 16}, "meta4");
    run("gpusq_compress48", [&](void *s) { return gpusq_compress48(w, vals4.as<uint8_t>(), meta4.as<uint8_t>(), n, k, s); }, vals4, meta4);
    return pair(vals4, meta4);
}

// vals4, meta4
PyObject *expand48(PyObject *const *a)
{
    const at::Tensor &vals4 = IN_U8(a[0], "vals4"), &meta4 = IN_U8(a[1], "meta4");
    const auto [N, K4] = matrix(vals4, "vals4");
    const int64_t K = K4 * 4;
    const int n = as_int(N), k = as_int(K);
    const uint8_t *v4 = vals4.const_data_ptr<uint8_t>(), *m4 = meta4.const_data_ptr<uint8_t>();
    Out vals(Py_None, vals4, at::kChar, {N, K / 2}, "vals"), meta(Py_None, vals4, at::kByte, {N, K / 8}, "meta");
    run("gpusq_expand48", [&](void *s) { return gpusq_expand48(v4, m4, vals.as<int8_t>(), meta.as<uint8_t>(), n, k, s); }, vals, meta);
    return pair(vals, meta);
}

// vals, meta, Wpacked
PyObject *pack24(PyObject *const *a)
{
    const at::Tensor &vals = IN_I8(a[0], "vals"), &meta = IN_U8(a[1], "meta");
    const auto [N, K2] = matrix(vals, "vals");
    const int n = as_int(N), k = as_int(K2 * 2);
    const int8_t *v = vals.const_data_ptr<int8_t>();
    const uint8_t *m = meta.const_data_ptr<uint8_t>();
    Out packed(a[2], vals, at::kByte, {(int64_t)gpusq_packed_bytes(n, k)}, "Wpacked");
    run("gpusq_pack24", [&](void *s) { return gpusq_pack24(v, m, packed.p(), n, k, s); }, packed);
    return packed.take();
}

// vals, meta, Wpacked
PyObject *pack24_f16(PyObject *const *a)
{
    const at::Tensor &vals = IN_F16(a[0], "vals"), &meta = IN_U8(a[1], "meta");
    const auto [N, K2] = matrix(vals, "vals");
    const int n = as_int(N), k = as_int(K2 * 2);
    const void *v = vals.const_data_ptr();
    const uint8_t *m = meta.const_data_ptr<uint8_t>();
    Out packed(a[2], vals, at::kByte, {(int64_t)gpusq_packed_bytes_f16(n, k)}, "Wpacked");
    run("gpusq_pack24_f16", [&](void *s) { return gpusq_pack24_f16(v, m, packed.p(), n, k, s); }, packed);
    return packed.take();
}

// ---- activations ----

// X, Xq, x_scale, scale_mode, workspace
template <int (*Fn)(const void *, int8_t *, float *, int, int64_t, int, void *, size_t, void *)>
PyObject *quantise_act(PyObject *const *a, const char *where)
{
    const at::Tensor &X = IN_F16(a[0], "X");
    const auto [M, K] = matrix(X, "X");
    const int64_t m = M;
    const int k = as_int(K), mode = int_arg(a[3]);
    if (mode == GPUSQ_SCALE_GIVEN && a[2] == Py_None) fail(PyExc_ValueError, "scale_mode GIVEN needs x_scale");
    const void *x = X.const_data_ptr();
    Out Xq(a[1], X, at::kChar, {M, K}, "Xq"), x_scale(a[2], X, at::kFloat, {1}, "x_scale");
    void *ws = nullptr;
    size_t ws_bytes = 0;
    if (a[4] != Py_None) {
        const at::Tensor &w = tensor(a[4], "workspace");
        ws = w.data_ptr();
        ws_bytes = (size_t)w.numel() * w.element_size();
    }
    const bool needs_own = a[4] == Py_None && mode == GPUSQ_SCALE_COMPUTE;
    at::Tensor own;
    run(where, [&](void *s) {
        if (needs_own) {
            ws_bytes = gpusq_quant_act_workspace(m, k);
            own = at::zeros({(int64_t)ws_bytes}, at::TensorOptions().dtype(at::kByte).device(X.device()));
            ws = own.data_ptr();
        }
        return Fn(x, Xq.as<int8_t>(), x_scale.as<float>(), mode, m, k, ws, ws_bytes, s);
    }, Xq, x_scale);
    return pair(Xq, x_scale);
}
PyObject *quant_act(PyObject *const *a) { return quantise_act<gpusq_quant_act>(a, "gpusq_quant_act"); }
PyObject *quant_act4(PyObject *const *a) { return quantise_act<gpusq_quant_act4>(a, "gpusq_quant_act4"); }

// X, absmax, Xq, x_scale
PyObject *quant_act_absmax(PyObject *const *a)
{
    const at::Tensor &X = IN_F16(a[0], "X");
    const auto [M, K] = matrix(X, "X");
    const int64_t m = M;
    const int k = as_int(K);
    const void *x = X.const_data_ptr();
    const float *absmax = address_as<float>(a[1], "absmax");
    Out Xq(a[2], X, at::kChar, {M, K}, "Xq"), x_scale(a[3], X, at::kFloat, {1}, "x_scale");
    run("gpusq_quant_act_absmax", [&](void *s) { return gpusq_quant_act_absmax(x, Xq.as<int8_t>(), x_scale.as<float>(), absmax, m, k, s); }, Xq, x_scale);
    return pair(Xq, x_scale);
}

// ---- layers ----

// Xq, weight operand, N, w_scale, x_scale, bias, act, out_type, out_scale, Y, status_buf
template <int (*Fn)(const int8_t *, const void *, const float *, const float *, const float *, int, int, const float *, void *, int64_t, int, int, int32_t *, void *)>
PyObject *gemm(PyObject *const *a, const char *where)
{
    const at::Tensor &Xq = IN_I8(a[0], "Xq");
    const auto [M, K] = matrix(Xq, "Xq");
    const int64_t m = M;
    const int N = int_arg(a[2]), k = as_int(K), act = int_arg(a[6]), out_type = int_arg(a[7]);
    const at::ScalarType type = out_type == GPUSQ_OUT_F16 ? at::kHalf : out_type == GPUSQ_OUT_I8 ? at::kChar : at::kInt;
    if (a[9] == Py_None && (out_type < 0 || out_type > 2)) fail(PyExc_KeyError, "out_type");
    const int8_t *x = Xq.const_data_ptr<int8_t>();
    const void *w = address(a[1], "weight");
    const float *w_scale = address_as<float>(a[3], "w_scale"), *x_scale = address_as<float>(a[4], "x_scale");
    const float *bias = address_as<float>(a[5], "bias"), *out_scale = address_as<float>(a[8], "out_scale");
    int32_t *status = address_as<int32_t>(a[10], "status_buf");
    Out Y(a[9], Xq, type, {M, N}, "Y");
    run(where, [&](void *s) { return Fn(x, w, w_scale, x_scale, bias, act, out_type, out_scale, Y.p(), m, N, k, status, s); }, Y);
    return Y.take();
}
int dense(const int8_t *Xq, const void *Wq, const float *ws, const float *xs, const float *bias, int act, int out_type,
          const float *os, void *Y, int64_t M, int N, int K, int32_t *status, void *s)
{
    return gpusq_gemm_i8_dense(Xq, static_cast<const int8_t *>(Wq), ws, xs, bias, act, out_type, os, Y, M, N, K, status, s);
}
PyObject *spgemm_i8(PyObject *const *a) { return gemm<gpusq_spgemm_i8>(a, "gpusq_spgemm_i8"); }
PyObject *gemm_i8_dense(PyObject *const *a) { return gemm<dense>(a, "gpusq_gemm_i8_dense"); }

// Xq, Wpacked, N, w_scale, x_scale, bias, act, Y, y_absmax, status_buf
PyObject *spgemm_i8_absmax(PyObject *const *a)
{
    const at::Tensor &Xq = IN_I8(a[0], "Xq");
    const auto [M, K] = matrix(Xq, "Xq");
    const int64_t m = M;
    const int N = int_arg(a[2]), k = as_int(K), act = int_arg(a[6]);
    const int8_t *x = Xq.const_data_ptr<int8_t>();
    const void *w = address(a[1], "Wpacked");
    const float *w_scale = address_as<float>(a[3], "w_scale"), *x_scale = address_as<float>(a[4], "x_scale"), *bias = address_as<float>(a[5], "bias");
    int32_t *status = address_as<int32_t>(a[9], "status_buf");
    Out Y(a[7], Xq, at::kHalf, {M, N}, "Y"), y_absmax(a[8], Xq, at::kFloat, {1}, "y_absmax");
    run("gpusq_spgemm_i8_absmax", [&](void *s) {
        return gpusq_spgemm_i8_absmax(x, w, w_scale, x_scale, bias, act, Y.p(), y_absmax.as<float>(), m, N, k, status, s);
    }, Y, y_absmax);
    return pair(Y, y_absmax);
}

// X, Wpacked, N, bias, act, out_type, Y, status_buf
PyObject *spgemm_f16(PyObject *const *a)
{
    const at::Tensor &X = IN_F16(a[0], "X");
    const auto [M, K] = matrix(X, "X");
    const int64_t m = M;
    const int N = int_arg(a[2]), k = as_int(K), act = int_arg(a[4]), out_type = int_arg(a[5]);
    const void *x = X.const_data_ptr(), *w = address(a[1], "Wpacked");
    const float *bias = address_as<float>(a[3], "bias");
    int32_t *status = address_as<int32_t>(a[7], "status_buf");
    Out Y(a[6], X, out_type == GPUSQ_OUT_F16 ? at::kHalf : at::kFloat, {M, N}, "Y");
    run("gpusq_spgemm_f16", [&](void *s) { return gpusq_spgemm_f16(x, w, bias, act, out_type, Y.p(), m, N, k, status, s); }, Y);
    return Y.take();
}

// GpusqError, torch.OutOfMemoryError; called once, before anything else
PyObject *set_errors(PyObject *const *a)
{
    Py_XSETREF(g_error, Py_NewRef(a[0]));
    Py_XSETREF(g_out_of_memory, Py_NewRef(a[1]));
    Py_RETURN_NONE;
}

// the wrappers of binding.py always pass this many arguments
template <PyObject *(*F)(PyObject *const *), int kArgs>
PyObject *entry(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    if (n != kArgs) {
        PyErr_Format(PyExc_TypeError, "%d arguments expected, %zd given", kArgs, n);
        return nullptr;
    }
    return guarded<F>(self, a, n);
}
#define ENTRY(name, args) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<name, args>)), METH_FASTCALL, nullptr}

PyMethodDef g_methods[] = {
    ENTRY(set_errors, 2), ENTRY(prune24, 4), ENTRY(prune48, 2), ENTRY(quant_weight, 3), ENTRY(quant_weight4, 3),
    ENTRY(compress24, 3), ENTRY(compress24_f16, 1), ENTRY(compress48, 1), ENTRY(expand48, 2), ENTRY(pack24, 3),
    ENTRY(pack24_f16, 3), ENTRY(quant_act, 5), ENTRY(quant_act4, 5), ENTRY(quant_act_absmax, 4), ENTRY(spgemm_i8, 11),
    ENTRY(gemm_i8_dense, 11), ENTRY(spgemm_i8_absmax, 10), ENTRY(spgemm_f16, 8), {nullptr, nullptr, 0, nullptr},
};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_gpusq_torch", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// built_for: the torch and the Python this module was compiled against (build.py)
PyMODINIT_FUNC PyInit__gpusq_torch()
{
    PyObject *m = PyModule_Create(&g_module);
    if (m && PyModule_AddStringConstant(m, "built_for", GPUSQ_BUILT_FOR) < 0) Py_CLEAR(m);
    return m;
}
