// The calls of binding.py that a decode loop or a data path makes many of, marshalled natively: tensors are checked, results
// allocated and the C entry point called without the interpreter in between.  Small calls are bound by the host: quantizing
// 352 x 2048 and decoding it again, with three allocations, took 21 us through ctypes for 10 us of kernels, now 11; a layer of
// one token and 4096 x 4096 7.8, now 6.3.
//
// Every function returns None for arguments that are not its plain case (other types, host tensors, another device than the
// current one, results the caller sized differently): binding.py then goes its own way, whose checks and errors are the
// reference.  A negative status of the library is returned as an int.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "../../include/mxint.h"

namespace {

PyTypeObject *g_format_type = nullptr;

struct Fallback {};                     // thrown where the plain case ends

// A CUDA tensor on device `dev` (-1: any, stored back); null for None.
const at::Tensor *tensor(PyObject *o, int *dev, bool needed)
{
    if (o == Py_None && !needed) return nullptr;
    if (!THPVariable_CheckExact(o)) throw Fallback();
    const at::Tensor &t = THPVariable_Unpack(o);
    if (!t.is_cuda() || t.layout() != at::kStrided) throw Fallback();
    const int d = t.get_device();
    if (*dev < 0) *dev = d;
    if (d != *dev) throw Fallback();
    return &t;
}
// Throws for a tensor without storage (the wrappers of vmap and grad, whose Python type is torch.Tensor as well).
void *ptr(const at::Tensor &t) { return t.data_ptr(); }
void *ptr(const at::Tensor *t) { return t ? t->data_ptr() : nullptr; }
const uint8_t *bytes_of(const at::Tensor &t) { return static_cast<const uint8_t *>(t.data_ptr()); }
const float *floats_of(const at::Tensor *t) { return static_cast<const float *>(ptr(t)); }

// A call of the library without the interpreter's lock.  Its arguments are evaluated by the caller, before: what throws there
// still holds the lock.
template <typename F, typename... A> mx_status_t unlocked(F call, A... args)
{
    mx_status_t s;
    Py_BEGIN_ALLOW_THREADS
    s = call(args...);
    Py_END_ALLOW_THREADS
    return s;
}

mx_format_t format(PyObject *o)
{
    if (!g_format_type || Py_TYPE(o) != g_format_type) throw Fallback();
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
        PyErr_Clear();
        throw Fallback();
    }
    mx_format_t f;
    const bool ok = b.len == (Py_ssize_t)sizeof(f);
    if (ok) std::memcpy(&f, b.buf, sizeof(f));
    PyBuffer_Release(&b);
    if (!ok) throw Fallback();
    return f;
}

int64_t integer(PyObject *o)
{
    if (!PyLong_CheckExact(o)) throw Fallback();
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) {
        PyErr_Clear();
        throw Fallback();
    }
    return v;
}

mx_dtype_t value_type(const at::Tensor &t)
{
    if (t.scalar_type() == at::kFloat) return MX_F32;
    if (t.scalar_type() == at::kBFloat16) return MX_BF16;
    throw Fallback();
}

// The current stream of the current device, which is the tensors' device; only for callers that name no stream.
void *stream_of(PyObject *stream, int dev)
{
    if (stream != Py_None || c10::cuda::current_device() != dev) throw Fallback();
    return c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream();
}

at::Tensor bytes(int64_t rows, int64_t cols, int dev)
{
    return at::empty({rows, cols}, at::TensorOptions().dtype(at::kByte).device(at::kCUDA, (c10::DeviceIndex)dev));
}

at::Tensor floats(int64_t rows, int64_t cols, int dev)
{
    return at::empty({rows, cols}, at::TensorOptions().dtype(at::kFloat).device(at::kCUDA, (c10::DeviceIndex)dev));
}
at::Tensor scratch(const at::Tensor *given, size_t need, int dev)
{
    if (given) return *given;
    const int64_t n = (int64_t)need;
    return at::empty({n > 256 ? n : 256}, at::TensorOptions().dtype(at::kByte).device(at::kCUDA, (c10::DeviceIndex)dev));
}

// Runs `call` and turns the end of the plain case into None, torch's errors into the ctypes route as well.
template <typename F> PyObject *guarded(F call)
{
    try {
        return call();
    } catch (const Fallback &) {
    } catch (const std::exception &) {
    }
    Py_RETURN_NONE;
}

// quantize(x, f, mant_out, exp_out, nonfinite_count, stream) -> (mant, exps)
PyObject *quantize(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 6) Py_RETURN_NONE;
    return guarded([&]() -> PyObject * {
        int dev = -1;
        const at::Tensor &x = *tensor(a[0], &dev, true);
        const mx_format_t f = format(a[1]);
        const at::Tensor *mant = tensor(a[2], &dev, false), *exps = tensor(a[3], &dev, false), *count = tensor(a[4], &dev, false);
        void *st = stream_of(a[5], dev);
        const mx_dtype_t dt = value_type(x);
        if (x.dim() != 2 || f.block <= 0 || f.block_rows <= 0) throw Fallback();
        const int64_t rows = x.size(0), K = x.size(1);
        at::Tensor m = mant ? *mant : bytes(rows, f.elem_bits <= 4 ? K / 2 : K, dev);
        at::Tensor e = exps ? *exps : bytes(rows / f.block_rows, K / f.block, dev);
        const mx_status_t s = unlocked(mx_quantize, ptr(x), dt, rows, K, x.stride(0), x.stride(1), f, ptr(m),
                                       static_cast<uint8_t *>(ptr(e)), static_cast<uint32_t *>(ptr(count)), st);
        if (s != MX_OK) return PyLong_FromLong(s);
        PyObject *out = PyTuple_New(2);
        if (!out) return nullptr;
        PyObject *pm = mant ? Py_NewRef(a[2]) : THPVariable_Wrap(std::move(m));
        PyObject *pe = exps ? Py_NewRef(a[3]) : THPVariable_Wrap(std::move(e));
        PyTuple_SET_ITEM(out, 0, pm);
        PyTuple_SET_ITEM(out, 1, pe);
        return out;
    });
}

// dequantize(mant, exps, K, f, bf16, out, stream) -> values
PyObject *dequantize(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 7) Py_RETURN_NONE;
    return guarded([&]() -> PyObject * {
        int dev = -1;
        const at::Tensor &mant = *tensor(a[0], &dev, true), &exps = *tensor(a[1], &dev, true);
        const int64_t K = integer(a[2]);
        const mx_format_t f = format(a[3]);
        const at::Tensor *given = tensor(a[5], &dev, false);
        void *st = stream_of(a[6], dev);
        if (mant.dim() < 1 || K < 0) throw Fallback();
        const int64_t rows = mant.size(0);
        if (given && (given->dim() != 2 || given->size(0) != rows || given->size(1) != K || given->stride(1) != 1)) throw Fallback();
        at::Tensor out = given ? *given
                               : at::empty({rows, K}, at::TensorOptions().dtype(a[4] == Py_True ? at::kBFloat16 : at::kFloat)
                                                          .device(at::kCUDA, (c10::DeviceIndex)dev));
        const mx_dtype_t dt = value_type(out);
        const mx_status_t s = unlocked(mx_dequantize, ptr(mant), bytes_of(exps), rows, K, f, ptr(out), dt, out.stride(0), st);
        if (s != MX_OK) return PyLong_FromLong(s);
        return given ? Py_NewRef(a[5]) : THPVariable_Wrap(std::move(out));
    });
}

// linear(x, fa, w_mant, w_exp, fw, N, bias, y, workspace, algo, stream) -> y
PyObject *linear(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 11) Py_RETURN_NONE;
    return guarded([&]() -> PyObject * {
        int dev = -1;
        const at::Tensor &x = *tensor(a[0], &dev, true);
        const mx_format_t fa = format(a[1]);
        const at::Tensor &wm = *tensor(a[2], &dev, true), &we = *tensor(a[3], &dev, true);
        const mx_format_t fw = format(a[4]);
        const int64_t N = integer(a[5]);
        const at::Tensor *bias = tensor(a[6], &dev, false), *given = tensor(a[7], &dev, false), *work = tensor(a[8], &dev, false);
        const mx_algo_t algo = (mx_algo_t)integer(a[9]);
        void *st = stream_of(a[10], dev);
        const mx_dtype_t dt = value_type(x);
        if (x.dim() != 2 || x.stride(1) != 1 || N < 0 || (given && given->dim() < 1)) throw Fallback();
        const int64_t M = x.size(0), K = x.size(1);
        at::Tensor y = given ? *given : floats(M, N, dev);
        const at::Tensor ws = scratch(work, work ? 0 : mx_workspace_bytes_ex(M, N, K, fa, fw, algo), dev);
        const mx_status_t s = unlocked(mx_linear_ex, ptr(x), dt, M, K, x.stride(0), fa, ptr(wm), bytes_of(we), fw, N,
                                       floats_of(bias), static_cast<float *>(ptr(y)), y.stride(0), ptr(ws), (size_t)ws.numel(), algo, st);
        if (s != MX_OK) return PyLong_FromLong(s);
        return given ? Py_NewRef(a[7]) : THPVariable_Wrap(std::move(y));
    });
}

bool rows_of_floats(const at::Tensor &t) { return t.dim() == 2 && t.stride(1) == 1 && t.scalar_type() == at::kFloat; }

// The result of a product with a fused tail: fp32 (`fy` None) or MXInt, the caller's tensors or new ones.
struct FusedResult {
    at::Tensor y, mant, exps;
    mx_format_t fy{};
    bool quantized;
    FusedResult(PyObject *fy_, const at::Tensor *y_, const at::Tensor *mant_, const at::Tensor *exps_, int64_t M, int64_t N, int dev)
        : quantized(fy_ != Py_None)
    {
        if (!quantized) {
            if (y_ && !rows_of_floats(*y_)) throw Fallback();
            y = y_ ? *y_ : floats(M, N, dev);
            return;
        }
        fy = format(fy_);
        if (fy.block <= 0 || fy.block_rows <= 0) throw Fallback();
        mant = mant_ ? *mant_ : bytes(M, fy.elem_bits <= 4 ? N / 2 : N, dev);
        exps = exps_ ? *exps_ : bytes(M / fy.block_rows, N / fy.block, dev);
    }
    float *y_ptr() const { return quantized ? nullptr : static_cast<float *>(y.data_ptr()); }
    int64_t ldy(int64_t N) const { return quantized ? N : y.stride(0); }
    void *mant_ptr() const { return quantized ? mant.data_ptr() : nullptr; }
    uint8_t *exp_ptr() const { return quantized ? static_cast<uint8_t *>(exps.data_ptr()) : nullptr; }
    PyObject *wrap(PyObject *y_, PyObject *mant_, PyObject *exps_)
    {
        if (!quantized) return y_ != Py_None ? Py_NewRef(y_) : THPVariable_Wrap(std::move(y));
        PyObject *out = PyTuple_New(2);
        if (!out) return nullptr;
        PyTuple_SET_ITEM(out, 0, mant_ != Py_None ? Py_NewRef(mant_) : THPVariable_Wrap(std::move(mant)));
        PyTuple_SET_ITEM(out, 1, exps_ != Py_None ? Py_NewRef(exps_) : THPVariable_Wrap(std::move(exps)));
        return out;
    }
};

mx_epilogue_t epilogue(const at::Tensor *bias, PyObject *relu, const at::Tensor *residual)
{
    if (residual && !rows_of_floats(*residual)) throw Fallback();
    mx_epilogue_t ep{};
    ep.bias = static_cast<const float *>(ptr(bias));
    ep.relu = relu == Py_True ? 1 : 0;
    ep.residual = static_cast<const float *>(ptr(residual));
    ep.ldr = residual ? residual->stride(0) : 0;
    return ep;
}

// linear_fused(x, fa, w_mant, w_exp, fw, N, bias, relu, residual, fy, y, y_mant, y_exp, layernorm, workspace, stream)
PyObject *linear_fused(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 16) Py_RETURN_NONE;
    return guarded([&]() -> PyObject * {
        int dev = -1;
        const at::Tensor &x = *tensor(a[0], &dev, true);
        const mx_format_t fa = format(a[1]);
        const at::Tensor &wm = *tensor(a[2], &dev, true), &we = *tensor(a[3], &dev, true);
        const mx_format_t fw = format(a[4]);
        const int64_t N = integer(a[5]);
        const at::Tensor *bias = tensor(a[6], &dev, false), *residual = tensor(a[8], &dev, false);
        const at::Tensor *y = tensor(a[10], &dev, false), *ym = tensor(a[11], &dev, false), *ye = tensor(a[12], &dev, false);
        mx_prologue_t pro{};
        if (a[13] != Py_None) {
            if (!PyTuple_CheckExact(a[13]) || PyTuple_GET_SIZE(a[13]) != 3 || !PyFloat_CheckExact(PyTuple_GET_ITEM(a[13], 2))) throw Fallback();
            pro.layernorm = 1;
            pro.ln_gamma = static_cast<const float *>(ptr(tensor(PyTuple_GET_ITEM(a[13], 0), &dev, false)));
            pro.ln_beta = static_cast<const float *>(ptr(tensor(PyTuple_GET_ITEM(a[13], 1), &dev, false)));
            pro.ln_eps = (float)PyFloat_AS_DOUBLE(PyTuple_GET_ITEM(a[13], 2));
        }
        const at::Tensor *work = tensor(a[14], &dev, false);
        void *st = stream_of(a[15], dev);
        const mx_dtype_t dt = value_type(x);
        if (x.dim() != 2 || x.stride(1) != 1 || N < 0) throw Fallback();
        const int64_t M = x.size(0), K = x.size(1);
        const mx_epilogue_t ep = epilogue(bias, a[7], residual);
        FusedResult r(a[9], y, ym, ye, M, N, dev);
        const at::Tensor ws = scratch(work, work ? 0 : mx_workspace_bytes_ex(M, N, K, fa, fw, MX_ALGO_TCGEN05), dev);
        const mx_status_t s = unlocked(mx_linear_fused, ptr(x), dt, M, K, x.stride(0), fa, pro.layernorm ? &pro : nullptr,
                                       ptr(wm), bytes_of(we), fw, N, &ep, r.y_ptr(), r.ldy(N), r.fy, r.mant_ptr(), r.exp_ptr(), ptr(ws),
                                       (size_t)ws.numel(), st);
        return s != MX_OK ? PyLong_FromLong(s) : r.wrap(a[10], a[11], a[12]);
    });
}

// gemm_fused(a_mant, a_exp, fa, w_mant, w_exp, fw, M, N, K, bias, relu, residual, fy, y, y_mant, y_exp, workspace, stream)
PyObject *gemm_fused(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 18) Py_RETURN_NONE;
    return guarded([&]() -> PyObject * {
        int dev = -1;
        const at::Tensor &am = *tensor(a[0], &dev, true), &ae = *tensor(a[1], &dev, true);
        const mx_format_t fa = format(a[2]);
        const at::Tensor &wm = *tensor(a[3], &dev, true), &we = *tensor(a[4], &dev, true);
        const mx_format_t fw = format(a[5]);
        const int64_t M = integer(a[6]), N = integer(a[7]), K = integer(a[8]);
        const at::Tensor *bias = tensor(a[9], &dev, false), *residual = tensor(a[11], &dev, false);
        const at::Tensor *y = tensor(a[13], &dev, false), *ym = tensor(a[14], &dev, false), *ye = tensor(a[15], &dev, false);
        const at::Tensor *work = tensor(a[16], &dev, false);
        void *st = stream_of(a[17], dev);
        if (M < 0 || N < 0 || K < 0) throw Fallback();
        const mx_epilogue_t ep = epilogue(bias, a[10], residual);
        FusedResult r(a[12], y, ym, ye, M, N, dev);
        const at::Tensor ws = scratch(work, work ? 0 : mx_workspace_bytes_ex(M, N, K, fa, fw, MX_ALGO_TCGEN05), dev);
        const mx_status_t s = unlocked(mx_gemm_fused, ptr(am), bytes_of(ae), fa, ptr(wm), bytes_of(we), fw, M, N, K, &ep,
                                       r.y_ptr(), r.ldy(N), r.fy, r.mant_ptr(), r.exp_ptr(), ptr(ws), (size_t)ws.numel(), st);
        return s != MX_OK ? PyLong_FromLong(s) : r.wrap(a[13], a[14], a[15]);
    });
}

// attention_fp(q, k, v, fqk, fv, heads, head_dim, scale, fp, causal, ctx, workspace, stream) -> ctx
PyObject *attention_fp(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 13) Py_RETURN_NONE;
    return guarded([&]() -> PyObject * {
        int dev = -1;
        const at::Tensor &q = *tensor(a[0], &dev, true), &k = *tensor(a[1], &dev, true), &v = *tensor(a[2], &dev, true);
        const mx_format_t fqk = format(a[3]), fv = format(a[4]), fp = format(a[8]);
        const int64_t heads = integer(a[5]), head_dim = integer(a[6]);
        if (!PyFloat_CheckExact(a[7])) throw Fallback();
        const float scale = (float)PyFloat_AS_DOUBLE(a[7]);
        const at::Tensor *given = tensor(a[10], &dev, false), *work = tensor(a[11], &dev, false);
        void *st = stream_of(a[12], dev);
        const mx_dtype_t dt = value_type(q);
        if (q.dim() != 2 || q.size(1) != heads * head_dim || (given && given->dim() < 1)) throw Fallback();
        for (const at::Tensor *t : {&q, &k, &v})
            if (t->dim() != 2 || t->sizes() != q.sizes() || t->scalar_type() != q.scalar_type() || t->stride(1) != 1) throw Fallback();
        const int64_t seq = q.size(0);
        at::Tensor ctx = given ? *given : floats(seq, heads * head_dim, dev);
        const at::Tensor ws = scratch(work, work ? 0 : mx_attention_workspace_bytes(seq, heads, head_dim), dev);
        const mx_status_t s = unlocked(mx_attention_fp, ptr(q), ptr(k), ptr(v), dt, q.stride(0), k.stride(0), v.stride(0), fqk,
                                       fv, seq, heads, head_dim, scale, a[9] == Py_True ? 1 : 0, fp, static_cast<float *>(ptr(ctx)),
                                       ctx.stride(0), ptr(ws), (size_t)ws.numel(), st);
        if (s != MX_OK) return PyLong_FromLong(s);
        return given ? Py_NewRef(a[10]) : THPVariable_Wrap(std::move(ctx));
    });
}

PyObject *set_format_type(PyObject *, PyObject *type)
{
    Py_INCREF(type);
    g_format_type = reinterpret_cast<PyTypeObject *>(type);
    Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"quantize", (PyCFunction)(void (*)(void))quantize, METH_FASTCALL, nullptr},
    {"dequantize", (PyCFunction)(void (*)(void))dequantize, METH_FASTCALL, nullptr},
    {"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, nullptr},
    {"linear_fused", (PyCFunction)(void (*)(void))linear_fused, METH_FASTCALL, nullptr},
    {"gemm_fused", (PyCFunction)(void (*)(void))gemm_fused, METH_FASTCALL, nullptr},
    {"attention_fp", (PyCFunction)(void (*)(void))attention_fp, METH_FASTCALL, nullptr},
    {"set_format_type", set_format_type, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&g_module); }
