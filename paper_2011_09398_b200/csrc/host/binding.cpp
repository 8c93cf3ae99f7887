// The call path of the Python binding in native code: argument checks, output allocation, the current
// stream and the C-ABI call, for the entry points a model runs per layer.
//
// What bounds these calls is host time: a small layer runs 2-4 us on the GPU, and the same marshalling in
// Python (attribute reads of up to six tensors, a stream lookup, a ctypes call with eight arguments and
// torch.empty) took 11 us per call, 15 us with the output allocated, so a network of small layers was paced
// by its caller.  Here a tensor argument is unwrapped to its at::Tensor once and every check is a field read.
//
// The checks, their order and their messages are the binding's (binding.py holds the Python signatures and
// documents the calls).  The GIL is released around every library call, as ctypes does.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>

#include "lce.h"

namespace {

PyObject *g_lce_error = nullptr;  // binding.LceError, set by setup()

// A Python exception is set; unwinds to the entry point.
struct Raised {};

[[noreturn]] void value_error(const std::string &text)
{
    PyErr_SetString(PyExc_ValueError, text.c_str());
    throw Raised{};
}

void check(int status, const char *where)
{
    if (status == LCE_OK) return;
    PyObject *e = PyObject_CallFunction(g_lce_error, "is", status, where);
    if (e) {
        PyErr_SetObject(g_lce_error, e);
        Py_DECREF(e);
    }
    throw Raised{};
}

const at::Tensor &tensor(PyObject *o, const char *name)
{
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
        throw Raised{};
    }
    return THPVariable_Unpack(o);
}

const char *dtype_name(at::ScalarType t)
{
    return t == at::kFloat ? "torch.float32" : t == at::kInt ? "torch.int32" : "torch.uint8";
}

void *device_pointer(const at::Tensor &t, at::ScalarType dtype, const char *name)
{
    if (!t.is_cuda()) value_error(std::string(name) + " must be a CUDA tensor (there is no CPU path)");
    if (t.scalar_type() != dtype || !t.is_contiguous()) value_error(std::string(name) + " must be contiguous " + dtype_name(dtype));
    return t.data_ptr();
}

void *device_pointer(PyObject *o, at::ScalarType dtype, const char *name)  // None -> null
{
    return o == Py_None ? nullptr : device_pointer(tensor(o, name), dtype, name);
}

void *host_pointer(PyObject *o, at::ScalarType dtype, const char *name)  // None -> null
{
    if (o == Py_None) return nullptr;
    const at::Tensor &t = tensor(o, name);
    if (t.is_cuda() || t.scalar_type() != dtype || !t.is_contiguous())
        value_error(std::string(name) + " must be a contiguous host " + dtype_name(dtype) + " tensor");
    return t.data_ptr();
}

void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

at::Tensor empty_like_device(at::IntArrayRef shape, at::ScalarType dtype, const at::Tensor &on)
{
    if (on.is_cuda()) return at::Tensor(at::detail::empty_cuda(shape, dtype, on.device(), c10::nullopt));
    return at::empty(shape, on.options().dtype(dtype));
}

// The descriptor is a ctypes structure with the layout of lce_bconv2d_desc.
struct Desc {
    Py_buffer view{};
    const lce_bconv2d_desc *d = nullptr;
    explicit Desc(PyObject *o)
    {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw Raised{};
        if (view.len != (Py_ssize_t)sizeof(lce_bconv2d_desc)) {
            PyBuffer_Release(&view);
            PyErr_SetString(PyExc_TypeError, "desc must be a BConv2dDesc");
            throw Raised{};
        }
        d = static_cast<const lce_bconv2d_desc *>(view.buf);
    }
    ~Desc() { PyBuffer_Release(&view); }
    Desc(const Desc &) = delete;
};

int64_t words(int64_t c) { return (c + 31) / 32; }

template <typename Call>
int without_gil(Call call)
{
    int st;
    Py_BEGIN_ALLOW_THREADS;
    st = call();
    Py_END_ALLOW_THREADS;
    return st;
}

// Every entry point: fixed number of positional arguments, C++ exceptions turned into Python ones.
template <PyObject *(*Body)(PyObject *const *), Py_ssize_t N>
PyObject *entry(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", N, n);
        return nullptr;
    }
    try {
        return Body(args);
    } catch (const Raised &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

PyObject *returned(PyObject *given, const at::Tensor &made)
{
    if (given == Py_None) return THPVariable_Wrap(made);
    Py_INCREF(given);
    return given;
}

PyObject *bitpack(PyObject *const *a)  // x, out
{
    const at::Tensor &x = tensor(a[0], "x");
    if (x.dim() == 0) value_error("x must have a channel axis");
    const int64_t C = x.size(-1), rows = C ? x.numel() / C : 0;
    at::Tensor made;
    if (a[1] == Py_None) {
        c10::SmallVector<int64_t, 6> shape(x.sizes().begin(), x.sizes().end());
        shape.back() = words(C);
        made = empty_like_device(shape, at::kInt, x);
    }
    const at::Tensor &out = a[1] == Py_None ? made : tensor(a[1], "out");
    auto *px = static_cast<const float *>(device_pointer(x, at::kFloat, "x"));
    auto *po = static_cast<uint32_t *>(device_pointer(out, at::kInt, "out"));
    void *s = current_stream();
    check(without_gil([&] { return lce_bitpack(px, po, rows, (int32_t)C, s); }), "lce_bitpack");
    return returned(a[1], made);
}

PyObject *unpack(PyObject *const *a)  // words, channels, out
{
    const at::Tensor &w = tensor(a[0], "words");
    const long C = PyLong_AsLong(a[1]);
    if (C == -1 && PyErr_Occurred()) throw Raised{};
    if (words(C) == 0) {  // the row count is the tensor's words divided by the words per row
        PyErr_SetString(PyExc_ZeroDivisionError, "integer division or modulo by zero");
        throw Raised{};
    }
    const int64_t rows = w.numel() / words(C);
    at::Tensor made;
    if (a[2] == Py_None) {
        c10::SmallVector<int64_t, 6> shape(w.sizes().begin(), w.sizes().end());
        if (shape.empty()) shape.push_back(C); else shape.back() = C;
        made = empty_like_device(shape, at::kFloat, w);
    }
    const at::Tensor &out = a[2] == Py_None ? made : tensor(a[2], "out");
    auto *pw = static_cast<const uint32_t *>(device_pointer(w, at::kInt, "words"));
    auto *po = static_cast<float *>(device_pointer(out, at::kFloat, "out"));
    void *s = current_stream();
    check(without_gil([&] { return lce_unpack(pw, po, rows, (int32_t)C, s); }), "lce_unpack");
    return returned(a[2], made);
}

// lce_bconv2d and lce_bconv2d_f32: desc, input, weights, multiplier, bias, thresholds, out
template <bool F32>
PyObject *bconv2d(PyObject *const *a)
{
    const Desc desc(a[0]);
    const lce_bconv2d_desc &d = *desc.d;
    int32_t oh = 0, ow = 0;
    check(lce_bconv2d_out_shape(&d, &oh, &ow), "lce_bconv2d_out_shape");
    const at::Tensor &input = tensor(a[1], "input"), &weights = tensor(a[2], "weights");
    const at::ScalarType out_dtype = d.out_type == LCE_OUT_FLOAT32 ? at::kFloat : at::kInt;
    at::Tensor made;
    if (a[6] == Py_None)
        made = empty_like_device({d.batch, oh, ow, d.out_type == LCE_OUT_BITPACKED ? words(d.out_c) : (int64_t)d.out_c}, out_dtype, input);
    const at::Tensor &out = a[6] == Py_None ? made : tensor(a[6], "out");
    const int64_t want_in = (int64_t)d.batch * d.in_h * d.in_w * (F32 ? (int64_t)d.in_c : words(d.in_c));
    const int64_t want_w = d.weights_packed ? (int64_t)(lce_bconv2d_packed_weights_bytes(&d) / 4)
                                            : (int64_t)d.out_c * d.kernel_h * d.kernel_w * words(d.in_c);
    if (input.numel() != want_in || weights.numel() != want_w) value_error("input / weights size does not match the descriptor");
    void *pi = device_pointer(input, F32 ? at::kFloat : at::kInt, "input");
    auto *pw = static_cast<const uint32_t *>(device_pointer(weights, at::kInt, "weights"));
    auto *pm = static_cast<const float *>(device_pointer(a[3], at::kFloat, "multiplier"));
    auto *pb = static_cast<const float *>(device_pointer(a[4], at::kFloat, "bias"));
    auto *pt = static_cast<const int32_t *>(device_pointer(a[5], at::kInt, "thresholds"));
    void *po = device_pointer(out, out_dtype, "out");
    void *s = current_stream();
    if (F32)
        check(without_gil([&] { return lce_bconv2d_f32(&d, static_cast<const float *>(pi), pw, pm, pb, pt, po, s); }), "lce_bconv2d_f32");
    else
        check(without_gil([&] { return lce_bconv2d(&d, static_cast<const uint32_t *>(pi), pw, pm, pb, pt, po, s); }), "lce_bconv2d");
    return returned(a[6], made);
}

PyObject *bconv2d_fused(PyObject *const *a)  // desc, input, weights, multiplier, bias, residual, out_float, out_packed
{
    const Desc desc(a[0]);
    auto *pi = static_cast<const uint32_t *>(device_pointer(tensor(a[1], "input"), at::kInt, "input"));
    auto *pw = static_cast<const uint32_t *>(device_pointer(tensor(a[2], "weights"), at::kInt, "weights"));
    auto *pm = static_cast<const float *>(device_pointer(tensor(a[3], "multiplier"), at::kFloat, "multiplier"));
    auto *pb = static_cast<const float *>(device_pointer(tensor(a[4], "bias"), at::kFloat, "bias"));
    auto *pr = static_cast<const float *>(device_pointer(a[5], at::kFloat, "residual"));
    auto *pf = static_cast<float *>(device_pointer(a[6], at::kFloat, "out_float"));
    auto *pp = static_cast<uint32_t *>(device_pointer(a[7], at::kInt, "out_packed"));
    void *s = current_stream();
    check(without_gil([&] { return lce_bconv2d_fused(desc.d, pi, pw, pm, pb, pr, pf, pp, s); }), "lce_bconv2d_fused");
    Py_RETURN_NONE;
}

PyObject *plan_run(PyObject *const *a)  // handle (int or None)
{
    void *h = a[0] == Py_None ? nullptr : PyLong_AsVoidPtr(a[0]);
    if (PyErr_Occurred()) throw Raised{};
    void *s = current_stream();
    check(without_gil([&] { return lce_plan_run(static_cast<const lce_plan *>(h), s); }), "lce_plan_run");
    Py_RETURN_NONE;
}

PyObject *bmaxpool(PyObject *const *a)  // words, channels, pool_h, pool_w, stride_h, stride_w, padding, out
{
    const at::Tensor &w = tensor(a[0], "words");
    int32_t v[6];
    for (int i = 0; i < 6; ++i) {
        const long x = PyLong_AsLong(a[1 + i]);
        if (x == -1 && PyErr_Occurred()) throw Raised{};
        v[i] = (int32_t)x;
    }
    if (w.dim() != 4) value_error("words must be [N, H, W, words per pixel]");
    const int64_t N = w.size(0), H = w.size(1), W = w.size(2), Cw = w.size(3);
    if (Cw != words(v[0])) value_error("last dimension does not match channels");
    at::Tensor made;
    if (a[7] == Py_None) {
        if (v[3] == 0 || v[4] == 0) {
            PyErr_SetString(PyExc_ZeroDivisionError, "integer division or modulo by zero");
            throw Raised{};
        }
        const auto extent = [&](int64_t size, int64_t k, int64_t s) {
            if (v[5] == LCE_PAD_VALID) return size >= k ? (size - k) / s + 1 : (int64_t)0;
            return (size + s - 1) / s;
        };
        made = empty_like_device({N, extent(H, v[1], v[3]), extent(W, v[2], v[4]), Cw}, at::kInt, w);
    }
    const at::Tensor &out = a[7] == Py_None ? made : tensor(a[7], "out");
    auto *pw = static_cast<const uint32_t *>(device_pointer(w, at::kInt, "words"));
    auto *po = static_cast<uint32_t *>(device_pointer(out, at::kInt, "out"));
    void *s = current_stream();
    check(without_gil([&] { return lce_bmaxpool(pw, po, (int32_t)N, (int32_t)H, (int32_t)W, v[0], v[1], v[2], v[3], v[4], v[5], s); }), "lce_bmaxpool");
    return returned(a[7], made);
}

PyObject *add_f32(PyObject *const *args)  // a, b, out
{
    const at::Tensor &a = tensor(args[0], "a"), &b = tensor(args[1], "b");
    at::Tensor made;
    if (args[2] == Py_None) made = empty_like_device(a.sizes(), a.scalar_type(), a);
    const at::Tensor &out = args[2] == Py_None ? made : tensor(args[2], "out");
    if (a.numel() != b.numel() || a.numel() != out.numel()) value_error("size mismatch");
    auto *pa = static_cast<const float *>(device_pointer(a, at::kFloat, "a"));
    auto *pb = static_cast<const float *>(device_pointer(b, at::kFloat, "b"));
    auto *po = static_cast<float *>(device_pointer(out, at::kFloat, "out"));
    const int64_t n = a.numel();
    void *s = current_stream();
    check(without_gil([&] { return lce_add_f32(pa, pb, po, n, s); }), "lce_add_f32");
    return returned(args[2], made);
}

// desc, input, weights, multiplier, bias, thresholds, out, workspace
template <bool ASYNC>
PyObject *bconv2d_host(PyObject *const *a)
{
    const Desc desc(a[0]);
    auto *pi = static_cast<const uint32_t *>(host_pointer(a[1], at::kInt, "input"));
    auto *pw = static_cast<const uint32_t *>(host_pointer(a[2], at::kInt, "weights"));
    auto *pm = static_cast<const float *>(host_pointer(a[3], at::kFloat, "multiplier"));
    auto *pb = static_cast<const float *>(host_pointer(a[4], at::kFloat, "bias"));
    auto *pt = static_cast<const int32_t *>(host_pointer(a[5], at::kInt, "thresholds"));
    void *po = host_pointer(a[6], desc.d->out_type == LCE_OUT_FLOAT32 ? at::kFloat : at::kInt, "out");
    const at::Tensor &ws = tensor(a[7], "workspace");
    void *pws = device_pointer(ws, at::kByte, "workspace");
    const size_t bytes = (size_t)ws.numel();
    void *s = current_stream();
    if (ASYNC)
        check(without_gil([&] { return lce_bconv2d_host_async(desc.d, pi, pw, pm, pb, pt, po, pws, bytes, s); }), "lce_bconv2d_host_async");
    else
        check(without_gil([&] { return lce_bconv2d_host(desc.d, pi, pw, pm, pb, pt, po, pws, bytes, s); }), "lce_bconv2d_host");
    Py_RETURN_NONE;
}

PyObject *setup(PyObject *const *a)  // LceError
{
    Py_INCREF(a[0]);
    Py_XSETREF(g_lce_error, a[0]);
    Py_RETURN_NONE;
}

#define LCE_METHOD(name, body, n) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(entry<body, n>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    LCE_METHOD("setup", setup, 1),
    LCE_METHOD("bitpack", bitpack, 2),
    LCE_METHOD("unpack", unpack, 3),
    LCE_METHOD("bconv2d", bconv2d<false>, 7),
    LCE_METHOD("bconv2d_f32", bconv2d<true>, 7),
    LCE_METHOD("bconv2d_fused", bconv2d_fused, 8),
    LCE_METHOD("plan_run", plan_run, 1),
    LCE_METHOD("bmaxpool", bmaxpool, 8),
    LCE_METHOD("add_f32", add_f32, 3),
    LCE_METHOD("bconv2d_host", bconv2d_host<false>, 8),
    LCE_METHOD("bconv2d_host_async", bconv2d_host<true>, 8),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_lce_host", "Native call path of the binding (see binding.py).", -1, g_methods,
                        nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__lce_host() { return PyModule_Create(&g_module); }
