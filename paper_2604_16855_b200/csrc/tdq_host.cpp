// The host side of the Python binding: takes torch tensors, checks the layout the C ABI assumes but cannot see,
// makes the outputs the caller did not pass and enqueues the call.
//
// One pass of a small layer is a few microseconds of GPU work, so what the host does per call decides its time:
// marshalled through ctypes a quantize_act + w4a4_linear pair took 27 us to issue (46 us with outputs and workspace
// made by the calls), of which the two calls into the library were about 11.  Here the tensors are read in C++: 5 to 8 us
// (8.5), two launches included.
//
// The functions take every argument by position (binding.py gives them names and defaults) and release the
// interpreter lock while the library works, as ctypes does.
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <string>

#include "../../include/tdq.h"

namespace {

PyObject* g_tdq_error = nullptr;   // binding.TdqError, set once by the binding

struct Bad {                       // a Python exception to raise
    PyObject* type;
    std::string text;
};

const at::Tensor* opt_tensor(PyObject* o) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) throw Bad{PyExc_TypeError, std::string("expected a torch.Tensor, got ") + Py_TYPE(o)->tp_name};
    return &THPVariable_Unpack(o);
}
const at::Tensor& tensor(PyObject* o) {
    const at::Tensor* t = opt_tensor(o);
    if (!t) throw Bad{PyExc_TypeError, "expected a torch.Tensor, got None"};
    return *t;
}
std::string dtype_name(at::ScalarType s) { return std::string("torch.") + torch::getTHPDtype(s)->name; }

void need_cuda(std::initializer_list<const at::Tensor*> ts) {
    for (const at::Tensor* t : ts)
        if (t && !t->is_cuda()) throw Bad{PyExc_ValueError, "tdq runs on CUDA tensors only; there is no CPU path"};
}
tdq_dtype dtype_id(const at::Tensor& t) {
    switch (t.scalar_type()) {
        case at::kFloat: return TDQ_F32;
        case at::kBFloat16: return TDQ_BF16;
        case at::kHalf: return TDQ_F16;   // outputs of the linear layer only; the library refuses it elsewhere
        default: throw Bad{PyExc_TypeError, "tdq takes float32, bfloat16 or (for outputs) float16 tensors, got " + dtype_name(t.scalar_type())};
    }
}
at::ScalarType dtype_arg(PyObject* o) {
    if (!THPDtype_Check(o)) throw Bad{PyExc_TypeError, "out_dtype must be a torch.dtype"};
    return reinterpret_cast<THPDtype*>(o)->scalar_type;
}

// One operand of the linear layer: type, contiguity and the device all operands share.
void check_operand(const char* name, const at::Tensor* t, at::ScalarType want, const at::Tensor*& first) {
    if (!t) return;
    if (t->scalar_type() != want)
        throw Bad{PyExc_TypeError, std::string(name) + " must be " + dtype_name(want) + ", got " + dtype_name(t->scalar_type())};
    if (!t->is_contiguous()) throw Bad{PyExc_ValueError, std::string(name) + " must be contiguous"};
    if (!first) first = t;
    else if (t->device() != first->device())
        throw Bad{PyExc_ValueError, std::string(name) + " is on " + t->device().str() + ", the other operands on " + first->device().str()};
}
// y may have a row pitch but its columns must be adjacent
void check_y(const at::Tensor& y, const at::Tensor* first) {
    if (y.dim() != 2 || (y.size(1) > 1 && y.stride(1) != 1))
        throw Bad{PyExc_ValueError, "y must be a matrix whose columns are adjacent in memory"};
    if (first && y.device() != first->device())
        throw Bad{PyExc_ValueError, "y is on " + y.device().str() + ", the operands on " + first->device().str()};
}

tdq_act_params params_arg(PyObject* o) {
    tdq_act_params p;
    if (o == Py_None) {
        tdq_default_act_params(&p);
        return p;
    }
    Py_buffer b;   // a ctypes structure exposes its bytes
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) {
        PyErr_Clear();
        throw Bad{PyExc_TypeError, "params must be an ActParams"};
    }
    const bool fits = b.len == (Py_ssize_t)sizeof p;
    if (fits) memcpy(&p, b.buf, sizeof p);
    PyBuffer_Release(&b);
    if (!fits) throw Bad{PyExc_TypeError, "params must be an ActParams"};
    return p;
}
int64_t int_arg(PyObject* o) {
    PyObject* i = PyNumber_Index(o);
    if (!i) throw python_error();
    const int64_t v = PyLong_AsLongLong(i);
    Py_DECREF(i);
    if (v == -1 && PyErr_Occurred()) throw python_error();
    return v;
}

template <typename T = void>
T* ptr(const at::Tensor* t) { return t ? reinterpret_cast<T*>(t->data_ptr()) : nullptr; }
template <typename T = void>
T* ptr(const at::Tensor& t) { return reinterpret_cast<T*>(t.data_ptr()); }
void* stream_of(const at::Tensor& t) { return c10::cuda::getCurrentCUDAStream(t.device().index()).stream(); }

void check(tdq_status st, const char* where) {
    if (st == TDQ_OK) return;
    PyObject* e = PyObject_CallFunction(g_tdq_error, "is", (int)st, where);
    if (e) {
        PyErr_SetObject(g_tdq_error, e);
        Py_DECREF(e);
    }
    throw python_error();
}
// Runs a library call without the interpreter lock, on the device of `on`.
template <typename F>
tdq_status call(const at::Tensor& on, F&& f) {
    pybind11::gil_scoped_release release;
    c10::cuda::CUDAGuard guard(on.device());
    return f(stream_of(on));
}

PyObject* tuple2(const at::Tensor& a, const at::Tensor& b) {
    PyObject* pa = THPVariable_Wrap(a);
    PyObject* pb = pa ? THPVariable_Wrap(b) : nullptr;
    PyObject* t = pb ? PyTuple_Pack(2, pa, pb) : nullptr;
    Py_XDECREF(pa);
    Py_XDECREF(pb);
    return t;
}
// Straight to the caching allocator: the dispatcher's share of at::empty is half of its time, and a small layer whose
// outputs the calls make allocates four times.
at::Tensor new_like(const at::Tensor& on, at::IntArrayRef sizes, at::ScalarType s) {
    return at::Tensor(at::detail::empty_cuda(sizes, s, on.device(), c10::nullopt));
}
// The caller's workspace, or one from the caching allocator for the length of the call (given back to the stream's pool, so
// whatever the stream runs next is ordered behind its use).  Every linear call writes what it reads of the workspace, so
// nothing has to be cleared.
struct Workspace {
    at::DataPtr own;
    void* ptr;
    size_t bytes;
    Workspace(const at::Tensor* given, const at::Tensor& on, int64_t M, int64_t I_pad, int64_t O, int64_t g) {
        if (given) {
            ptr = given->data_ptr();
            bytes = (size_t)given->numel();
        } else {
            c10::cuda::CUDAGuard guard(on.device());
            bytes = tdq_linear_workspace_bytes(M, I_pad, O, (int32_t)g);
            own = c10::cuda::CUDACachingAllocator::get()->allocate(bytes);
            ptr = own.get();
        }
    }
};
at::Tensor workspace_for(const at::Tensor& on, int64_t M, int64_t I_pad, int64_t O, int64_t g) {
    return new_like(on, {(int64_t)tdq_linear_workspace_bytes(M, I_pad, O, (int32_t)g)}, at::kByte);
}

// quantize_act(x, params, codes, scale, offset)
PyObject* quantize_act(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0]);
    need_cuda({&x});
    const tdq_act_params p = params_arg(a[1]);
    const int64_t C = x.size(-1);
    const at::Tensor x2 = x.dim() == 2 ? x : x.reshape({-1, C});
    if (x2.stride(-1) != 1) throw Bad{PyExc_ValueError, "the channel axis must be contiguous"};
    const int64_t M = x2.size(0), g = p.group_size;
    if (g == 0) throw Bad{PyExc_ZeroDivisionError, "group_size is 0"};
    const int64_t K = (C + g - 1) / g;
    const at::Tensor *oc = opt_tensor(a[2]), *os = opt_tensor(a[3]), *oo = opt_tensor(a[4]);
    const at::Tensor codes = oc ? *oc : new_like(x, {M, K * g / 2}, at::kByte);
    const at::Tensor scale = os ? *os : new_like(x, {M, K}, at::kFloat);
    if (M > 0) {   // an empty tensor has no device pointer to pass
        const tdq_dtype dt = dtype_id(x2);
        check(call(x, [&](void* st) {
                  return tdq_quantize_act(ptr(x2), dt, 1, M, C, M > 1 ? x2.stride(0) : C, &p, ptr<uint8_t>(codes), ptr<float>(scale),
                                          ptr<float>(oo), st);
              }), "tdq_quantize_act");
    }
    return tuple2(codes, scale);
}

// quantize_act_fixed(x, radius, g, codes, scale, offset)
PyObject* quantize_act_fixed(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0]);
    const at::Tensor *oc = opt_tensor(a[3]), *os = opt_tensor(a[4]), *oo = opt_tensor(a[5]);
    need_cuda({&x, oc, os, oo});
    const double radius = PyFloat_AsDouble(a[1]);
    if (radius == -1.0 && PyErr_Occurred()) throw python_error();
    const int64_t g = int_arg(a[2]), C = x.size(-1);
    if (g == 0) throw Bad{PyExc_ZeroDivisionError, "group size is 0"};
    const at::Tensor x2 = x.dim() == 2 ? x : x.reshape({-1, C});
    const int64_t M = x2.size(0);
    const at::Tensor codes = oc ? *oc : new_like(x, {M, C / 2}, at::kByte);
    const at::Tensor scale = os ? *os : new_like(x, {M, std::max<int64_t>(C / g, 1)}, at::kFloat);
    const tdq_dtype dt = dtype_id(x2);
    check(call(x, [&](void* st) {
              return tdq_quantize_act_fixed(ptr(x2), dt, 1, M, C, M > 1 ? x2.stride(0) : C, (int32_t)g, (float)radius, ptr<uint8_t>(codes),
                                            ptr<float>(scale), ptr<float>(oo), st);
          }), "tdq_quantize_act_fixed");
    return tuple2(codes, scale);
}

// quantize_act_nchw(x, params, codes, scale, offset)
PyObject* quantize_act_nchw(PyObject* const* a) {
    const at::Tensor& x = tensor(a[0]);
    const at::Tensor *oc = opt_tensor(a[2]), *os = opt_tensor(a[3]), *oo = opt_tensor(a[4]);
    need_cuda({&x, oc, os, oo});
    const tdq_act_params p = params_arg(a[1]);
    if (x.dim() != 4 || !x.is_contiguous()) throw Bad{PyExc_ValueError, "x must be a contiguous [B, C, H, W] tensor"};
    const int64_t B = x.size(0), C = x.size(1), H = x.size(2), W = x.size(3), M = B * H * W;
    const at::Tensor codes = oc ? *oc : new_like(x, {M, C / 2}, at::kByte);
    const at::Tensor scale = os ? *os : new_like(x, {M, std::max<int64_t>(C / 32, 1)}, at::kFloat);
    const tdq_dtype dt = dtype_id(x);
    check(call(x, [&](void* st) {
              return tdq_quantize_act_nchw(ptr(x), dt, B, C, H, W, &p, ptr<uint8_t>(codes), ptr<float>(scale), ptr<float>(oo), st);
          }), "tdq_quantize_act_nchw");
    return tuple2(codes, scale);
}

// quantize_weight(w, pad_to, wcodes, wscale)
PyObject* quantize_weight(PyObject* const* a) {
    const at::Tensor& w0 = tensor(a[0]);
    need_cuda({&w0});
    const at::Tensor w = w0.contiguous();
    if (w.dim() != 2) throw Bad{PyExc_ValueError, "w must be a matrix [O, I]"};
    const int64_t O = w.size(0), I = w.size(1), pad = int_arg(a[1]);
    if (pad == 0) throw Bad{PyExc_ZeroDivisionError, "pad_to is 0"};
    const int64_t I_pad = (I + pad - 1) / pad * pad;
    const at::Tensor *oc = opt_tensor(a[2]), *os = opt_tensor(a[3]);
    const at::Tensor codes = oc ? *oc : new_like(w, {O, I_pad / 2}, at::kByte);
    const at::Tensor scale = os ? *os : new_like(w, {O}, at::kFloat);
    const tdq_dtype dt = dtype_id(w);
    check(call(w, [&](void* st) {
              return tdq_quantize_weight(ptr(w), dt, O, I, (int32_t)pad, ptr<uint8_t>(codes), ptr<float>(scale), st);
          }), "tdq_quantize_weight");
    return tuple2(codes, scale);
}

// w4a4_linear(xcodes, xscale, wcodes, wscale, bias, g, out_dtype, y, acc_debug, workspace, pow2)
PyObject* w4a4_linear(PyObject* const* a) {
    const at::Tensor &xc = tensor(a[0]), &xs = tensor(a[1]), &wc = tensor(a[2]), &ws = tensor(a[3]);
    const at::Tensor* bias = opt_tensor(a[4]);
    need_cuda({&xc, &xs, &wc, &ws, bias});
    const int64_t g = int_arg(a[5]);
    const at::Tensor *oy = opt_tensor(a[7]), *acc = opt_tensor(a[8]), *ow = opt_tensor(a[9]);
    const bool pow2 = a[10] == Py_True;
    if (xc.dim() != 2) throw Bad{PyExc_ValueError, "xcodes must be a matrix"};
    if (wc.dim() < 1) throw Bad{PyExc_ValueError, "wcodes must be a matrix"};
    const int64_t M = xc.size(0), I_pad = 2 * xc.size(1), O = wc.size(0);
    const at::Tensor y = oy ? *oy : new_like(xc, {M, O}, dtype_arg(a[6]));
    const at::Tensor* first = nullptr;
    check_operand("xcodes", &xc, at::kByte, first);
    check_operand("xscale", &xs, at::kFloat, first);
    check_operand("wcodes", &wc, at::kByte, first);
    check_operand("wscale", &ws, at::kFloat, first);
    check_operand("bias", bias, at::kFloat, first);
    check_operand("workspace", ow, at::kByte, first);
    check_operand("acc_debug", acc, at::kInt, first);
    check_y(y, first);
    const tdq_dtype dt = dtype_id(y);
    const Workspace workspace(ow, xc, M, I_pad, O, g);
    const int64_t y_stride = M > 0 ? y.stride(0) : O;
    check(call(xc, [&](void* st) {
              if (pow2)
                  return tdq_w4a4_linear_pow2(ptr<uint8_t>(xc), ptr<float>(xs), ptr<uint8_t>(wc), ptr<float>(ws), ptr<float>(bias), M, I_pad,
                                              O, (int32_t)g, ptr(y), dt, y_stride, workspace.ptr, workspace.bytes, st);
              return tdq_w4a4_linear(ptr<uint8_t>(xc), ptr<float>(xs), ptr<uint8_t>(wc), ptr<float>(ws), ptr<float>(bias), M, I_pad, O,
                                     (int32_t)g, ptr(y), dt, y_stride, ptr<int32_t>(acc), workspace.ptr, workspace.bytes, st);
          }), pow2 ? "tdq_w4a4_linear_pow2" : "tdq_w4a4_linear");
    return THPVariable_Wrap(y);
}

// w4a4_linear_static(xcodes, xscale, wcodes, wscale, bias, g, y, wait)
PyObject* w4a4_linear_static(PyObject* const* a) {
    const at::Tensor &xc = tensor(a[0]), &xs = tensor(a[1]), &wc = tensor(a[2]), &ws = tensor(a[3]), &y = tensor(a[6]);
    const at::Tensor* bias = opt_tensor(a[4]);
    need_cuda({&xc, &xs, &wc, &ws, bias, &y});
    const int64_t g = int_arg(a[5]);
    const int wait = PyObject_IsTrue(a[7]);
    if (wait < 0) throw python_error();
    if (xc.dim() != 2) throw Bad{PyExc_ValueError, "xcodes must be a matrix"};
    if (wc.dim() < 1) throw Bad{PyExc_ValueError, "wcodes must be a matrix"};
    const int64_t M = xc.size(0), O = wc.size(0);
    const at::Tensor* first = nullptr;
    check_operand("xcodes", &xc, at::kByte, first);
    check_operand("xscale", &xs, at::kFloat, first);
    check_operand("wcodes", &wc, at::kByte, first);
    check_operand("wscale", &ws, at::kFloat, first);
    check_operand("bias", bias, at::kFloat, first);
    check_y(y, first);
    const tdq_dtype dt = dtype_id(y);
    check(call(xc, [&](void* st) {
              return tdq_w4a4_linear_static(ptr<uint8_t>(xc), ptr<float>(xs), ptr<uint8_t>(wc), ptr<float>(ws), ptr<float>(bias), M,
                                            2 * xc.size(1), O, (int32_t)g, ptr(y), dt, M > 0 ? y.stride(0) : O, wait, st);
          }), "tdq_w4a4_linear_static");
    Py_INCREF(a[6]);
    return a[6];
}

// quant_linear_fused(x, wcodes, wscale, bias, params, out_dtype, y, workspace)
PyObject* quant_linear_fused(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0]), &wc = tensor(a[1]), &ws = tensor(a[2]);
    const at::Tensor *bias = opt_tensor(a[3]), *oy = opt_tensor(a[6]), *ow = opt_tensor(a[7]);
    need_cuda({&x, &wc, &ws, bias});
    const tdq_act_params p = params_arg(a[4]);
    const int64_t C = x.size(-1);
    const at::Tensor x2 = x.dim() == 2 ? x : x.reshape({-1, C});
    if (wc.dim() != 2) throw Bad{PyExc_ValueError, "wcodes must be a matrix"};
    const int64_t M = x2.size(0), O = wc.size(0);
    const at::Tensor y = oy ? *oy : new_like(x, {M, O}, dtype_arg(a[5]));
    if (C > 1 && x2.stride(1) != 1) throw Bad{PyExc_ValueError, "the channels of x must be adjacent in memory"};
    const at::Tensor* first = nullptr;
    check_operand("wcodes", &wc, at::kByte, first);
    check_operand("wscale", &ws, at::kFloat, first);
    check_operand("bias", bias, at::kFloat, first);
    check_operand("workspace", ow, at::kByte, first);
    check_y(y, first);
    if (x2.device() != first->device())
        throw Bad{PyExc_ValueError, "x is on " + x2.device().str() + ", the weights on " + first->device().str()};
    const tdq_dtype xdt = dtype_id(x2), ydt = dtype_id(y);
    const Workspace workspace(ow, x, M, wc.size(1) * 2, O, p.group_size);
    check(call(x, [&](void* st) {
              return tdq_quant_linear_fused(ptr(x2), xdt, 1, M, C, M > 1 ? x2.stride(0) : C, &p, ptr<uint8_t>(wc), ptr<float>(ws),
                                            ptr<float>(bias), O, ptr(y), ydt, y.stride(0), workspace.ptr, workspace.bytes, st);
          }), "tdq_quant_linear_fused");
    return THPVariable_Wrap(y);
}

// quant_linear_host(x_host, wcodes, wscale, bias, params, out_dtype, y_host)  ->  (y_host, buffers)
PyObject* quant_linear_host(PyObject* const* a) {
    const at::Tensor &x = tensor(a[0]), &wc = tensor(a[1]), &ws = tensor(a[2]);
    const at::Tensor *bias = opt_tensor(a[3]), *oy = opt_tensor(a[6]);
    need_cuda({&wc, &ws, bias});
    const tdq_act_params p = params_arg(a[4]);
    if (x.dim() != 2) throw Bad{PyExc_ValueError, "x_host must be a matrix"};
    const int64_t M = x.size(0), C = x.size(1), O = wc.size(0), g = p.group_size;
    if (g == 0) throw Bad{PyExc_ZeroDivisionError, "group_size is 0"};
    const int64_t K = (C + g - 1) / g, I_pad = K * g;
    const at::ScalarType yt = dtype_arg(a[5]);
    const at::Tensor x_dev = new_like(wc, {M, C}, x.scalar_type()), codes = new_like(wc, {M, I_pad / 2}, at::kByte);
    const at::Tensor scale = new_like(wc, {M, K}, at::kFloat), y_dev = new_like(wc, {M, O}, yt);
    const at::Tensor y = oy ? *oy : at::empty({M, O}, at::TensorOptions().dtype(yt)).pin_memory();
    const at::Tensor workspace = workspace_for(wc, M, I_pad, O, g);
    const tdq_dtype xdt = dtype_id(x), ydt = dtype_id(y);
    check(call(wc, [&](void* st) {
              return tdq_quant_linear_host(ptr(x), xdt, 1, M, C, &p, ptr<uint8_t>(wc), ptr<float>(ws), ptr<float>(bias), O, ptr(y), ydt,
                                           ptr(x_dev), ptr<uint8_t>(codes), ptr<float>(scale), ptr(y_dev), ptr(workspace),
                                           (size_t)workspace.numel(), st);
          }), "tdq_quant_linear_host");
    PyObject* bufs = PyTuple_New(5);
    if (!bufs) return nullptr;
    const at::Tensor* keep[5] = {&workspace, &x_dev, &codes, &scale, &y_dev};
    for (int i = 0; i < 5; ++i) PyTuple_SET_ITEM(bufs, i, THPVariable_Wrap(*keep[i]));
    PyObject* py = THPVariable_Wrap(y);
    PyObject* t = PyTuple_Pack(2, py, bufs);
    Py_DECREF(py);
    Py_DECREF(bufs);
    return t;
}

// Argument count, and C++ exceptions as Python ones.
template <PyObject* (*F)(PyObject* const*), int N>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != N) {
        PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", N, n);
        return nullptr;
    }
    try {
        return F(args);
    } catch (const Bad& b) {
        PyErr_SetString(b.type, b.text.c_str());
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

PyObject* set_error_class(PyObject*, PyObject* cls) {
    Py_INCREF(cls);
    Py_XSETREF(g_tdq_error, cls);
    Py_RETURN_NONE;
}

#define TDQ_ENTRY(NAME, N) {#NAME, (PyCFunction)(void (*)(void))entry<NAME, N>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    TDQ_ENTRY(quantize_act, 5), TDQ_ENTRY(quantize_act_fixed, 6), TDQ_ENTRY(quantize_act_nchw, 5), TDQ_ENTRY(quantize_weight, 4),
    TDQ_ENTRY(w4a4_linear, 11), TDQ_ENTRY(w4a4_linear_static, 8), TDQ_ENTRY(quant_linear_fused, 8), TDQ_ENTRY(quant_linear_host, 7),
    {"set_error_class", set_error_class, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
#undef TDQ_ENTRY

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tdq_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tdq_host(void) { return PyModule_Create(&module); }
