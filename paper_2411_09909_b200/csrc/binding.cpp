// Native half of amx.py: the argument marshalling of its hot functions as a CPython extension module.
//
// Through ctypes a call costs 15-30 us of host time (argument conversion, a Python-level allocation per output and
// per scratch buffer, the stream lookup), more than the GPU needs for a small layer.  Here a call unpacks the tensors,
// allocates through the caching allocator without the dispatcher, takes the current stream and enters the C ABI:
// about 3 us plus the launches, which run without the interpreter lock.  Nothing is kept between calls.
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "amx.h"

namespace {

PyObject* g_error = nullptr;      // amx.AmxError

[[nodiscard]] PyObject* fail(const char* what, int rc) {
    PyErr_Format(g_error, "%s: %s (%d)", what, amx_status_string(rc), rc);
    return nullptr;
}
[[nodiscard]] bool require(bool ok, const char* what) {
    if (!ok) PyErr_SetString(PyExc_AssertionError, what);
    return ok;
}
// A tensor argument; nullptr with a Python error set when the object is not one.
const at::Tensor* tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(g_error, "%s must be a tensor", name);
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}
const at::Tensor* device_tensor(PyObject* o, at::ScalarType dtype, const char* name) {
    const at::Tensor* t = tensor(o, name);
    if (t && (!t->is_cuda() || t->scalar_type() != dtype)) {
        PyErr_Format(g_error, "%s must be a CUDA tensor of %s", name, c10::toString(dtype));
        return nullptr;
    }
    return t;
}
// The same for a matrix (checked first: a shape is wrong on every device).
const at::Tensor* device_matrix(PyObject* o, at::ScalarType dtype, const char* name) {
    const at::Tensor* t = tensor(o, name);
    if (t && t->dim() != 2) {
        PyErr_Format(PyExc_ValueError, "%s must be a matrix, not a tensor of %lld dimensions", name, (long long)t->dim());
        return nullptr;
    }
    return t ? device_tensor(o, dtype, name) : nullptr;
}
at::Tensor empty(at::IntArrayRef sizes, at::ScalarType dtype, const at::Tensor& like) {
    return at::detail::empty_cuda(sizes, dtype, like.device(), std::nullopt);
}
at::Tensor scratch(size_t bytes, const at::Tensor& like) {
    return empty({(int64_t)(bytes > 256 ? bytes : 256)}, at::kByte, like);
}
// Enters the library with the interpreter lock given up (a launch waits when the stream's queue is full); the arguments have
// been evaluated by then.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename... P, typename... A>
int enter(int (*fn)(P...), A... args) {
    const Unlocked unlocked;
    return fn(static_cast<P>(args)...);
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
uint8_t* u8(const at::Tensor& t) { return static_cast<uint8_t*>(t.data_ptr()); }
float* f32(const at::Tensor& t) { return static_cast<float*>(t.data_ptr()); }
PyObject* wrap(at::Tensor t) { return THPVariable_Wrap(std::move(t)); }
PyObject* tuple(std::initializer_list<at::Tensor> ts) {
    PyObject* r = PyTuple_New((Py_ssize_t)ts.size());
    Py_ssize_t i = 0;
    for (const at::Tensor& t : ts) PyTuple_SET_ITEM(r, i++, wrap(t));
    return r;
}
int64_t as_int(PyObject* o) { return PyLong_AsLongLong(o); }
// Leading dimension of a row-major matrix (a single row may carry any stride).
int64_t lead(const at::Tensor& t) { return t.size(0) > 1 ? t.stride(0) : std::max(t.size(1), t.stride(0)); }

#define ARGS(n)                                                                              \
    if (nargs != (n)) {                                                                      \
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");                       \
        return nullptr;                                                                      \
    }
#define INTS_OK                                                                              \
    if (PyErr_Occurred()) return nullptr;

// quantize(x, group_size, fmt) -> (codes, scales)
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(3)
    const at::Tensor* x = device_tensor(a[0], at::kBFloat16, "x");
    if (!x) return nullptr;
    const int64_t gs = as_int(a[1]), fmt = as_int(a[2]);
    INTS_OK
    if (!require(x->dim() == 2 && x->stride(1) == 1, "x must be a row-major matrix")) return nullptr;
    if (gs <= 0) return fail("amx_quantize", AMX_ERR_SHAPE);
    const int64_t rows = x->size(0), K = x->size(1);
    at::Tensor codes = empty({rows, K / 2}, at::kByte, *x), scales = empty({rows, K / gs, 2}, at::kByte, *x);
    const int rc = enter(amx_quantize_fmt, x->data_ptr(), rows, K, lead(*x), (int)gs, (int)fmt, u8(codes), u8(scales), stream());
    if (rc) return fail(fmt ? "amx_quantize_fmt" : "amx_quantize", rc);
    return tuple({codes, scales});
    END_HANDLE_TH_ERRORS
}

// fake_quantize(x, group_size, fmt, out) -> out
PyObject* fake_quantize(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(4)
    const at::Tensor* x = device_tensor(a[0], at::kBFloat16, "x");
    if (!x) return nullptr;
    const int64_t gs = as_int(a[1]), fmt = as_int(a[2]);
    INTS_OK
    if (!require(x->dim() == 2 && x->stride(1) == 1, "x must be a row-major matrix")) return nullptr;
    at::Tensor out;
    if (a[3] == Py_None) out = empty({x->size(0), x->size(1)}, at::kBFloat16, *x);
    else {
        const at::Tensor* o = tensor(a[3], "out");
        if (!o || !require(o->sizes() == x->sizes() && o->stride(1) == 1, "out must have the shape of x and contiguous rows"))
            return nullptr;
        out = *o;
    }
    const int rc = enter(amx_fake_quantize, x->data_ptr(), x->size(0), x->size(1), lead(*x), (int)gs, (int)fmt, out.data_ptr(),
                         lead(out), stream());
    if (rc) return fail("amx_fake_quantize", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// dequantize(codes, scales, group_size, bf16) -> out
PyObject* dequantize(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(4)
    const at::Tensor *c = device_tensor(a[0], at::kByte, "codes"), *s = c ? device_tensor(a[1], at::kByte, "scales") : nullptr;
    if (!s) return nullptr;
    const int64_t gs = as_int(a[2]);
    const bool bf16 = PyObject_IsTrue(a[3]);
    INTS_OK
    const int64_t rows = c->size(0), K = c->size(1) * 2;
    at::Tensor out = empty({rows, K}, bf16 ? at::kBFloat16 : at::kFloat, *c);
    const int rc = enter(amx_dequantize, u8(*c), u8(*s), rows, K, (int)gs, bf16 ? AMX_OUT_BF16 : AMX_OUT_F32, out.data_ptr(), K, stream());
    if (rc) return fail("amx_dequantize", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// quant_error(x, codes, scales, group_size) -> four doubles
PyObject* quant_error(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(4)
    const at::Tensor* x = device_tensor(a[0], at::kBFloat16, "x");
    const at::Tensor *c = x ? device_tensor(a[1], at::kByte, "codes") : nullptr, *s = c ? device_tensor(a[2], at::kByte, "scales") : nullptr;
    if (!s) return nullptr;
    const int64_t gs = as_int(a[3]);
    INTS_OK
    if (!require(x->dim() == 2 && x->stride(1) == 1 && c->is_contiguous() && s->is_contiguous(), "x must be a row-major matrix, codes and scales contiguous"))
        return nullptr;
    at::Tensor out = empty({4}, at::kDouble, *x);
    const size_t need = amx_quant_error_workspace_bytes();
    at::Tensor ws = scratch(need, *x);
    const int rc = enter(amx_quant_error, x->data_ptr(), x->size(0), x->size(1), x->stride(0), u8(*c), u8(*s), (int)gs,
                         static_cast<double*>(out.data_ptr()), ws.data_ptr(), (size_t)ws.numel(), stream());
    if (rc) return fail("amx_quant_error", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// The optional out / workspace arguments of a product: allocated when None.
bool out_and_workspace(PyObject* out_arg, PyObject* ws_arg, int64_t M, int64_t N, at::ScalarType dtype, size_t need,
                       const at::Tensor& like, at::Tensor& out, at::Tensor& ws) {
    if (out_arg == Py_None) out = empty({M, N}, dtype, like);
    else {
        const at::Tensor* o = tensor(out_arg, "out");
        if (!o) return false;
        out = *o;
    }
    if (ws_arg == Py_None) ws = scratch(need, like);
    else {
        const at::Tensor* w = tensor(ws_arg, "workspace");
        if (!w) return false;
        ws = *w;
    }
    return true;
}

// gemm(a_codes, a_scales, w_codes, w_scales, group_size, flags, out, workspace) -> out
PyObject* gemm(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(8)
    static const char* const names[4] = {"a_codes", "a_scales", "w_codes", "w_scales"};
    const at::Tensor* t[4];
    for (int i = 0; i < 4; ++i) {
        t[i] = device_tensor(a[i], at::kByte, names[i]);
        if (!t[i] || !require(t[i]->is_contiguous(), "operands must be contiguous")) return nullptr;
    }
    const int64_t gs = as_int(a[4]), flags = as_int(a[5]);
    INTS_OK
    const int64_t M = t[0]->size(0), K = t[0]->size(1) * 2, N = t[2]->size(0);
    if (!require(t[2]->size(1) * 2 == K, "operands differ in K")) return nullptr;
    at::Tensor out, ws;
    const size_t need = a[7] == Py_None ? amx_workspace_bytes(M, N, K, (int)gs, (uint32_t)flags) : 0;
    if (!out_and_workspace(a[6], a[7], M, N, at::kFloat, need, *t[0], out, ws)) return nullptr;
    const int rc = enter(amx_gemm, u8(*t[0]), u8(*t[1]), u8(*t[2]), u8(*t[3]), M, N, K, (int)gs, (uint32_t)flags, f32(out), out.stride(0),
                         ws.data_ptr(), (size_t)ws.numel(), stream());
    if (rc) return fail("amx_gemm", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// quant_gemm(a, w_codes, w_scales, group_size, flags, out, workspace, w_bf16) -> out
PyObject* quant_gemm(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(8)
    const at::Tensor* x = device_matrix(a[0], at::kBFloat16, "a");
    if (!x) return nullptr;
    const at::Tensor *wc = nullptr, *ws_ = nullptr, *wb = nullptr;
    if (a[7] != Py_None) {
        wb = device_matrix(a[7], at::kBFloat16, "w_bf16");
        if (!wb || !require(a[1] == Py_None && a[2] == Py_None && wb->stride(1) == 1 && wb->size(1) == x->size(1),
                            "w_bf16 is a row-major matrix with the columns of a and the only weight"))
            return nullptr;
    } else if (!(wc = tensor(a[1], "w_codes")) || !(ws_ = tensor(a[2], "w_scales"))) return nullptr;
    const int64_t gs = as_int(a[3]), flags = as_int(a[4]);
    INTS_OK
    const int64_t M = x->size(0), K = x->size(1), N = wb ? wb->size(0) : wc->size(0);
    if (wc && !require(wc->numel() >= N * (K / 2) && (gs <= 0 || ws_->numel() >= N * (K / gs) * 2), "the weight has fewer columns than a"))
        return nullptr;
    at::Tensor out, ws;
    const size_t need = a[6] == Py_None
        ? amx_quant_gemm_workspace_bytes(M, N, K, (int)gs, ((uint32_t)flags & ~AMX_GEMM_CAST_IN_KERNEL) | (wb ? AMX_WEIGHT_BF16 : 0)) : 0;
    if (!out_and_workspace(a[5], a[6], M, N, at::kFloat, need, *x, out, ws)) return nullptr;
    const int rc = enter(amx_quant_gemm, x->data_ptr(), x->stride(0), wc ? u8(*wc) : nullptr, ws_ ? u8(*ws_) : nullptr,
                         wb ? wb->data_ptr() : nullptr, wb ? wb->stride(0) : 0, M, N, K, (int)gs, (uint32_t)flags, f32(out),
                         out.stride(0), ws.data_ptr(), (size_t)ws.numel(), stream());
    if (rc) return fail("amx_quant_gemm", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// quantize_prepared(x, is_weight, group_size, prepared, fmt, want_codes) -> (codes or None, scales, prepared)
PyObject* quantize_prepared(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(6)
    const at::Tensor* x = device_tensor(a[0], at::kBFloat16, "x");
    if (!x) return nullptr;
    const int is_weight = PyObject_IsTrue(a[1]), want_codes = PyObject_IsTrue(a[5]);
    const int64_t gs = as_int(a[2]), fmt = as_int(a[4]);
    INTS_OK
    if (!require(x->is_contiguous() && x->dim() == 2, "x must be a contiguous matrix")) return nullptr;
    if (gs <= 0) return fail("amx_quantize_prepared", AMX_ERR_SHAPE);
    const int64_t rows = x->size(0), K = x->size(1);
    at::Tensor codes, scales = empty({rows, K / gs, 2}, at::kByte, *x), buf;
    if (want_codes) codes = empty({rows, K / 2}, at::kByte, *x);
    if (a[3] != Py_None) {
        const at::Tensor* p = tensor(a[3], "prepared");
        if (!p) return nullptr;
        buf = *p;
    } else buf = scratch(amx_prepared_bytes(rows, K, (int)gs, is_weight), *x);
    const int rc = enter(amx_quantize_prepared_fmt, x->data_ptr(), rows, K, (int)gs, is_weight, (int)fmt, want_codes ? u8(codes) : nullptr,
                         u8(scales), buf.data_ptr(), (size_t)buf.numel(), stream());
    if (rc) return fail(fmt ? "amx_quantize_prepared_fmt" : "amx_quantize_prepared", rc);
    PyObject* r = PyTuple_New(3);
    if (want_codes) PyTuple_SET_ITEM(r, 0, wrap(codes));
    else {
        Py_INCREF(Py_None);
        PyTuple_SET_ITEM(r, 0, Py_None);
    }
    PyTuple_SET_ITEM(r, 1, wrap(scales));
    PyTuple_SET_ITEM(r, 2, wrap(buf));
    return r;
    END_HANDLE_TH_ERRORS
}

// gemm_prepared(a_prepared, w_prepared, M, N, K, group_size, out, workspace, sym, bf16) -> out
PyObject* gemm_prepared(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(10)
    const at::Tensor *pa = tensor(a[0], "a_prepared"), *pw = pa ? tensor(a[1], "w_prepared") : nullptr;
    if (!pw) return nullptr;
    const int64_t M = as_int(a[2]), N = as_int(a[3]), K = as_int(a[4]), gs = as_int(a[5]);
    const int sym = PyObject_IsTrue(a[8]);
    int bf16 = PyObject_IsTrue(a[9]);
    INTS_OK
    at::Tensor out, ws;
    const size_t need = a[7] == Py_None ? amx_gemm_prepared_workspace_bytes(M, N, K, (int)gs) : 0;
    if (!out_and_workspace(a[6], a[7], M, N, bf16 ? at::kBFloat16 : at::kFloat, need, *pa, out, ws)) return nullptr;
    bf16 = out.scalar_type() == at::kBFloat16;
    if (!bf16 && (!out.is_cuda() || out.scalar_type() != at::kFloat)) {
        PyErr_SetString(g_error, "out must be a CUDA tensor of torch.float32");
        return nullptr;
    }
    const int rc = enter(amx_gemm_prepared_ex, pa->data_ptr(), pw->data_ptr(), M, N, K, (int)gs,
                         (bf16 ? AMX_PREP_OUT_BF16 : 0) | (sym ? AMX_PREP_ONE_PLANE : 0), out.data_ptr(), out.stride(0),
                         ws.data_ptr(), (size_t)ws.numel(), stream());
    if (rc) return fail(bf16 ? "amx_gemm_prepared_ex" : "amx_gemm_prepared", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// attention_heads(q, k, v, flags, workspace) -> O fp32 [H, L, d]
PyObject* attention_heads(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(5)
    const at::Tensor* t[3];
    for (int i = 0; i < 3; ++i) {
        t[i] = device_tensor(a[i], at::kBFloat16, "q/k/v");
        if (!t[i] || !require(t[i]->dim() == 3 && t[i]->is_contiguous() && t[i]->size(1) == t[0]->size(1) && t[i]->size(2) == t[0]->size(2),
                              "q, k and v must be contiguous and agree in length and head dimension"))
            return nullptr;
    }
    if (!require(t[1]->size(0) == t[2]->size(0), "k and v must have the same number of heads")) return nullptr;
    const int64_t flags = as_int(a[3]);
    INTS_OK
    const int64_t H = t[0]->size(0), KV = t[1]->size(0), L = t[0]->size(1), d = t[0]->size(2);
    at::Tensor out, ws;
    if (a[4] == Py_None) ws = scratch(amx_attention_workspace_bytes_for(L, d, (uint32_t)flags), *t[0]);
    else {
        const at::Tensor* w = tensor(a[4], "workspace");
        if (!w) return nullptr;
        ws = *w;
    }
    out = empty({H, L, d}, at::kFloat, *t[0]);
    const int rc = enter(amx_attention_gqa, t[0]->data_ptr(), t[1]->data_ptr(), t[2]->data_ptr(), H, KV, L, d, (uint32_t)flags, f32(out),
                         ws.data_ptr(), (size_t)ws.numel(), stream());
    if (rc) return fail(KV == H ? "amx_attention" : "amx_attention_gqa", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

// quantize_nvfp4(x, asym, prepared_as: 0 none, 1 left, 2 right) -> (codes, scales, tensor_scale[, prepared])
PyObject* quantize_nvfp4(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(3)
    const at::Tensor* x = device_tensor(a[0], at::kBFloat16, "x");
    if (!x) return nullptr;
    const int asym = PyObject_IsTrue(a[1]);
    const int64_t as = as_int(a[2]);
    INTS_OK
    if (!require(x->dim() == 2 && x->stride(1) == 1, "x must be a row-major matrix")) return nullptr;
    const int64_t rows = x->size(0), K = x->size(1);
    at::Tensor codes = empty({rows, K / 2}, at::kByte, *x), scales = empty({rows, K / 16, 2}, at::kByte, *x),
               ts = empty({2}, at::kFloat, *x), prep;
    if (as) {
        prep = empty({(int64_t)amx_nvfp4_prepared_bytes(rows, K, as == 2)}, at::kByte, *x);
    }
    const int rc = enter(amx_quantize_nvfp4, x->data_ptr(), rows, K, x->stride(0), asym ? AMX_NV_ASYMMETRIC : 0, u8(codes), u8(scales), f32(ts),
                         as == 2, as ? prep.data_ptr() : nullptr, as ? (size_t)prep.numel() : 0, stream());
    if (rc) return fail("amx_quantize_nvfp4", rc);
    return as ? tuple({codes, scales, ts, prep}) : tuple({codes, scales, ts});
    END_HANDLE_TH_ERRORS
}

// gemm_nvfp4(a_prepared, w_prepared, M, N, K, workspace, sym) -> out
PyObject* gemm_nvfp4(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    ARGS(7)
    const at::Tensor *pa = tensor(a[0], "a_prepared"), *pw = pa ? tensor(a[1], "w_prepared") : nullptr;
    if (!pw) return nullptr;
    const int64_t M = as_int(a[2]), N = as_int(a[3]), K = as_int(a[4]);
    const int sym = PyObject_IsTrue(a[6]);
    INTS_OK
    at::Tensor out, ws;
    if (!out_and_workspace(Py_None, a[5], M, N, at::kFloat, 256, *pa, out, ws)) return nullptr;
    auto* fn = sym ? amx_gemm_nvfp4_sym : amx_gemm_nvfp4;
    const int rc = enter(fn, pa->data_ptr(), pw->data_ptr(), M, N, K, f32(out), N, ws.data_ptr(), (size_t)ws.numel(), stream());
    if (rc) return fail("amx_gemm_nvfp4", rc);
    return wrap(out);
    END_HANDLE_TH_ERRORS
}

PyObject* set_error(PyObject*, PyObject* cls) {
    Py_INCREF(cls);
    Py_XSETREF(g_error, cls);
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(quantize), FAST(fake_quantize), FAST(dequantize), FAST(quant_error), FAST(gemm), FAST(quant_gemm),
                         FAST(quantize_prepared), FAST(gemm_prepared), FAST(attention_heads), FAST(quantize_nvfp4), FAST(gemm_nvfp4),
                         {"set_error", set_error, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_amx_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__amx_native() { return PyModule_Create(&module); }
