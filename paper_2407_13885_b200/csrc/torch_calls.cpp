// Native form of the tensor entry points in binding.py: checks the arguments, allocates the result, looks up the stream
// and calls the C ABI of libattnw.so.  No arithmetic of the method is here.
//
// Why it exists: a small call spends 3 to 13 us on the GPU, and the same steps in Python (argument checks, torch.empty,
// device context, current stream, ctypes marshalling) took 13 to 20 us, so the host was the bound of every small call.  Now 4.5 to 7 us: softmax_rows
// of 4096 x 1000 float32 back to back 13.4 -> 6.3 us (5.0 us on the GPU), one head of 256 keys 15.4 -> 12.3 us.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

#include "../../include/attnw.h"

namespace {

PyObject* g_error = nullptr;  // binding.AttnwError, handed over once by binding.py

// A tensor without storage (torch.func's wrappers) throws when it is asked for its address, so every entry point asks while it
// holds the interpreter's lock: HANDLE_TH_ERRORS needs the lock to turn the exception into a Python one.

// A CUDA tensor of the wanted type, contiguous and on the device of the call's first tensor (`like`; nullptr for that one itself, and
// its kernel would read another GPU's memory); nullptr with a Python exception set otherwise.
const at::Tensor* tensor_arg(PyObject* obj, const char* name, at::ScalarType type, const char* type_name, const at::Tensor* like) {
    if (!THPVariable_Check(obj) || !THPVariable_Unpack(obj).is_cuda()) {
        PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor", name);
        return nullptr;
    }
    const at::Tensor& t = THPVariable_Unpack(obj);
    if (t.scalar_type() != type) {
        PyErr_Format(PyExc_TypeError, "%s must have dtype %s, got %s", name, type_name, at::toString(t.scalar_type()));
        return nullptr;
    }
    if (!t.is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
        return nullptr;
    }
    if (like && t.device() != like->device()) {
        PyErr_Format(PyExc_ValueError, "%s must be on %s like the other tensors, got %s", name, like->device().str().c_str(),
                     t.device().str().c_str());
        return nullptr;
    }
    return &t;
}

const at::Tensor* bf16_arg(PyObject* obj, const char* name, const at::Tensor* like) {
    return tensor_arg(obj, name, at::kBFloat16, "torch.bfloat16", like);
}

// The result: the caller's tensor `obj` (bfloat16, or also float32 where `f32_allowed`), or a new one where it is None.
bool output_arg(PyObject* obj, const char* name, at::IntArrayRef shape, at::ScalarType new_type, bool f32_allowed, bool exact_type,
                const char* shape_text, const at::Tensor& like, at::Tensor* out) {
    if (obj == Py_None) {
        *out = at::empty(shape, like.options().dtype(new_type).requires_grad(false));
        return true;
    }
    const bool f32 = f32_allowed && THPVariable_Check(obj) && THPVariable_Unpack(obj).scalar_type() == at::kFloat;
    if (exact_type || f32 || (THPVariable_Check(obj) && THPVariable_Unpack(obj).scalar_type() == at::kBFloat16)) {
        const at::Tensor* t = tensor_arg(obj, name, f32 ? at::kFloat : at::kBFloat16, f32 ? "torch.float32" : "torch.bfloat16", &like);
        if (!t) return false;
        if (t->sizes() == shape) {
            *out = *t;
            return true;
        }
    } else if (!THPVariable_Check(obj) || !THPVariable_Unpack(obj).is_cuda()) {
        PyErr_Format(PyExc_TypeError, "%s must be a CUDA tensor", name);
        return false;
    }
    PyErr_Format(PyExc_ValueError, "%s must be %s", name, shape_text);
    return false;
}

// Same meaning as in Python: None = torch's current stream of the device that is current.
bool stream_arg(PyObject* obj, void** out) {
    if (obj == Py_None) {
        *out = static_cast<void*>(c10::cuda::getCurrentCUDAStream().stream());
        return true;
    }
    *out = PyLong_AsVoidPtr(obj);
    return !PyErr_Occurred();
}

bool float_arg(PyObject* obj, float* out) {
    PyObject* f = PyNumber_Float(obj);
    if (!f) return false;
    *out = static_cast<float>(PyFloat_AS_DOUBLE(f));
    Py_DECREF(f);
    return true;
}

PyObject* failed(int code, const char* where) {
    PyObject* e = PyObject_CallFunction(g_error, "is", code, where);
    if (e) {
        PyErr_SetObject(g_error, e);
        Py_DECREF(e);
    }
    return nullptr;
}

bool count_is(Py_ssize_t n, Py_ssize_t want) {
    if (n != want) PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return n == want;
}

// None = torch's default type, as everywhere in torch.
bool is_float32(PyObject* dtype, bool* f32) {
    if (dtype == Py_None || THPDtype_Check(dtype)) {
        const at::ScalarType t = dtype == Py_None ? c10::get_default_dtype_as_scalartype() : reinterpret_cast<THPDtype*>(dtype)->scalar_type;
        *f32 = t == at::kFloat;
        if (*f32 || t == at::kBFloat16) return true;
    }
    PyErr_SetString(PyExc_ValueError, "out_dtype must be torch.bfloat16 or torch.float32");
    return false;
}

// attnw_fused(Q, K, scale, P, out_dtype, stream)
PyObject* py_attnw_fused(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!count_is(n, 6)) return nullptr;
    const at::Tensor *q, *k;
    if (!(q = bf16_arg(a[0], "Q", nullptr)) || !(k = bf16_arg(a[1], "K", q))) return nullptr;
    if (q->dim() != 4 || q->sizes() != k->sizes()) {
        PyErr_SetString(PyExc_ValueError, "Q and K must both be [B, H, N, d]");
        return nullptr;
    }
    const int64_t B = q->size(0), H = q->size(1), N = q->size(2), d = q->size(3);
    bool f32 = false;
    float scale;
    if ((a[3] == Py_None && !is_float32(a[4], &f32)) || !float_arg(a[2], &scale)) return nullptr;
    const void *q_ptr = q->data_ptr(), *k_ptr = k->data_ptr();
    at::Tensor p;
    if (!output_arg(a[3], "P", {B, H, N, N}, f32 ? at::kFloat : at::kBFloat16, true, false,
                    "[B, H, N, N] in bfloat16 or float32", *q, &p))
        return nullptr;
    const c10::cuda::CUDAGuard guard(q->device());
    void* stream;
    if (!stream_arg(a[5], &stream)) return nullptr;
    const auto entry = p.scalar_type() == at::kBFloat16 ? attnw_fused : attnw_fused_f32;
    void* p_ptr = p.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = entry(q_ptr, k_ptr, p_ptr, static_cast<int>(B), static_cast<int>(H), static_cast<int>(N), static_cast<int>(d), scale, stream);
    Py_END_ALLOW_THREADS
    if (rc != ATTNW_OK) return failed(rc, "attnw_fused");
    if (a[3] != Py_None) return Py_NewRef(a[3]);
    return THPVariable_Wrap(std::move(p));
    END_HANDLE_TH_ERRORS
}

// attn_fused(Q, K, V, scale, O, stream)
PyObject* py_attn_fused(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!count_is(n, 6)) return nullptr;
    const at::Tensor *q, *k, *v;
    if (!(q = bf16_arg(a[0], "Q", nullptr)) || !(k = bf16_arg(a[1], "K", q)) || !(v = bf16_arg(a[2], "V", q))) return nullptr;
    if (q->dim() != 4 || q->sizes() != k->sizes() || q->sizes() != v->sizes()) {
        PyErr_SetString(PyExc_ValueError, "Q, K and V must all be [B, H, N, d]");
        return nullptr;
    }
    float scale;
    if (!float_arg(a[3], &scale)) return nullptr;
    const void *q_ptr = q->data_ptr(), *k_ptr = k->data_ptr(), *v_ptr = v->data_ptr();
    const int B = static_cast<int>(q->size(0)), H = static_cast<int>(q->size(1)), N = static_cast<int>(q->size(2)), d = static_cast<int>(q->size(3));
    at::Tensor o;
    if (!output_arg(a[4], "O", q->sizes(), at::kBFloat16, false, true, "[B, H, N, d]", *q, &o)) return nullptr;
    const c10::cuda::CUDAGuard guard(q->device());
    void* stream;
    if (!stream_arg(a[5], &stream)) return nullptr;
    void* o_ptr = o.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = attn_fused(q_ptr, k_ptr, v_ptr, o_ptr, B, H, N, d, scale, stream);
    Py_END_ALLOW_THREADS
    if (rc != ATTNW_OK) return failed(rc, "attn_fused");
    if (a[4] != Py_None) return Py_NewRef(a[4]);
    return THPVariable_Wrap(std::move(o));
    END_HANDLE_TH_ERRORS
}

// project_qk(X, Wq, Wk, Q, K, stream)
PyObject* py_project_qk(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!count_is(n, 6)) return nullptr;
    const at::Tensor *x, *wq, *wk;
    if (!(x = bf16_arg(a[0], "X", nullptr)) || !(wq = bf16_arg(a[1], "Wq", x)) || !(wk = bf16_arg(a[2], "Wk", x))) return nullptr;
    if (x->dim() != 3 || wq->dim() != 3 || wq->sizes() != wk->sizes() || wq->size(2) != x->size(2)) {
        PyErr_SetString(PyExc_ValueError, "X must be [B, N, d_model] and Wq, Wk [H, d, d_model]");
        return nullptr;
    }
    const int64_t B = x->size(0), N = x->size(1), d_model = x->size(2), H = wq->size(0), d = wq->size(1);
    const void *x_ptr = x->data_ptr(), *wq_ptr = wq->data_ptr(), *wk_ptr = wk->data_ptr();
    at::Tensor q, k;
    if (!output_arg(a[3], "Q", {B, H, N, d}, at::kBFloat16, false, true, "[B, H, N, d]", *x, &q) ||
        !output_arg(a[4], "K", {B, H, N, d}, at::kBFloat16, false, true, "[B, H, N, d]", *x, &k))
        return nullptr;
    const c10::cuda::CUDAGuard guard(x->device());
    void* stream;
    if (!stream_arg(a[5], &stream)) return nullptr;
    void *q_ptr = q.data_ptr(), *k_ptr = k.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = attnw_project_qk(x_ptr, wq_ptr, wk_ptr, q_ptr, k_ptr, static_cast<int>(B), static_cast<int>(N), static_cast<int>(d_model),
                          static_cast<int>(H), static_cast<int>(d), stream);
    Py_END_ALLOW_THREADS
    if (rc != ATTNW_OK) return failed(rc, "attnw_project_qk");
    PyObject* pq = a[3] != Py_None ? Py_NewRef(a[3]) : THPVariable_Wrap(std::move(q));
    PyObject* pk = a[4] != Py_None ? Py_NewRef(a[4]) : THPVariable_Wrap(std::move(k));
    PyObject* pair = pq && pk ? PyTuple_Pack(2, pq, pk) : nullptr;
    Py_XDECREF(pq);
    Py_XDECREF(pk);
    return pair;
    END_HANDLE_TH_ERRORS
}

// softmax_rows(S, P, out_dtype, stream)
PyObject* py_softmax_rows(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (!count_is(n, 4)) return nullptr;
    const at::Tensor* s = tensor_arg(a[0], "S", at::kFloat, "torch.float32", nullptr);
    if (!s) return nullptr;
    if (s->dim() != 2) {
        PyErr_SetString(PyExc_ValueError, "S must be [rows, cols]");
        return nullptr;
    }
    bool f32 = false;
    if (a[1] == Py_None && !is_float32(a[2], &f32)) return nullptr;
    const long long rows = s->size(0), cols = s->size(1);
    const void* s_ptr = s->data_ptr();
    at::Tensor p;
    if (!output_arg(a[1], "P", s->sizes(), f32 ? at::kFloat : at::kBFloat16, true, false,
                    "[rows, cols] in bfloat16 or float32", *s, &p))
        return nullptr;
    const c10::cuda::CUDAGuard guard(s->device());
    void* stream;
    if (!stream_arg(a[3], &stream)) return nullptr;
    const auto entry = p.scalar_type() == at::kBFloat16 ? softmax_rows : softmax_rows_f32;
    void* p_ptr = p.data_ptr();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = entry(s_ptr, p_ptr, rows, cols, stream);
    Py_END_ALLOW_THREADS
    if (rc != ATTNW_OK) return failed(rc, "softmax_rows");
    if (a[1] != Py_None) return Py_NewRef(a[1]);
    return THPVariable_Wrap(std::move(p));
    END_HANDLE_TH_ERRORS
}

PyObject* py_set_error(PyObject*, PyObject* type) {
    Py_XSETREF(g_error, Py_NewRef(type));
    Py_RETURN_NONE;
}

template <typename F>
PyCFunction fast(F f) {
    return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f));
}

PyMethodDef g_methods[] = {
    {"attnw_fused", fast(py_attnw_fused), METH_FASTCALL, "attnw_fused(Q, K, scale, P, out_dtype, stream)"},
    {"attn_fused", fast(py_attn_fused), METH_FASTCALL, "attn_fused(Q, K, V, scale, O, stream)"},
    {"project_qk", fast(py_project_qk), METH_FASTCALL, "project_qk(X, Wq, Wk, Q, K, stream)"},
    {"softmax_rows", fast(py_softmax_rows), METH_FASTCALL, "softmax_rows(S, P, out_dtype, stream)"},
    {"set_error", py_set_error, METH_O, "the exception type for attnw status codes"},
    {nullptr, nullptr, 0, nullptr},
};
#ifndef ATTNW_BUILT_FOR
#error "build.py passes the torch and the Python that the module is built for and looks for them in it later"
#endif
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_attnw_torch", ATTNW_BUILT_FOR, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__attnw_torch() { return PyModule_Create(&g_module); }
