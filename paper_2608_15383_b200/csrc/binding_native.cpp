// CPython side of the calls a decode loop makes once or twice per layer: argument checks, output allocation, stream
// lookup and the C-ABI call, in C++.  Through ctypes and torch's Python API the same steps took 11 us of host time per
// call (17 us with outputs to allocate), more than the kernels of a one-token layer; here they take 1 to 2 us besides
// the launches themselves.  No arithmetic, no CUDA calls of its own: the entry points of libexmoe.so come in as
// addresses (set_entry_points), everything else is marshalling with the rules of binding.py.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>

#include "../../include/exmoe.h"

// read from the file before it is loaded (build.native_is_current)
extern "C" __attribute__((used)) const char exmoe_native_torch_tag[] = EXMOE_TORCH_TAG;

namespace {

decltype(&exmoe_route) g_route = nullptr;
decltype(&exmoe_moe_forward) g_forward = nullptr;
decltype(&exmoe_moe_forward_host) g_forward_host = nullptr;

PyObject *s_d_model, *s_d_ff, *s_experts, *s_top_k, *s_group, *s_cuda_stream;

PyObject* bad_tensor(const char* what, bool cuda, const char* dtype) {
    PyErr_Format(PyExc_ValueError, "%s: need a contiguous %s tensor of %s", what, cuda ? "CUDA" : "CPU", dtype);
    return nullptr;
}
const at::Tensor* tensor(PyObject* o, at::ScalarType dt, bool cuda, const char* what, const char* name) {
    if (THPVariable_Check(o)) {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.is_cuda() == cuda && t.scalar_type() == dt && t.is_contiguous()) return &t;
    }
    bad_tensor(what, cuda, name);
    return nullptr;
}
constexpr const char *kBf16 = "torch.bfloat16", *kF32 = "torch.float32", *kI32 = "torch.int32";

// int(o): whatever Python's int() takes, a float or a zero-dimensional array among them
bool to_int(PyObject* o, int* v) {
    PyObject* i = PyLong_CheckExact(o) ? Py_NewRef(o) : PyNumber_Long(o);
    if (!i) return false;
    const long x = PyLong_AsLong(i);
    Py_DECREF(i);
    if (x == -1 && PyErr_Occurred()) return false;
    *v = (int)x;
    return true;
}
bool int_attr(PyObject* o, PyObject* name, int* v) {
    PyObject* a = PyObject_GetAttr(o, name);
    if (!a) return false;
    const bool ok = to_int(a, v);
    Py_DECREF(a);
    return ok;
}
bool shape_of(PyObject* o, exmoe_shape* s) {
    if (!int_attr(o, s_d_model, &s->d_model) || !int_attr(o, s_d_ff, &s->d_ff) || !int_attr(o, s_experts, &s->num_experts) ||
        !int_attr(o, s_top_k, &s->top_k))
        return false;
    if (!int_attr(o, s_group, &s->group_size)) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
        PyErr_Clear();
        s->group_size = 128;
    }
    return true;
}
bool stream_of(PyObject* o, void** st) {
    if (o == Py_None) {
        *st = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject* a = PyObject_GetAttr(o, s_cuda_stream);
    if (!a) return false;
    *st = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
    return !(PyErr_Occurred());
}
at::Tensor empty_on(const at::Tensor& like, at::IntArrayRef sizes, at::ScalarType dt) {
    return at::detail::empty_cuda(sizes, dt, like.device(), std::nullopt);
}
// Every entry returns the result object, or the (non-zero) status as an int, or nullptr with an exception set (torch's
// own, an exhausted allocator among them, translated as torch does).
template <typename F>
PyObject* guarded(F f) {
    HANDLE_TH_ERRORS
    return f();
    END_HANDLE_TH_ERRORS
}

// route(shape, hidden, w_router, bias, topk_ids, topk_weights, stream) -> (ids, weights)
PyObject* route(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 7) return PyErr_Format(PyExc_TypeError, "route: 7 arguments");
    return guarded([&]() -> PyObject* {
        exmoe_shape s;
        if (!shape_of(a[0], &s)) return nullptr;
        const at::Tensor *h, *w, *b = nullptr, *i = nullptr, *p = nullptr;
        if (!(h = tensor(a[1], at::kBFloat16, true, "hidden", kBf16))) return nullptr;
        if (!(w = tensor(a[2], at::kBFloat16, true, "w_router", kBf16))) return nullptr;
        if (a[3] != Py_None && !(b = tensor(a[3], at::kFloat, true, "bias", kF32))) return nullptr;
        if (a[4] != Py_None && !(i = tensor(a[4], at::kInt, true, "topk_ids", kI32))) return nullptr;
        if (a[5] != Py_None && !(p = tensor(a[5], at::kFloat, true, "topk_weights", kF32))) return nullptr;
        void* st;
        if (!stream_of(a[6], &st)) return nullptr;
        const int T = (int)h->size(0);
        at::Tensor ids = i ? *i : empty_on(*h, {T, s.top_k}, at::kInt);
        at::Tensor wts = p ? *p : empty_on(*h, {T, s.top_k}, at::kFloat);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = g_route(&s, h->data_ptr(), w->data_ptr(), b ? static_cast<const float*>(b->data_ptr()) : nullptr, T,
                     static_cast<int32_t*>(ids.data_ptr()), static_cast<float*>(wts.data_ptr()), st);
        Py_END_ALLOW_THREADS
        if (rc) return PyLong_FromLong(rc);
        PyObject* oi = i ? Py_NewRef(a[4]) : THPVariable_Wrap(std::move(ids));
        PyObject* op = p ? Py_NewRef(a[5]) : THPVariable_Wrap(std::move(wts));
        PyObject* r = oi && op ? PyTuple_Pack(2, oi, op) : nullptr;
        Py_XDECREF(oi);
        Py_XDECREF(op);
        return r;
    });
}

// forward(handle, layer, hidden, topk_ids, topk_weights, out, stream) -> out
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 7) return PyErr_Format(PyExc_TypeError, "forward: 7 arguments");
    return guarded([&]() -> PyObject* {
        exmoe_cache* c = static_cast<exmoe_cache*>(PyLong_AsVoidPtr(a[0]));
        int layer;
        if (PyErr_Occurred() || !to_int(a[1], &layer)) return nullptr;
        const at::Tensor *h, *i, *p, *o = nullptr;
        if (!(h = tensor(a[2], at::kBFloat16, true, "hidden", kBf16))) return nullptr;
        if (!(i = tensor(a[3], at::kInt, true, "topk_ids", kI32))) return nullptr;
        if (!(p = tensor(a[4], at::kFloat, true, "topk_weights", kF32))) return nullptr;
        if (a[5] != Py_None && !(o = tensor(a[5], at::kBFloat16, true, "out", kBf16))) return nullptr;
        void* st;
        if (!stream_of(a[6], &st)) return nullptr;
        at::Tensor out = o ? *o : empty_on(*h, h->sizes(), at::kBFloat16);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = g_forward(c, layer, h->data_ptr(), static_cast<const int32_t*>(i->data_ptr()), static_cast<const float*>(p->data_ptr()),
                       (int)h->size(0), out.data_ptr(), st);
        Py_END_ALLOW_THREADS
        if (rc) return PyLong_FromLong(rc);
        return o ? Py_NewRef(a[5]) : THPVariable_Wrap(std::move(out));
    });
}

// forward_host(handle, layer, hidden, topk_ids, topk_weights, out, stream) -> None (host tensors, `out` given)
PyObject* forward_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 7) return PyErr_Format(PyExc_TypeError, "forward_host: 7 arguments");
    return guarded([&]() -> PyObject* {
        exmoe_cache* c = static_cast<exmoe_cache*>(PyLong_AsVoidPtr(a[0]));
        int layer;
        if (PyErr_Occurred() || !to_int(a[1], &layer)) return nullptr;
        const at::Tensor *h, *i, *p, *o;
        if (!(h = tensor(a[2], at::kBFloat16, false, "hidden", kBf16))) return nullptr;
        if (!(i = tensor(a[3], at::kInt, false, "topk_ids", kI32))) return nullptr;
        if (!(p = tensor(a[4], at::kFloat, false, "topk_weights", kF32))) return nullptr;
        if (!(o = tensor(a[5], at::kBFloat16, false, "out", kBf16))) return nullptr;
        void* st;
        if (!stream_of(a[6], &st)) return nullptr;
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = g_forward_host(c, layer, h->data_ptr(), static_cast<const int32_t*>(i->data_ptr()),
                            static_cast<const float*>(p->data_ptr()), (int)h->size(0), o->data_ptr(), st);
        Py_END_ALLOW_THREADS
        if (rc) return PyLong_FromLong(rc);
        Py_RETURN_NONE;
    });
}

// set_entry_points(exmoe_route, exmoe_moe_forward, exmoe_moe_forward_host): addresses in the loaded libexmoe.so
PyObject* set_entry_points(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != 3) return PyErr_Format(PyExc_TypeError, "set_entry_points: 3 addresses");
    g_route = reinterpret_cast<decltype(g_route)>(PyLong_AsVoidPtr(a[0]));
    g_forward = reinterpret_cast<decltype(g_forward)>(PyLong_AsVoidPtr(a[1]));
    g_forward_host = reinterpret_cast<decltype(g_forward_host)>(PyLong_AsVoidPtr(a[2]));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"route", reinterpret_cast<PyCFunction>(route), METH_FASTCALL, nullptr},
    {"forward", reinterpret_cast<PyCFunction>(forward), METH_FASTCALL, nullptr},
    {"forward_host", reinterpret_cast<PyCFunction>(forward_host), METH_FASTCALL, nullptr},
    {"set_entry_points", reinterpret_cast<PyCFunction>(set_entry_points), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_exmoe_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__exmoe_native(void) {
    s_d_model = PyUnicode_InternFromString("d_model");
    s_d_ff = PyUnicode_InternFromString("d_ff");
    s_experts = PyUnicode_InternFromString("num_experts");
    s_top_k = PyUnicode_InternFromString("top_k");
    s_group = PyUnicode_InternFromString("group_size");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return PyModule_Create(&module);
}
