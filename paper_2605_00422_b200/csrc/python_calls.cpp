// The per-call half of the Python binding: argument checks, device pointers and the current stream of the hot entry points, in
// native code.  Through ctypes a grouped call cost about 17 microseconds of interpreter time (argument arrays, type checks,
// stream lookup), more than the GPU needs for it at decode; here it is well under two.  The functions return the library's
// status; bwla.py turns it into an exception.  The library's entry points are handed over as addresses (`bind`), so that
// whichever build of the library the process has loaded is the one that is called.  As through ctypes, other threads run while the
// library works, and what PyTorch throws (a tensor without memory of its own, a stream of a device that is not there) becomes a Python
// exception.
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "bwla.h"

namespace {

struct Entry {
    decltype(&bwla_w1ax_linear_group) group;
    decltype(&bwla_w1ax_linear) linear;
    decltype(&bwla_layer_w1a16_linear) a16;
    decltype(&bwla_pack_signs) pack;
} entry;

PyObject *name_handle, *name_n, *name_k;      // of a layer: "_h", its handle as an integer; "N", "K"

const char* dtype_name(at::ScalarType t) {
    return t == at::kBFloat16 ? "torch.bfloat16" : t == at::kFloat ? "torch.float32" : t == at::kInt ? "torch.int32" : "another type";
}

// The tensor behind `o` when it is a CUDA tensor of this type (and number of dimensions), else NULL with TypeError set.
const at::Tensor* need(PyObject* o, at::ScalarType type, const char* name, int ndim) {
    const at::Tensor* t = THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr;
    if (!t || !t->is_cuda() || t->scalar_type() != type || (ndim > 0 && t->dim() != ndim)) {
        if (ndim > 0) PyErr_Format(PyExc_TypeError, "%s: expected a CUDA tensor of %s with %d dims", name, dtype_name(type), ndim);
        else PyErr_Format(PyExc_TypeError, "%s: expected a CUDA tensor of %s", name, dtype_name(type));
        return nullptr;
    }
    if (t->numel() > 0 && t->stride(-1) != 1) {
        PyErr_Format(PyExc_TypeError, "%s: innermost dimension must be contiguous", name);
        return nullptr;
    }
    return t;
}
const at::Tensor* tensor(PyObject* o, const char* name) {
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s: expected a tensor", name);
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}
void* stream() { return (void*)c10::cuda::getCurrentCUDAStream().stream(); }
// The layer's handle, NULL when it has been destroyed (the library refuses that); false with an exception set for other objects.
bool handle_of(PyObject* layer, const bwla_layer** out) {
    PyObject* h = PyObject_GetAttr(layer, name_handle);
    if (!h) return false;
    *out = h == Py_None ? nullptr : (const bwla_layer*)PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}
bool size_of(PyObject* layer, PyObject* name, int64_t* out) {
    PyObject* v = PyObject_GetAttr(layer, name);
    if (!v) return false;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}
// The library's call, with the interpreter free for other threads.
template <typename F, typename... A>
PyObject* unlocked(F entry_point, A... args) {
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = entry_point(args...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}
struct Ref {
    PyObject* o;
    explicit Ref(PyObject* p) : o(p) {}
    ~Ref() { Py_XDECREF(o); }
    Ref(const Ref&) = delete;
};

// group(layers, x, outs, workspace) -> status
PyObject* call_group(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    if (nargs != 4) { PyErr_SetString(PyExc_TypeError, "group(layers, x, outs, workspace)"); return nullptr; }
    const at::Tensor* x = need(args[1], at::kBFloat16, "x", 2);
    if (!x || PyObject_Size(args[0]) < 0 || PyObject_Size(args[2]) < 0) return nullptr;
    Ref layers(PySequence_Fast(args[0], "layers: expected a sequence")), outs(PySequence_Fast(args[2], "outs: expected a sequence"));
    if (!layers.o || !outs.o) return nullptr;
    constexpr Py_ssize_t kMost = 4;                   // what the library takes
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(layers.o), n_out = PySequence_Fast_GET_SIZE(outs.o);
    const int64_t M = x->size(0);
    const bwla_layer* h[kMost] = {};
    void* o[kMost] = {};                              // (fewer outputs than layers: the library refuses the missing ones)
    int64_t ldo[kMost] = {};
    for (Py_ssize_t i = 0; i < n_out; ++i) {
        const at::Tensor* t = need(PySequence_Fast_GET_ITEM(outs.o, i), at::kBFloat16, "out", 2);
        if (!t) return nullptr;
        if (i >= n) { PyErr_SetString(PyExc_IndexError, "more outputs than layers"); return nullptr; }
        if (i < kMost) { o[i] = t->data_ptr(); ldo[i] = t->stride(0); }
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject* layer = PySequence_Fast_GET_ITEM(layers.o, i);
        const bwla_layer* handle = nullptr;
        if (!handle_of(layer, &handle)) return nullptr;
        if (i >= kMost) continue;
        h[i] = handle;
        if (M == 0 && i < n_out && !size_of(layer, name_n, &ldo[i])) return nullptr;
    }
    const at::Tensor* ws = tensor(args[3], "workspace");
    if (!ws) return nullptr;
    return unlocked(entry.group, h, (int)n, (const void*)x->data_ptr(), M, M > 0 ? x->stride(0) : x->size(1), (void* const*)o, (const int64_t*)ldo,
                    ws->data_ptr(), (size_t)ws->numel(), stream());
    END_HANDLE_TH_ERRORS
}

// a16(layer, x, out, workspace) -> status
PyObject* call_a16(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    if (nargs != 4) { PyErr_SetString(PyExc_TypeError, "a16(layer, x, out, workspace)"); return nullptr; }
    const at::Tensor *x = need(args[1], at::kBFloat16, "x", 2), *out, *ws;
    if (!x || !(out = need(args[2], at::kBFloat16, "out", 2)) || !(ws = tensor(args[3], "workspace"))) return nullptr;
    const bwla_layer* h = nullptr;
    if (!handle_of(args[0], &h)) return nullptr;
    const int64_t M = x->size(0);
    int64_t ldx = x->stride(0), ldo = out->stride(0);
    if (M == 0 && (!size_of(args[0], name_k, &ldx) || !size_of(args[0], name_n, &ldo))) return nullptr;
    return unlocked(entry.a16, h, (const void*)x->data_ptr(), M, ldx, out->data_ptr(), ldo, ws->data_ptr(), (size_t)ws->numel(), stream());
    END_HANDLE_TH_ERRORS
}

// linear(x, P1, P2, bits, packed, alpha, U, V, mu, out, workspace) -> status; U, V, mu may be None
PyObject* call_linear(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    if (nargs != 11) { PyErr_SetString(PyExc_TypeError, "linear: eleven arguments"); return nullptr; }
    const at::Tensor *x = need(args[0], at::kBFloat16, "x", 2), *packed, *alpha, *U = nullptr, *V = nullptr, *mu = nullptr, *P1, *P2, *out, *ws;
    if (!x || !(packed = need(args[4], at::kInt, "packed", 2)) || !(alpha = need(args[5], at::kFloat, "alpha", 1))) return nullptr;
    const int64_t M = x->size(0), K = x->size(1), N = packed->size(0);
    int64_t r = 0;
    if (args[6] != Py_None) {
        if (!(U = need(args[6], at::kBFloat16, "U", 2)) || !(V = need(args[7], at::kBFloat16, "V", 2))) return nullptr;
        r = U->size(1);
        if (!U->is_contiguous() || !V->is_contiguous() || V->size(0) != r || V->size(1) != K || U->size(0) != N) {
            PyErr_SetString(PyExc_TypeError, "U must be contiguous [N][r] and V contiguous [r][K]");
            return nullptr;
        }
    }
    if (args[8] != Py_None && !(mu = need(args[8], at::kFloat, "mu", 1))) return nullptr;
    if (!(P1 = tensor(args[1], "P1")) || !(P2 = tensor(args[2], "P2"))) return nullptr;
    if (!packed->is_contiguous() || !P1->is_contiguous() || !P2->is_contiguous()) {
        PyErr_SetString(PyExc_TypeError, "packed, P1 and P2 must be contiguous");
        return nullptr;
    }
    if (!(out = need(args[9], at::kBFloat16, "out", 2)) || !(ws = tensor(args[10], "workspace"))) return nullptr;
    const long bits = PyLong_AsLong(args[3]);
    if (bits == -1 && PyErr_Occurred()) return nullptr;
    return unlocked(entry.linear, (const void*)x->data_ptr(), M, K, M > 0 ? x->stride(0) : K, (const float*)P1->data_ptr(), (int)P1->size(0),
                    (const float*)P2->data_ptr(), (int)P2->size(0), (int)bits, (const uint32_t*)packed->data_ptr(), (const float*)alpha->data_ptr(),
                    mu ? (const float*)mu->data_ptr() : nullptr, U ? (const void*)U->data_ptr() : nullptr, V ? (const void*)V->data_ptr() : nullptr, (int)r,
                    out->data_ptr(), N, M > 0 ? out->stride(0) : N, ws->data_ptr(), (size_t)ws->numel(), stream());
    END_HANDLE_TH_ERRORS
}

// pack(w, packed) -> status
PyObject* call_pack(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    if (nargs != 2) { PyErr_SetString(PyExc_TypeError, "pack(w, packed)"); return nullptr; }
    const at::Tensor* w = tensor(args[0], "w");
    if (!w) return nullptr;
    if (w->scalar_type() != at::kFloat && w->scalar_type() != at::kBFloat16) { PyErr_SetString(PyExc_TypeError, "w must be fp32 or bf16"); return nullptr; }
    const at::Tensor* packed;
    if (!need(args[0], w->scalar_type(), "w", 2) || !(packed = need(args[1], at::kInt, "packed", 2))) return nullptr;
    const int64_t N = w->size(0), K = w->size(1);
    return unlocked(entry.pack, (const void*)w->data_ptr(), w->scalar_type() == at::kFloat ? BWLA_DTYPE_F32 : BWLA_DTYPE_BF16, N, K,
                    N > 0 ? w->stride(0) : K, (uint32_t*)packed->data_ptr(), stream());
    END_HANDLE_TH_ERRORS
}

// bind(group, linear, a16, pack): the library's entry points as addresses
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != 4) { PyErr_SetString(PyExc_TypeError, "bind: four addresses"); return nullptr; }
    void* p[4];
    for (int i = 0; i < 4; ++i) {
        p[i] = PyLong_AsVoidPtr(args[i]);
        if (!p[i]) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: null address"); return nullptr; }
    }
    entry.group = (decltype(entry.group))p[0];
    entry.linear = (decltype(entry.linear))p[1];
    entry.a16 = (decltype(entry.a16))p[2];
    entry.pack = (decltype(entry.pack))p[3];
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
    {"group", (PyCFunction)(void (*)(void))call_group, METH_FASTCALL, nullptr},
    {"a16", (PyCFunction)(void (*)(void))call_a16, METH_FASTCALL, nullptr},
    {"linear", (PyCFunction)(void (*)(void))call_linear, METH_FASTCALL, nullptr},
    {"pack", (PyCFunction)(void (*)(void))call_pack, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) {
    name_handle = PyUnicode_InternFromString("_h");
    name_n = PyUnicode_InternFromString("N");
    name_k = PyUnicode_InternFromString("K");
    return name_handle && name_n && name_k ? PyModule_Create(&module_def) : nullptr;
}
