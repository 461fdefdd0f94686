// Marshalling of the calls of a decode step (append, predict, decode) for torch: checks the tensors, takes their device
// pointers and the current stream, and calls the C ABI.  Nothing is computed or kept here.
//
// Through ctypes the checks and conversions of a step's 30 arguments took 20 us of Python, more than a small step takes on
// the GPU; here they take about 2.  The entry points arrive as addresses (ctypes holds the library), so this module links
// only against torch.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "../../include/eta.h"

namespace {

// classes of the binding: the exception, the ctypes structures
PyObject* g_error = nullptr;
PyObject *g_desc = nullptr, *g_pages = nullptr, *g_decode_params = nullptr, *g_params = nullptr;

bool fail(const char* name, const char* what) {
    PyErr_Format(g_error, "%s must be %s", name, what);
    return false;
}

const char* dtype_name(at::ScalarType t) {
    switch (t) {
        case at::kBFloat16: return "torch.bfloat16";
        case at::kFloat: return "torch.float32";
        case at::kInt: return "torch.int32";
        case at::kByte: return "torch.uint8";
        case at::kHalf: return "torch.float16";
        default: return nullptr;
    }
}

// Device pointer of a CUDA tensor of the given type; None gives a null pointer.  With `pinned`, a page-locked host tensor
// passes too (the device can address it as it is).
bool pointer(PyObject* o, at::ScalarType type, const char* name, void** out, bool pinned = false, at::ScalarType other = at::ScalarType::Undefined) {
    *out = nullptr;
    if (o == Py_None) return true;
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor or None", name);
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() && !(pinned && t.is_pinned())) return fail(name, "a CUDA tensor (no CPU path exists)");
    const at::ScalarType s = t.scalar_type();
    if (s != type && (other == at::ScalarType::Undefined || s != other)) {
        const char* got = dtype_name(s);
        if (other != at::ScalarType::Undefined)
            PyErr_Format(g_error, "%s must be float16 (compact records) or uint8 (packed records), got %s", name, got ? got : "another type");
        else
            PyErr_Format(g_error, "%s must be %s, got %s", name, dtype_name(type), got ? got : "another type");
        return false;
    }
    *out = t.data_ptr();
    return true;
}
bool musig_pointer(PyObject* o, void** out) { return pointer(o, at::kHalf, "musig", out, false, at::kByte); }

// The bytes of a ctypes structure of the binding's class `cls`
template <typename T>
struct Struct {
    Py_buffer view = {};
    bool held = false;
    const T* get(PyObject* o, PyObject* cls) {
        const int is = PyObject_IsInstance(o, cls);
        if (is <= 0) {
            if (is == 0) PyErr_Format(PyExc_TypeError, "%R expected, got %s", cls, Py_TYPE(o)->tp_name);
            return nullptr;
        }
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return nullptr;
        held = true;
        if ((size_t)view.len != sizeof(T)) {
            PyErr_SetString(PyExc_TypeError, "a structure of the wrong size");
            return nullptr;
        }
        return static_cast<const T*>(view.buf);
    }
    ~Struct() { if (held) PyBuffer_Release(&view); }
};

bool number(PyObject* o, const char* name, double* out) {
    PyObject* v = PyObject_GetAttrString(o, name);
    if (!v) return false;
    *out = PyFloat_AsDouble(v);
    Py_DECREF(v);
    return !(*out == -1.0 && PyErr_Occurred());
}
// what a ctypes integer field makes of a value: any integer (or what has __index__), modulo 2^32; floats are refused
bool integer(PyObject* o, const char* name, uint32_t* out) {
    PyObject* v = PyObject_GetAttrString(o, name);
    if (!v) return false;
    *out = (uint32_t)PyLong_AsUnsignedLongMask(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}
// A DecodeParams is read field by field, with the results its c() would have; anything else goes through its c().
bool params_of(PyObject* o, eta_params* p) {
    if ((PyObject*)Py_TYPE(o) != g_decode_params) {
        PyObject* c = PyObject_CallMethod(o, "c", nullptr);
        if (!c) return false;
        bool ok;
        {
            Struct<eta_params> ps;
            const eta_params* from = ps.get(c, g_params);
            ok = from != nullptr;
            if (ok) *p = *from;
        }
        Py_DECREF(c);
        return ok;
    }
    double z, a, beta, scale;
    uint32_t lwb, window;
    if (!number(o, "z", &z) || !number(o, "a", &a) || !number(o, "beta", &beta) || !number(o, "scale", &scale) ||
        !integer(o, "lwb", &lwb) || !integer(o, "rescue_window", &window) || !integer(o, "flags", &p->flags))
        return false;
    p->z = (float)z; p->a = (float)a; p->beta = (float)beta; p->scale = (float)scale;
    p->lwb = (int32_t)lwb; p->rescue_window = (int32_t)window;
    return true;
}

template <typename F>
bool entry(PyObject* o, F* out) {
    *out = reinterpret_cast<F>(PyLong_AsVoidPtr(o));
    return *out || !PyErr_Occurred();
}

bool count(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
    return false;
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

#define PTR(o, type, name) pointer(o, type, #name, (void**)&name)

// (address, desc, [pages,] K, seq_lens, musig, mnorm, flags) -> return code
template <bool PAGED>
PyObject* append(PyObject*, PyObject* const* v, Py_ssize_t n) {
    using Plain = int (*)(const eta_cache_desc*, const void*, const int32_t*, void*, float*, uint32_t, void*);
    using Paged = int (*)(const eta_cache_desc*, const eta_page_table*, const void*, const int32_t*, void*, float*, uint32_t, void*);
    void* fn;
    Struct<eta_cache_desc> ds;
    Struct<eta_page_table> ps;
    void *K, *seq_lens, *musig, *mnorm;
    if (!count(n, PAGED ? 8 : 7) || !entry(v[0], &fn)) return nullptr;
    const eta_cache_desc* desc = ds.get(v[1], g_desc);
    if (!desc) return nullptr;
    const eta_page_table* pages = nullptr;
    if (PAGED && !(pages = ps.get(v[2], g_pages))) return nullptr;
    v += PAGED ? 3 : 2;
    if (!PTR(v[0], at::kBFloat16, K) || !PTR(v[1], at::kInt, seq_lens) || !musig_pointer(v[2], &musig) || !PTR(v[3], at::kFloat, mnorm))
        return nullptr;
    const uint32_t flags = (uint32_t)PyLong_AsUnsignedLongMask(v[4]);
    if (PyErr_Occurred()) return nullptr;
    void* const s = stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    if (PAGED) rc = reinterpret_cast<Paged>(fn)(desc, pages, K, (const int32_t*)seq_lens, musig, (float*)mnorm, flags, s);
    else rc = reinterpret_cast<Plain>(fn)(desc, K, (const int32_t*)seq_lens, musig, (float*)mnorm, flags, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// (address, q, W, bias, tau) -> return code
PyObject* predict(PyObject*, PyObject* const* v, Py_ssize_t n) {
    using F = int (*)(int32_t, int32_t, int32_t, const void*, const float*, const float*, float*, void*);
    F fn;
    void *q, *W, *bias, *tau;
    if (!count(n, 5) || !entry(v[0], &fn)) return nullptr;
    if (!THPVariable_Check(v[1])) { PyErr_SetString(PyExc_TypeError, "q must be a torch.Tensor"); return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(v[1]);
    if (t.dim() != 3) { PyErr_SetString(PyExc_ValueError, "q must be [batch, n_q_heads, head_dim]"); return nullptr; }
    const int32_t b = (int32_t)t.size(0), h = (int32_t)t.size(1), d = (int32_t)t.size(2);
    if (!PTR(v[1], at::kBFloat16, q) || !PTR(v[2], at::kFloat, W) || !PTR(v[3], at::kFloat, bias) || !PTR(v[4], at::kFloat, tau))
        return nullptr;
    void* const s = stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(b, h, d, q, (const float*)W, (const float*)bias, (float*)tau, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// (address, desc, [pages,] params, q, K, V, seq_lens, musig, mnorm, tau, head_const, out, sel_mask, stats, status
//  [, workspace]) -> return code
enum class Decode { PLAIN, PAGED, STATIC };
template <Decode KIND>
PyObject* decode(PyObject*, PyObject* const* v, Py_ssize_t n) {
    using Plain = int (*)(const eta_cache_desc*, const eta_params*, const void*, const void*, const void*, const int32_t*, const void*,
                          const float*, const float*, const float*, float*, uint8_t*, int32_t*, uint32_t*, void*, size_t, void*);
    using Paged = int (*)(const eta_cache_desc*, const eta_page_table*, const eta_params*, const void*, const void*, const void*,
                          const int32_t*, const void*, const float*, const float*, const float*, float*, uint8_t*, int32_t*,
                          uint32_t*, void*, size_t, void*);
    using Static = int (*)(const eta_cache_desc*, const eta_params*, const void*, const void*, const void*, const int32_t*, const void*,
                           const float*, const float*, const float*, float*, uint8_t*, int32_t*, uint32_t*, void*);
    constexpr bool PAGED = KIND == Decode::PAGED, WS = KIND != Decode::STATIC;
    void* fn;
    Struct<eta_cache_desc> ds;
    Struct<eta_page_table> ps;
    eta_params p;
    void *q, *K, *V, *seq_lens, *musig, *mnorm, *tau, *head_const, *out, *sel_mask, *stats, *status, *workspace = nullptr;
    if (!count(n, 15 + PAGED + WS) || !entry(v[0], &fn)) return nullptr;
    const eta_cache_desc* desc = ds.get(v[1], g_desc);
    if (!desc) return nullptr;
    const eta_page_table* pages = nullptr;
    if (PAGED && !(pages = ps.get(v[2], g_pages))) return nullptr;
    v += PAGED ? 3 : 2;
    if (!params_of(v[0], &p)) return nullptr;
    if (!PTR(v[1], at::kBFloat16, q) || !PTR(v[2], at::kBFloat16, K) || !PTR(v[3], at::kBFloat16, V) || !PTR(v[4], at::kInt, seq_lens) ||
        !musig_pointer(v[5], &musig) || !PTR(v[6], at::kFloat, mnorm) || !PTR(v[7], at::kFloat, tau) ||
        !PTR(v[8], at::kFloat, head_const) || !pointer(v[9], at::kFloat, "out", &out, true) || !PTR(v[10], at::kByte, sel_mask) ||
        !PTR(v[11], at::kInt, stats) || !PTR(v[12], at::kInt, status) || (WS && !PTR(v[13], at::kByte, workspace)))
        return nullptr;
    const size_t bytes = workspace ? (size_t)THPVariable_Unpack(v[13]).numel() : 0;
    void* const s = stream();
    int rc;
    Py_BEGIN_ALLOW_THREADS
    if (KIND == Decode::PAGED)
        rc = reinterpret_cast<Paged>(fn)(desc, pages, &p, q, K, V, (const int32_t*)seq_lens, musig, (const float*)mnorm, (const float*)tau,
                                         (const float*)head_const, (float*)out, (uint8_t*)sel_mask, (int32_t*)stats,
                                         (uint32_t*)status, workspace, bytes, s);
    else if (KIND == Decode::PLAIN)
        rc = reinterpret_cast<Plain>(fn)(desc, &p, q, K, V, (const int32_t*)seq_lens, musig, (const float*)mnorm, (const float*)tau,
                                         (const float*)head_const, (float*)out, (uint8_t*)sel_mask, (int32_t*)stats,
                                         (uint32_t*)status, workspace, bytes, s);
    else
        rc = reinterpret_cast<Static>(fn)(desc, &p, q, K, V, (const int32_t*)seq_lens, musig, (const float*)mnorm, (const float*)tau,
                                          (const float*)head_const, (float*)out, (uint8_t*)sel_mask, (int32_t*)stats,
                                          (uint32_t*)status, s);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// the eta_params a call would get, as bytes (for the tests)
PyObject* params(PyObject*, PyObject* const* v, Py_ssize_t n) {
    eta_params p;
    if (!count(n, 1) || !params_of(v[0], &p)) return nullptr;
    return PyBytes_FromStringAndSize(reinterpret_cast<const char*>(&p), sizeof p);
}

// (EtaError, CacheDesc, PageTable, DecodeParams, Params)
PyObject* set_classes(PyObject*, PyObject* const* v, Py_ssize_t n) {
    if (!count(n, 5)) return nullptr;
    PyObject** const to[5] = {&g_error, &g_desc, &g_pages, &g_decode_params, &g_params};
    for (int k = 0; k < 5; ++k) {
        Py_INCREF(v[k]);
        Py_XSETREF(*to[k], v[k]);
    }
    Py_RETURN_NONE;
}

// no C++ exception (torch reports its errors with them) crosses into the interpreter
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* v, Py_ssize_t n) {
    try {
        return F(self, v, n);
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

PyMethodDef methods[] = {
    {"append", (PyCFunction)(void (*)(void))guarded<append<false>>, METH_FASTCALL, nullptr},
    {"append_paged", (PyCFunction)(void (*)(void))guarded<append<true>>, METH_FASTCALL, nullptr},
    {"predict", (PyCFunction)(void (*)(void))guarded<predict>, METH_FASTCALL, nullptr},
    {"decode", (PyCFunction)(void (*)(void))guarded<decode<Decode::PLAIN>>, METH_FASTCALL, nullptr},
    {"decode_paged", (PyCFunction)(void (*)(void))guarded<decode<Decode::PAGED>>, METH_FASTCALL, nullptr},
    {"decode_static", (PyCFunction)(void (*)(void))guarded<decode<Decode::STATIC>>, METH_FASTCALL, nullptr},
    {"params", (PyCFunction)(void (*)(void))guarded<params>, METH_FASTCALL, nullptr},
    {"set_classes", (PyCFunction)(void (*)(void))set_classes, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_eta_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__eta_torch(void) { return PyModule_Create(&module); }
