// Argument marshalling of the Python binding in native code: tensors to pointers, the current stream, one call into
// libxfp.so.  A 4096 x 4096 GEMV takes 4 us on the device; ctypes took 9 us of host time to queue it (nine arguments
// converted one by one, three attribute look-ups per tensor, a Python-level stream object), which bounded every decode
// step that was not captured in a graph.
//
// Every function returns the library's status code.  The library's entry points arrive as addresses (bind), so that the
// module serves whichever build of libxfp.so the binding has loaded.
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/xfp.h"

namespace {

struct Entry {
    decltype(&xfp_pack) pack;
    decltype(&xfp_gemv_v2) gemv_v2;
    decltype(&xfp_gemv_v2a) gemv_v2a;
    decltype(&xfp_gemv_typed) gemv_typed;
    decltype(&xfp_gemv_grouped_typed) grouped_typed;
    decltype(&xfp_gemv_host) gemv_host;
    decltype(&xfp_gemv_v2_noalloc) noalloc;
    decltype(&xfp_gemm_typed) gemm_typed;
    decltype(&xfp_dequant) dequant;
    decltype(&xfp_pack) pack_counted;
} g;

// One call's arguments; the first problem sets a Python exception and `bad`.
struct Args {
    PyObject* const* a;
    bool bad = false;
    Args(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : a(args) {
        if (n != want) { PyErr_Format(PyExc_TypeError, "%zd arguments, %zd expected", n, want); bad = true; }
        else if (!g.gemv_v2) { PyErr_SetString(PyExc_RuntimeError, "libxfp.so is not bound"); bad = true; }
    }
    const at::Tensor* tensor(int i) {
        if (bad || a[i] == Py_None) return nullptr;
        if (!THPVariable_Check(a[i])) {
            PyErr_Format(PyExc_TypeError, "a tensor is expected, not %s", Py_TYPE(a[i])->tp_name);
            bad = true;
            return nullptr;
        }
        return &THPVariable_Unpack(a[i]);
    }
    // what f throws (a sparse or a fake tensor has no data pointer, a symbolic size no value) as a Python exception: through a C
    // function it would end the process
    template <class F>
    auto guarded(F&& f) -> decltype(f()) {
        try { return f(); }
        catch (const c10::Error& e) { PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace()); }
        catch (const std::exception& e) { PyErr_SetString(PyExc_RuntimeError, e.what()); }
        bad = true;
        return {};
    }
    // the integer that method `name` of argument i returns: objects that are no tensors but have a tensor's methods (a storage, a
    // caller's own handle) are taken as the tensors are
    size_t method(int i, const char* name) {
        if (bad) return 0;
        PyObject* r = PyObject_CallMethod(a[i], name, nullptr);
        const size_t v = r ? PyLong_AsSize_t(r) : 0;
        Py_XDECREF(r);
        if (PyErr_Occurred()) bad = true;
        return v;
    }
    bool duck(int i) const { return !bad && a[i] != Py_None && !THPVariable_Check(a[i]); }
    void* ptr(int i) {
        if (duck(i)) return (void*)method(i, "data_ptr");
        const at::Tensor* t = tensor(i);
        return t ? guarded([&] { return t->data_ptr(); }) : nullptr;
    }
    void* buffer(int i, size_t* bytes) {
        if (duck(i)) {
            *bytes = method(i, "numel");
            *bytes *= method(i, "element_size");
        } else {
            const at::Tensor* t = tensor(i);
            *bytes = t ? guarded([&] { return t->nbytes(); }) : 0;
        }
        return ptr(i);
    }
    // as int() takes it: whole numbers of any kind, floats cut
    int32_t integer(int i) {
        if (bad) return 0;
        long v = -1;
        if (PyLong_Check(a[i])) v = PyLong_AsLong(a[i]);
        else if (PyObject* n = PyNumber_Long(a[i])) { v = PyLong_AsLong(n); Py_DECREF(n); }
        if (v == -1 && PyErr_Occurred()) bad = true;
        return (int32_t)v;
    }
    int32_t truth(int i) {
        if (bad) return 0;
        const int v = PyObject_IsTrue(a[i]);
        if (v < 0) bad = true;
        return v;
    }
    // the ctypes structure's own memory
    xfp_desc desc(int i) {
        xfp_desc d{};
        Py_buffer b;
        if (bad) return d;
        if (PyObject_GetBuffer(a[i], &b, PyBUF_SIMPLE)) { bad = true; return d; }
        if (b.len != (Py_ssize_t)sizeof d) { PyErr_SetString(PyExc_TypeError, "an XfpDesc is expected"); bad = true; }
        else memcpy(&d, b.buf, sizeof d);
        PyBuffer_Release(&b);
        return d;
    }
    // None: the current stream of the current device; else a torch stream or the address of one
    void* stream(int i) {
        if (bad) return nullptr;
        if (a[i] == Py_None) return guarded([] { return (void*)c10::cuda::getCurrentCUDAStream().stream(); });
        PyObject* v = PyObject_GetAttrString(a[i], "cuda_stream");
        if (!v) { PyErr_Clear(); v = Py_NewRef(a[i]); }
        PyObject* n = PyNumber_Long(v);
        Py_DECREF(v);
        if (!n) { bad = true; return nullptr; }
        void* p = PyLong_AsVoidPtr(n);
        Py_DECREF(n);
        if (!p && PyErr_Occurred()) bad = true;
        return p;
    }
    // XFP_T_* of a tensor's type (a KeyError for the others, as a look-up in a table gives)
    int32_t type(int i) {
        const at::Tensor* t = tensor(i);
        if (!t) { if (!bad) { PyErr_SetString(PyExc_TypeError, "a tensor is expected, not None"); bad = true; } return 0; }
        switch (t->scalar_type()) {
            case at::kFloat: return XFP_T_F32;
            case at::kHalf: return XFP_T_F16;
            case at::kBFloat16: return XFP_T_BF16;
            default: PyErr_SetString(PyExc_KeyError, toString(t->scalar_type())); bad = true; return 0;
        }
    }
};

template <class F>
PyObject* call(const Args& x, F&& f) {
    if (x.bad) return nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

// (mode, desc, packed, x, batch, y, y_is_fp16, workspace, stream); mode -1: the descriptor's; batch None: the rows of x (every
// integer goes to the library as it is, which refuses those that are no batch)
PyObject* gemv(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 9);
    int32_t mode = a.integer(0);
    const xfp_desc d = a.desc(1);
    const void* packed = a.ptr(2);
    const bool rows = !a.bad && args[4] == Py_None;
    const at::Tensor* x = rows ? a.tensor(3) : nullptr;
    const int32_t batch = !rows ? a.integer(4) : x ? a.guarded([&] { return x->dim() == 2 ? (int32_t)x->size(0) : 1; }) : 0;
    void* y = a.ptr(5);
    const int32_t half = a.truth(6);
    size_t bytes;
    void* ws = a.buffer(7, &bytes);
    void* s = a.stream(8);
    if (mode < 0) mode = d.mode;
    const uint16_t* xp = (const uint16_t*)a.ptr(3);
    return call(a, [&] { return (mode ? g.gemv_v2a : g.gemv_v2)(&d, packed, xp, batch, y, half, ws, bytes, s); });
}

// (desc, packed, x, batch, y, workspace, stream)
PyObject* gemv_typed(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 7);
    const xfp_desc d = a.desc(0);
    const void* packed = a.ptr(1);
    const void* x = a.ptr(2);
    const int32_t xt = a.type(2), batch = a.integer(3);
    void* y = a.ptr(4);
    const int32_t yt = a.type(4);
    size_t bytes;
    void* ws = a.buffer(5, &bytes);
    void* s = a.stream(6);
    return call(a, [&] { return g.gemv_typed(&d, packed, x, xt, batch, y, yt, ws, bytes, s); });
}

// (desc, n, packed, x, x_type, y, y_type, epilogue, weights, workspace, stream)
PyObject* grouped(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 11);
    const xfp_desc d = a.desc(0);
    const int32_t blobs = a.integer(1);
    const auto packed = (const void* const*)a.ptr(2);
    const auto x = (const void* const*)a.ptr(3);
    const int32_t xt = a.integer(4);
    const auto y = (void* const*)a.ptr(5);
    const int32_t yt = a.integer(6), epi = a.integer(7);
    const float* w = (const float*)a.ptr(8);
    size_t bytes;
    void* ws = a.buffer(9, &bytes);
    void* s = a.stream(10);
    return call(a, [&] { return g.grouped_typed(&d, blobs, packed, x, xt, y, yt, epi, w, ws, bytes, s); });
}

// (desc, packed, x, y, workspace, stream): the rows of x are its first dimension
PyObject* gemm(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 6);
    const xfp_desc d = a.desc(0);
    const void* packed = a.ptr(1);
    const at::Tensor* x = a.tensor(2);
    const int32_t xt = a.type(2);
    void* y = a.ptr(3);
    const int32_t yt = a.type(3);
    size_t bytes;
    void* ws = a.buffer(4, &bytes);
    void* s = a.stream(5);
    const int32_t m = x ? a.guarded([&] { return x->dim() ? (int32_t)x->size(0) : 0; }) : 0;
    const void* xp = a.ptr(2);
    return call(a, [&] { return g.gemm_typed(&d, packed, xp, xt, m, y, yt, ws, bytes, s); });
}

// (desc, packed, x_host, x_dev, batch, y_host, y_dev, y_is_fp16, workspace, stream)
PyObject* gemv_host(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 10);
    const xfp_desc d = a.desc(0);
    const void* packed = a.ptr(1);
    const uint16_t* xh = (const uint16_t*)a.ptr(2);
    uint16_t* xd = (uint16_t*)a.ptr(3);
    const int32_t batch = a.integer(4);
    void *yh = a.ptr(5), *yd = a.ptr(6);
    const int32_t half = a.truth(7);
    size_t bytes;
    void* ws = a.buffer(8, &bytes);
    void* s = a.stream(9);
    return call(a, [&] { return g.gemv_host(&d, packed, xh, xd, batch, yh, yd, half, ws, bytes, s); });
}

// (desc, packed, x, batch, y, y_is_fp16, stream)
PyObject* noalloc(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 7);
    const xfp_desc d = a.desc(0);
    const void* packed = a.ptr(1);
    const uint16_t* x = (const uint16_t*)a.ptr(2);
    const int32_t batch = a.integer(3);
    void* y = a.ptr(4);
    const int32_t half = a.truth(5);
    void* s = a.stream(6);
    return call(a, [&] { return g.noalloc(&d, packed, x, batch, y, half, s); });
}

// (desc, packed, W, stream)
PyObject* dequant(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 4);
    const xfp_desc d = a.desc(0);
    const void* packed = a.ptr(1);
    uint16_t* W = (uint16_t*)a.ptr(2);
    void* s = a.stream(3);
    return call(a, [&] { return g.dequant(&d, packed, W, s); });
}

// (desc, idx, codebook, gid, gscale, gmid, rowptr, ocol, oval, packed, err_word, stream)
PyObject* pack_by(decltype(&xfp_pack) f, PyObject* const* args, Py_ssize_t n) {
    Args a(args, n, 12);
    const xfp_desc d = a.desc(0);
    void* p[8];
    for (int i = 0; i < 8; ++i) p[i] = a.ptr(1 + i);
    size_t bytes;
    void* packed = a.buffer(9, &bytes);
    int32_t* err = (int32_t*)a.ptr(10);
    void* s = a.stream(11);
    return call(a, [&] {
        return f(&d, (const uint8_t*)p[0], (const uint16_t*)p[1], (const uint8_t*)p[2], (const uint16_t*)p[3],
                 (const uint16_t*)p[4], (const int32_t*)p[5], p[6], (const uint16_t*)p[7], packed, bytes, err, s);
    });
}
PyObject* pack(PyObject*, PyObject* const* args, Py_ssize_t n) { return pack_by(g.pack, args, n); }
PyObject* pack_counted(PyObject*, PyObject* const* args, Py_ssize_t n) { return pack_by(g.pack_counted, args, n); }

// bind(addresses of xfp_pack, xfp_gemv_v2, xfp_gemv_v2a, xfp_gemv_typed, xfp_gemv_grouped_typed, xfp_gemv_host,
//      xfp_gemv_v2_noalloc, xfp_gemm_typed, xfp_dequant, xfp_pack_counted)
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t n) {
    void** slot = (void**)&g;
    constexpr Py_ssize_t kSlots = sizeof g / sizeof(void*);
    if (n != kSlots) { PyErr_Format(PyExc_TypeError, "bind takes %zd addresses", kSlots); return nullptr; }
    for (Py_ssize_t i = 0; i < n; ++i) {
        slot[i] = PyLong_AsVoidPtr(args[i]);
        if (!slot[i]) { if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "a null entry point"); return nullptr; }
    }
    Py_RETURN_NONE;
}

#define XFP_METHOD(f) {#f, (PyCFunction)(void*)f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {XFP_METHOD(bind), XFP_METHOD(gemv), XFP_METHOD(gemv_typed), XFP_METHOD(grouped), XFP_METHOD(gemm),
                         XFP_METHOD(gemv_host), XFP_METHOD(noalloc), XFP_METHOD(dequant), XFP_METHOD(pack),
                         XFP_METHOD(pack_counted),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_xfp_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__xfp_native() { return PyModule_Create(&module); }
