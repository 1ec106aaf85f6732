// Python's way into the C ABI: takes tensors and configuration structs as the binding's functions get them and calls the library.
//
// The host side of a small step is its longest part (four calls of 4.6 to 6.2 us where a launch is about 2): marshalling thirty pointers
// through ctypes and Python attribute calls costs more than half as much again as the launches.  Here a pointer is read from the tensor
// object itself and the stream from PyTorch's current one.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <exception>

#include "../../include/vardrop.h"

namespace {

// The arguments of one call; the first problem leaves a Python exception set and `ok` false.
struct Args {
    PyObject* const* a;
    bool ok = true;
    Py_buffer cfg_view{};
    bool has_cfg = false;

    explicit Args(PyObject* const* args) : a(args) {}
    ~Args() { if (has_cfg) PyBuffer_Release(&cfg_view); }

    // device address of a tensor (or of anything with a data_ptr method); None: NULL
    template <typename T = void>
    T* ptr(int i) {
        PyObject* t = a[i];
        if (!ok || t == Py_None) return nullptr;
        if (THPVariable_Check(t)) return static_cast<T*>(THPVariable_Unpack(t).data_ptr());
        PyObject* v = PyObject_CallMethod(t, "data_ptr", nullptr);
        void* p = v ? PyLong_AsVoidPtr(v) : nullptr;
        Py_XDECREF(v);
        ok = !PyErr_Occurred();
        return static_cast<T*>(p);
    }
    // a ctypes struct through the buffer protocol
    template <typename T>
    const T* cfg(int i) {
        if (!ok) return nullptr;
        has_cfg = PyObject_GetBuffer(a[i], &cfg_view, PyBUF_SIMPLE) == 0;
        if (has_cfg && cfg_view.len < static_cast<Py_ssize_t>(sizeof(T))) PyErr_SetString(PyExc_TypeError, "configuration struct of another kind");
        ok = !PyErr_Occurred();
        return static_cast<const T*>(cfg_view.buf);
    }
    size_t bytes(int i) {
        if (!ok) return 0;
        if (THPVariable_Check(a[i])) return THPVariable_Unpack(a[i]).nbytes();
        PyObject* n = PyObject_CallMethod(a[i], "numel", nullptr);
        PyObject* e = n ? PyObject_CallMethod(a[i], "element_size", nullptr) : nullptr;
        const size_t r = e ? PyLong_AsSize_t(n) * PyLong_AsSize_t(e) : 0;
        Py_XDECREF(n);
        Py_XDECREF(e);
        ok = !PyErr_Occurred();
        return r;
    }
};

// Runs `call` with PyTorch's current stream and without the interpreter lock; returns its status.
template <typename F>
PyObject* finish(const Args& args, F call) {
    if (!args.ok) return nullptr;
    void* const stream = c10::cuda::getCurrentCUDAStream().stream();
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = call(stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}
template <int kCount, typename F>
PyObject* guarded(PyObject* const* a, Py_ssize_t n, F body) {
    if (n != kCount) return PyErr_Format(PyExc_TypeError, "%d arguments expected, %zd given", kCount, n);
    try {
        Args args(a);
        return body(args);
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

PyObject* hash(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<6>(a, n, [](Args& g) {
        const auto x = g.ptr<const float>(0);
        const auto cfg = g.cfg<vardrop_hash_cfg>(1);
        const auto keys = g.ptr<uint64_t>(2);
        const auto freqs = g.ptr<int32_t>(3);
        const auto amp = g.ptr<float>(4);
        const auto ws = g.ptr(5);
        const size_t nb = g.bytes(5);
        return finish(g, [=](void* s) { return vardrop_hash(x, cfg, keys, freqs, amp, ws, nb, s); });
    });
}
PyObject* select(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<10>(a, n, [](Args& g) {
        const auto keys = g.ptr<const uint64_t>(0);
        const auto cfg = g.cfg<vardrop_select_cfg>(1);
        int32_t* o[7];
        for (int i = 0; i < 7; ++i) o[i] = g.ptr<int32_t>(2 + i);
        const auto ws = g.ptr(9);
        const size_t nb = g.bytes(9);
        return finish(g, [=](void* s) { return vardrop_select(keys, cfg, o[0], o[1], o[2], o[3], o[4], o[5], o[6], ws, nb, s); });
    });
}
PyObject* select_static(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<9>(a, n, [](Args& g) {
        const auto keys = g.ptr<const uint64_t>(0);
        const auto cfg = g.cfg<vardrop_select_cfg>(1);
        int32_t* o[7];
        for (int i = 0; i < 7; ++i) o[i] = g.ptr<int32_t>(2 + i);
        return finish(g, [=](void* s) { return vardrop_select_static(keys, cfg, o[0], o[1], o[2], o[3], o[4], o[5], o[6], s); });
    });
}
PyObject* gather_rows(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<5>(a, n, [](Args& g) {
        const auto x = g.ptr<const float>(0);
        const auto sel = g.ptr<const int32_t>(1), n_sel = g.ptr<const int32_t>(2);
        const auto cfg = g.cfg<vardrop_gather_cfg>(3);
        const auto out = g.ptr<float>(4);
        return finish(g, [=](void* s) { return vardrop_gather_rows(x, sel, n_sel, cfg, out, s); });
    });
}
PyObject* attn_fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<9>(a, n, [](Args& g) {
        const void* const q = g.ptr(0);
        const void* const k = g.ptr(1);
        const void* const v = g.ptr(2);
        const auto sel = g.ptr<const int32_t>(3), n_sel = g.ptr<const int32_t>(4);
        const auto cfg = g.cfg<vardrop_attn_cfg>(5);
        const auto o = g.ptr(6);
        const auto lse = g.ptr<float>(7);
        const auto ws = g.ptr(8);
        const size_t nb = g.bytes(8);
        return finish(g, [=](void* s) { return vardrop_attn_fwd(q, k, v, sel, n_sel, cfg, o, lse, ws, nb, s); });
    });
}
PyObject* attn_bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<14>(a, n, [](Args& g) {
        const void* const q = g.ptr(0);
        const void* const k = g.ptr(1);
        const void* const v = g.ptr(2);
        const void* const o = g.ptr(3);
        const auto lse = g.ptr<const float>(4);
        const void* const d_o = g.ptr(5);
        const auto sel = g.ptr<const int32_t>(6), n_sel = g.ptr<const int32_t>(7), inv = g.ptr<const int32_t>(8);
        const auto cfg = g.cfg<vardrop_attn_cfg>(9);
        const auto dq = g.ptr(10), dk = g.ptr(11), dv = g.ptr(12), ws = g.ptr(13);
        const size_t nb = g.bytes(13);
        return finish(g, [=](void* s) { return vardrop_attn_bwd(q, k, v, o, lse, d_o, sel, n_sel, inv, cfg, dq, dk, dv, ws, nb, s); });
    });
}
PyObject* pearson_max(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded<5>(a, n, [](Args& g) {
        const auto x = g.ptr<const float>(0);
        const auto cfg = g.cfg<vardrop_pearson_cfg>(1);
        const auto rho = g.ptr<float>(2);
        const auto above = g.ptr<int32_t>(3);
        const auto ws = g.ptr(4);
        const size_t nb = g.bytes(4);
        return finish(g, [=](void* s) { return vardrop_pearson_max(x, cfg, rho, above, ws, nb, s); });
    });
}

#define VD_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {VD_METHOD(hash), VD_METHOD(select), VD_METHOD(select_static), VD_METHOD(gather_rows), VD_METHOD(attn_fwd), VD_METHOD(attn_bwd),
                           VD_METHOD(pearson_max), {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" PyObject* PyInit__marshal(void) { return PyModule_Create(&g_module); }
