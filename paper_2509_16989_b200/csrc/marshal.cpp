// The calls of binding.py that a decode loop makes, for plain arguments: tensors of the expected kind go to the C functions of libptqtp.so
// without a detour through Python attributes and ctypes.  A call took the host 5.1 to 5.7 us, 2.4 to 3.1 of them the launch itself; 2.6 to
// 3.6 like this (3072 x 1024, format 3, call after call: 5.4 -> 2.9 us, where the device takes 2.3).  Whatever is not plain -- subclasses,
// wrapped or traced tensors, active function or dispatch modes, other types and layouts -- is left to binding.py: the functions here
// return None and have done nothing.
#include <Python.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>
#include "ptqtp.h"

namespace {

using Gemv = decltype(&ptqtp_gemv);
using GemvHost = decltype(&ptqtp_gemv_host);
using Skinny = decltype(&ptqtp_gemm_skinny);
using SkinnyWs = decltype(&ptqtp_gemm_skinny_ws);
struct Functions {
    Gemv gemv;
    GemvHost gemv_host;
    Skinny skinny;
    SkinnyWs skinny_ws;
} g_fn = {};
bool g_bound = false;              // until bind() the functions leave every call to binding.py

const c10::DispatchKeySet kWrapped({c10::DispatchKey::FuncTorchBatched, c10::DispatchKey::FuncTorchVmapMode, c10::DispatchKey::FuncTorchGradWrapper,
                                    c10::DispatchKey::Functionalize, c10::DispatchKey::Python, c10::DispatchKey::Batched});

// A tensor that binding.py would take as it is: contiguous, of this type, on a device (or, host, in host memory).
const at::Tensor* plain(PyObject* o, at::ScalarType type, bool host = false) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || t.scalar_type() != type || !t.has_storage() || t.key_set().has_any(kWrapped)) return nullptr;
    if (host ? !t.device().is_cpu() : !t.is_cuda()) return nullptr;
    return t.layout() == at::kStrided && t.is_contiguous() ? &t : nullptr;
}
// N, K, format
bool plain_shape(PyObject* const* a, ptqtp_shape& s) {
    long v[3];
    for (int i = 0; i < 3; ++i) {
        if (!PyLong_CheckExact(a[i])) return false;
        int overflow = 0;
        v[i] = PyLong_AsLongAndOverflow(a[i], &overflow);
        if (overflow || v[i] < 0 || v[i] > 0x7fffffffL) return false;
    }
    s = {(int32_t)v[0], (int32_t)v[1], 128, (int32_t)v[2]};
    return true;
}
bool modes() { return at::impl::torch_function_mode_enabled() || c10::impl::TorchDispatchModeTLS::any_modes_set(); }

#define PTQTP_NOT_PLAIN() Py_RETURN_NONE
// The call itself, on the current stream, without the interpreter's lock (a full launch queue blocks).
#define PTQTP_CALL(expr)                                               \
    void* const stream = c10::cuda::getCurrentCUDAStream().stream();   \
    ptqtp_status st;                                                   \
    Py_BEGIN_ALLOW_THREADS st = (expr);                                \
    Py_END_ALLOW_THREADS return PyLong_FromLong((long)st)

// (packed, x, y, N, K, format)
PyObject* gemv(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ptqtp_shape s;
    if (n != 6 || !g_bound || modes() || !plain_shape(a + 3, s)) PTQTP_NOT_PLAIN();
    const at::Tensor *p = plain(a[0], at::kByte), *x = plain(a[1], at::kHalf), *y = plain(a[2], at::kHalf);
    if (!p || !x || !y) PTQTP_NOT_PLAIN();
    void *pp = p->data_ptr(), *xp = x->data_ptr(), *yp = y->data_ptr();
    const size_t bytes = (size_t)p->numel();
    PTQTP_CALL(g_fn.gemv(&s, pp, bytes, static_cast<uint16_t*>(xp), static_cast<uint16_t*>(yp), stream));
}
// (packed, x_host, y_host, x_dev, y_dev, N, K, format)
PyObject* gemv_host(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ptqtp_shape s;
    if (n != 8 || !g_bound || modes() || !plain_shape(a + 5, s)) PTQTP_NOT_PLAIN();
    const at::Tensor *p = plain(a[0], at::kByte), *xh = plain(a[1], at::kHalf, true), *yh = plain(a[2], at::kHalf, true), *xd = plain(a[3], at::kHalf),
                     *yd = plain(a[4], at::kHalf);
    if (!p || !xh || !yh || !xd || !yd) PTQTP_NOT_PLAIN();
    void *pp = p->data_ptr(), *xhp = xh->data_ptr(), *yhp = yh->data_ptr(), *xdp = xd->data_ptr(), *ydp = yd->data_ptr();
    const size_t bytes = (size_t)p->numel();
    PTQTP_CALL(g_fn.gemv_host(&s, pp, bytes, static_cast<uint16_t*>(xhp), static_cast<uint16_t*>(yhp), static_cast<uint16_t*>(xdp),
                              static_cast<uint16_t*>(ydp), stream));
}
// (packed, X, Y, N, K, format)
PyObject* gemm_skinny(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ptqtp_shape s;
    if (n != 6 || !g_bound || modes() || !plain_shape(a + 3, s)) PTQTP_NOT_PLAIN();
    const at::Tensor *p = plain(a[0], at::kByte), *x = plain(a[1], at::kHalf), *y = plain(a[2], at::kHalf);
    if (!p || !x || !y || x->dim() < 1 || x->size(0) > 0x7fffffffL) PTQTP_NOT_PLAIN();
    void *pp = p->data_ptr(), *xp = x->data_ptr(), *yp = y->data_ptr();
    const size_t bytes = (size_t)p->numel();
    const int32_t m = (int32_t)x->size(0);
    PTQTP_CALL(g_fn.skinny(&s, pp, bytes, m, static_cast<uint16_t*>(xp), static_cast<uint16_t*>(yp), stream));
}
// (packed, X, Y, workspace, N, K, format)
PyObject* gemm_skinny_ws(PyObject*, PyObject* const* a, Py_ssize_t n) {
    ptqtp_shape s;
    if (n != 7 || !g_bound || modes() || !plain_shape(a + 4, s)) PTQTP_NOT_PLAIN();
    const at::Tensor *p = plain(a[0], at::kByte), *x = plain(a[1], at::kHalf), *y = plain(a[2], at::kHalf), *w = plain(a[3], at::kByte);
    if (!p || !x || !y || !w || x->dim() < 1 || x->size(0) > 0x7fffffffL) PTQTP_NOT_PLAIN();
    void *pp = p->data_ptr(), *xp = x->data_ptr(), *yp = y->data_ptr(), *wp = w->data_ptr();
    const size_t bytes = (size_t)p->numel(), room = (size_t)w->numel();
    const int32_t m = (int32_t)x->size(0);
    PTQTP_CALL(g_fn.skinny_ws(&s, pp, bytes, m, static_cast<uint16_t*>(xp), static_cast<uint16_t*>(yp), wp, room, stream));
}
// The addresses of the C functions, in the order of Functions.
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void* f[4];
    if (n != 4) { PyErr_SetString(PyExc_TypeError, "four addresses"); return nullptr; }
    for (int i = 0; i < 4; ++i) {
        f[i] = PyLong_AsVoidPtr(a[i]);
        if (PyErr_Occurred()) return nullptr;
        if (!f[i]) { PyErr_SetString(PyExc_ValueError, "a null address"); return nullptr; }
    }
    g_fn = {reinterpret_cast<Gemv>(f[0]), reinterpret_cast<GemvHost>(f[1]), reinterpret_cast<Skinny>(f[2]), reinterpret_cast<SkinnyWs>(f[3])};
    g_bound = true;
    Py_RETURN_NONE;
}

// C++ exceptions (a tensor without data) end here: binding.py says what is wrong.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    try {
        return F(self, a, n);
    } catch (...) {
        Py_RETURN_NONE;
    }
}
#define PTQTP_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<name>)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {PTQTP_METHOD(gemv), PTQTP_METHOD(gemv_host), PTQTP_METHOD(gemm_skinny), PTQTP_METHOD(gemm_skinny_ws), PTQTP_METHOD(bind),
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__marshal() {
    PyObject* m = PyModule_Create(&g_module);
    if (m && PyModule_AddStringConstant(m, "torch_version", PTQTP_TORCH_VERSION) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
