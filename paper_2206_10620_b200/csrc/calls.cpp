// CPython extension with the enqueueing calls of the C ABI: argument marshalling only.  A layer of a
// small problem runs in a few microseconds, of which ctypes would take more than one.
#define PY_SSIZE_T_CLEAN
#define Py_LIMITED_API 0x030A0000
#include <Python.h>

#include "blockgemm.h"
#include "dwconv.h"

static decltype(&xgen_patconv_run) p_conv;
static decltype(&xgen_patconv_run_fused) p_fused;
static decltype(&xgen_blockgemm_run) p_gemm;
static decltype(&xgen_dwconv_run) p_dw;

// Addresses are ints; None is the null pointer.
static void *ptr(PyObject *o) { return o == Py_None ? nullptr : PyLong_AsVoidPtr(o); }
static int32_t i32(PyObject *o) { return (int32_t)PyLong_AsLong(o); }
static bool count(Py_ssize_t got, Py_ssize_t want) {
    if (got == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments, not %zd", want, got);
    return false;
}
static PyObject *status(xgen_status s) { return PyLong_FromLong((long)s); }

// bind(addresses of run, run_fused, blockgemm_run, dwconv_run)
static PyObject *bind(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (!count(n, 4)) return nullptr;
    p_conv = reinterpret_cast<decltype(p_conv)>(ptr(a[0]));
    p_fused = reinterpret_cast<decltype(p_fused)>(ptr(a[1]));
    p_gemm = reinterpret_cast<decltype(p_gemm)>(ptr(a[2]));
    p_dw = reinterpret_cast<decltype(p_dw)>(ptr(a[3]));
    if (PyErr_Occurred()) return nullptr;
    Py_RETURN_NONE;
}

// conv / dw(handle, x, n, h, w, bias, relu, y, stream)
template <bool DW> static PyObject *run(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (!count(n, 9)) return nullptr;
    void *const h = ptr(a[0]), *const x = ptr(a[1]), *const bias = ptr(a[5]), *const y = ptr(a[7]), *const st = ptr(a[8]);
    const int32_t in = i32(a[2]), ih = i32(a[3]), iw = i32(a[4]), relu = PyObject_IsTrue(a[6]);
    if (PyErr_Occurred()) return nullptr;
    xgen_status s;
    Py_BEGIN_ALLOW_THREADS
    if (DW) s = p_dw(static_cast<const xgen_dwconv_packed *>(h), x, in, ih, iw, bias, relu, y, st);
    else s = p_conv(static_cast<const xgen_patconv_packed *>(h), x, in, ih, iw, bias, relu, y, st);
    Py_END_ALLOW_THREADS
    return status(s);
}

// fused(handle, x, n, h, w, bias, y, stream, relu, pool, residual, scale, zero point)
static PyObject *fused(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (!count(n, 13)) return nullptr;
    void *const h = ptr(a[0]), *const x = ptr(a[1]), *const bias = ptr(a[5]), *const y = ptr(a[6]), *const st = ptr(a[7]);
    const int32_t in = i32(a[2]), ih = i32(a[3]), iw = i32(a[4]);
    xgen_patconv_epilogue ep;
    ep.relu = PyObject_IsTrue(a[8]);
    ep.pool = i32(a[9]);
    ep.residual_dev = ptr(a[10]);
    ep.requant_scale_dev = static_cast<const float *>(ptr(a[11]));
    ep.requant_zero_point = i32(a[12]);
    if (PyErr_Occurred()) return nullptr;
    xgen_status s;
    Py_BEGIN_ALLOW_THREADS
    s = p_fused(static_cast<const xgen_patconv_packed *>(h), x, in, ih, iw, bias, &ep, y, st);
    Py_END_ALLOW_THREADS
    return status(s);
}

// gemm(handle, x, rows, bias, relu, y, stream)
static PyObject *gemm(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (!count(n, 7)) return nullptr;
    void *const h = ptr(a[0]), *const x = ptr(a[1]), *const bias = ptr(a[3]), *const y = ptr(a[5]), *const st = ptr(a[6]);
    const int64_t m = PyLong_AsLongLong(a[2]);
    const int32_t relu = PyObject_IsTrue(a[4]);
    if (PyErr_Occurred()) return nullptr;
    xgen_status s;
    Py_BEGIN_ALLOW_THREADS
    s = p_gemm(static_cast<const xgen_blockgemm_packed *>(h), x, m, bias, relu, y, st);
    Py_END_ALLOW_THREADS
    return status(s);
}

template <typename F> static PyCFunction fast(F f) { return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)); }
static PyMethodDef methods[] = {
    {"bind", fast(bind), METH_FASTCALL, nullptr},   {"conv", fast(run<false>), METH_FASTCALL, nullptr},
    {"fused", fast(fused), METH_FASTCALL, nullptr}, {"gemm", fast(gemm), METH_FASTCALL, nullptr},
    {"dw", fast(run<true>), METH_FASTCALL, nullptr}, {nullptr, nullptr, 0, nullptr}};
// What the extension was made from: build.py looks for it in the file.
extern "C" __attribute__((used, visibility("default"))) const char xgen_calls_tag[] = XGEN_CALLS_TAG;
static PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&module); }
