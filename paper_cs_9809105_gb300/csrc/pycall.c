/* pycall.c -- the Python binding's per-step calls (hsmm_gemm, hsmm_gemv) as a CPython module.
 *
 * ctypes converts every argument of a call through Python objects and the binding built a
 * configuration and scalar objects besides: on the Grace host a gemv cost 8.5 us before its
 * kernels were launched, a product 6.7, more than the small ones take on the GPU.  Here the
 * arguments arrive as plain integers and numbers (vector call), the configuration and the scalars
 * live on the C stack.  The library's functions are bound by address (bind), so nothing is linked.
 * As with ctypes, the GIL is released during the call.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "hsmm.h"

typedef hsmm_status_t (*gemm_fn)(const hsmm_config_t*, hsmm_op_t, hsmm_op_t, int64_t, int64_t, int64_t, const void*,
                                 const void*, int64_t, const void*, int64_t, const void*, void*, int64_t, void*);
typedef hsmm_status_t (*gemv_fn)(const hsmm_config_t*, hsmm_op_t, int64_t, int64_t, const void*, const void*, int64_t,
                                 const void*, int64_t, const void*, void*, int64_t, void*);
static gemm_fn g_gemm;
static gemv_fn g_gemv;

typedef union {
    double d[2];
    float f;
    int32_t i;
} scalar_t;

/* one number as the scalar of a compute type; 0 on success */
static int to_scalar(PyObject* v, int code, scalar_t* out) {
    if (code == HSMM_C_64F) {
        const Py_complex z = PyComplex_AsCComplex(v);
        out->d[0] = z.real;
        out->d[1] = z.imag;
    } else if (code == HSMM_R_32I) {
        PyObject* n = PyNumber_Long(v);
        if (!n) return -1;
        out->i = (int32_t)(uint32_t)PyLong_AsUnsignedLongLongMask(n);
        Py_DECREF(n);
    } else {
        const double x = PyFloat_AsDouble(v);
        if (code == HSMM_R_64F) out->d[0] = x;
        else out->f = (float)x;
    }
    return PyErr_Occurred() ? -1 : 0;
}

/* n integers (sizes, codes, addresses up to 2^64 - 1) */
static int to_ints(PyObject* const* args, int n, int64_t* out) {
    for (int i = 0; i < n; ++i) {
        out[i] = PyLong_AsLongLong(args[i]);
        if (out[i] == -1 && PyErr_Occurred()) {
            if (!PyErr_ExceptionMatches(PyExc_OverflowError)) return -1;
            PyErr_Clear();
            out[i] = (int64_t)PyLong_AsUnsignedLongLong(args[i]);
            if (PyErr_Occurred()) return -1;
        }
    }
    return 0;
}

static void* ptr(int64_t v) { return (void*)(uintptr_t)v; }

/* gemm(a, b, c, compute, slices, bits, workspace, workspace_bytes, tile_n, ring_p, ring_k,
 *      scalar code, transA, transB, m, n, k, A, lda, B, ldb, C, ldc, stream, alpha, beta) */
static PyObject* call_gemm(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
    int64_t v[24];
    scalar_t alpha, beta;
    hsmm_config_t c;
    hsmm_status_t st;
    (void)self;
    if (nargs != 26 || !g_gemm) {
        PyErr_SetString(PyExc_TypeError, "gemm: 26 arguments and a bound library");
        return NULL;
    }
    if (to_ints(args, 24, v) || to_scalar(args[24], (int)v[11], &alpha) || to_scalar(args[25], (int)v[11], &beta))
        return NULL;
    memset(&c, 0, sizeof(c));
    c.a = (hsmm_dtype_t)v[0];
    c.b = (hsmm_dtype_t)v[1];
    c.c = (hsmm_dtype_t)v[2];
    c.compute = (hsmm_compute_t)v[3];
    c.ozaki_slices = (int)v[4];
    c.ozaki_bits = (int)v[5];
    c.workspace = ptr(v[6]);
    c.workspace_bytes = (size_t)v[7];
    c.tile_n = (int)v[8];
    c.ring_p = (int)v[9];
    c.ring_k = (int)v[10];
    Py_BEGIN_ALLOW_THREADS
    st = g_gemm(&c, (hsmm_op_t)v[12], (hsmm_op_t)v[13], v[14], v[15], v[16], &alpha, ptr(v[17]), v[18], ptr(v[19]),
                v[20], &beta, ptr(v[21]), v[22], ptr(v[23]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

/* gemv(a, c, workspace, workspace_bytes, trans, m, n, A, lda, x, incx, y, incy, stream, alpha, beta) */
static PyObject* call_gemv(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
    int64_t v[14];
    scalar_t alpha, beta;
    hsmm_config_t c;
    hsmm_status_t st;
    (void)self;
    if (nargs != 16 || !g_gemv) {
        PyErr_SetString(PyExc_TypeError, "gemv: 16 arguments and a bound library");
        return NULL;
    }
    if (to_ints(args, 14, v) || to_scalar(args[14], (int)v[1], &alpha) || to_scalar(args[15], (int)v[1], &beta))
        return NULL;
    memset(&c, 0, sizeof(c));
    c.a = c.b = (hsmm_dtype_t)v[0];
    c.c = (hsmm_dtype_t)v[1];
    c.workspace = ptr(v[2]);
    c.workspace_bytes = (size_t)v[3];
    Py_BEGIN_ALLOW_THREADS
    st = g_gemv(&c, (hsmm_op_t)v[4], v[5], v[6], &alpha, ptr(v[7]), v[8], ptr(v[9]), v[10], &beta, ptr(v[11]), v[12],
                ptr(v[13]));
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
}

/* bind(address of hsmm_gemm, address of hsmm_gemv) */
static PyObject* call_bind(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
    int64_t v[2];
    (void)self;
    if (nargs != 2) {
        PyErr_SetString(PyExc_TypeError, "bind: two addresses");
        return NULL;
    }
    if (to_ints(args, 2, v)) return NULL;
    g_gemm = (gemm_fn)(uintptr_t)v[0];
    g_gemv = (gemv_fn)(uintptr_t)v[1];
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"gemm", (PyCFunction)(void (*)(void))call_gemm, METH_FASTCALL, "hsmm_gemm"},
                                {"gemv", (PyCFunction)(void (*)(void))call_gemv, METH_FASTCALL, "hsmm_gemv"},
                                {"bind", (PyCFunction)(void (*)(void))call_bind, METH_FASTCALL, "bind the library"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_hsmmcall", "per-step calls of libhsmm", -1, methods,
                                    NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__hsmmcall(void) { return PyModule_Create(&module); }
