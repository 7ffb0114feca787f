/* CPython entry to the launching functions of libbitcos.so: integers in, status out.
 *
 * A decode-sized product keeps the GPU busy for 2 to 8 us, so what the caller spends on the way into the library counts:
 * a ctypes call with nine converted arguments costs about 2 us more than the vectorcall below.  Pointers (device or
 * host), sizes and the stream are passed as Python integers, NULL as 0.  bind() takes the addresses of the library's
 * functions, so this module does not link against it.  The GIL is released around the library, as ctypes does. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>
#include <string.h>

static int take(PyObject *const *args, Py_ssize_t n, Py_ssize_t want, const char *name, int64_t *v) {
    if (n != want) {
        PyErr_Format(PyExc_TypeError, "%s takes %zd integers, got %zd", name, want, n);
        return -1;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        v[i] = PyLong_AsLongLong(args[i]);
        if (v[i] == -1 && PyErr_Occurred()) return -1;
    }
    return 0;
}

#define P(i) ((void *)(uintptr_t)v[i])
#define I(i) ((int)v[i])
#define Z(i) ((size_t)v[i])
#define L(i) (v[i])
#define TYPES(...) __VA_ARGS__
#define CALL(name, count, types, ...)                                                       \
    static int (*p_##name)(types);                                                          \
    static PyObject *name(PyObject *self, PyObject *const *args, Py_ssize_t n) {            \
        int64_t v[count];                                                                   \
        int status;                                                                         \
        (void)self;                                                                         \
        if (take(args, n, count, #name, v)) return NULL;                                    \
        if (!p_##name) {                                                                    \
            PyErr_SetString(PyExc_RuntimeError, #name " is not bound");                     \
            return NULL;                                                                    \
        }                                                                                   \
        Py_BEGIN_ALLOW_THREADS status = p_##name(__VA_ARGS__);                              \
        Py_END_ALLOW_THREADS return PyLong_FromLong(status);                                \
    }

/* (W, x, x_scale, batch, y, acc_debug, workspace, workspace_bytes, stream) */
#define GEMV_TYPES TYPES(void *, void *, void *, int, void *, void *, void *, size_t, void *)
CALL(bitcos_gemv, 9, GEMV_TYPES, P(0), P(1), P(2), I(3), P(4), P(5), P(6), Z(7), P(8))
CALL(bitcos_gemv_group_scales, 9, GEMV_TYPES, P(0), P(1), P(2), I(3), P(4), P(5), P(6), Z(7), P(8))
/* (W, x_bf16, batch, y, acc_debug, workspace, workspace_bytes, stream) */
CALL(bitcos_gemv_bf16, 8, TYPES(void *, void *, int, void *, void *, void *, size_t, void *), P(0), P(1), I(2), P(3), P(4),
     P(5), Z(6), P(7))
/* (W, x_bf16, batch, y, workspace, workspace_bytes, stream) */
CALL(bitcos_gemv_blend_bf16, 7, TYPES(void *, void *, int, void *, void *, size_t, void *), P(0), P(1), I(2), P(3), P(4), Z(5),
     P(6))
/* (words, scales, M, K, x, x_scale, batch, y, acc_debug, workspace, workspace_bytes, stream) */
#define PLAIN_TYPES TYPES(void *, void *, int64_t, int64_t, void *, void *, int, void *, void *, void *, size_t, void *)
CALL(trit5_gemv, 12, PLAIN_TYPES, P(0), P(1), L(2), L(3), P(4), P(5), I(6), P(7), P(8), P(9), Z(10), P(11))
CALL(bit2_gemv, 12, PLAIN_TYPES, P(0), P(1), L(2), L(3), P(4), P(5), I(6), P(7), P(8), P(9), Z(10), P(11))
/* (jobs, n_jobs, batch, stream) */
#define MULTI_TYPES TYPES(void *, int, int, void *)
CALL(bitcos_gemv_multi, 4, MULTI_TYPES, P(0), I(1), I(2), P(3))
CALL(bitcos_gemv_multi_bf16, 4, MULTI_TYPES, P(0), I(1), I(2), P(3))
CALL(bitcos_gemv_multi_group_scales, 4, MULTI_TYPES, P(0), I(1), I(2), P(3))
/* (jobs, n_jobs, batch, prev, n_prev, next, n_next, stream) */
CALL(bitcos_gemv_multi_chained, 8, TYPES(void *, int, int, void *, int, void *, int, void *), P(0), I(1), I(2), P(3), I(4), P(5),
     I(6), P(7))
/* (jobs, phases, n_jobs, batch, in_host, in_device, in_bytes, out_host, out_device, out_bytes, stream) */
CALL(bitcos_gemv_phases_host, 11, TYPES(void *, void *, int, int, void *, void *, size_t, void *, void *, size_t, void *), P(0),
     P(1), I(2), I(3), P(4), P(5), Z(6), P(7), P(8), Z(9), P(10))
/* (x_bf16, batch, K, group, xq, x_scale, stream) */
CALL(bitcos_quantize_activations, 7, TYPES(void *, int, int64_t, int, void *, void *, void *), P(0), I(1), L(2), I(3), P(4), P(5),
     P(6))
/* (pair_expert, pair_xrow, n_pairs, n_experts, group_expert, group_begin, pair_xrow_sorted, order, n_groups, stream) */
CALL(bitcos_group_pairs_device, 10, TYPES(void *, void *, int, int, void *, void *, void *, void *, void *, void *), P(0), P(1),
     I(2), I(3), P(4), P(5), P(6), P(7), P(8), P(9))
/* (experts, n_experts, M, K, group_expert, group_begin, n_groups, pair_xrow, n_pairs, max_group_size, x, n_xrows, x_scale, y,
   acc_debug, workspace, workspace_bytes, stream) */
#define GROUPED_TYPES                                                                                                             \
    TYPES(void *, int, int64_t, int64_t, void *, void *, int, void *, int, int, void *, int, void *, void *, void *, void *, size_t, \
          void *)
#define GROUPED_ARGS                                                                                                               \
    P(0), I(1), L(2), L(3), P(4), P(5), I(6), P(7), I(8), I(9), P(10), I(11), P(12), P(13), P(14), P(15), Z(16), P(17)
CALL(bitcos_gemv_grouped, 18, GROUPED_TYPES, GROUPED_ARGS)
CALL(trit5_gemv_grouped, 18, GROUPED_TYPES, GROUPED_ARGS)
CALL(bit2_gemv_grouped, 18, GROUPED_TYPES, GROUPED_ARGS)
/* the same with (n_groups_device, max_groups) in place of n_groups */
CALL(bitcos_gemv_grouped_lists, 19,
     TYPES(void *, int, int64_t, int64_t, void *, void *, void *, int, void *, int, int, void *, int, void *, void *, void *, void *,
           size_t, void *),
     P(0), I(1), L(2), L(3), P(4), P(5), P(6), I(7), P(8), I(9), I(10), P(11), I(12), P(13), P(14), P(15), P(16), Z(17), P(18))

#define EVERY(X)                                                                                                           \
    X(bitcos_gemv) X(bitcos_gemv_group_scales) X(bitcos_gemv_bf16) X(bitcos_gemv_blend_bf16) X(trit5_gemv) X(bit2_gemv)    \
    X(bitcos_gemv_multi) X(bitcos_gemv_multi_bf16) X(bitcos_gemv_multi_group_scales) X(bitcos_gemv_multi_chained)          \
    X(bitcos_gemv_phases_host) X(bitcos_quantize_activations) X(bitcos_group_pairs_device) X(bitcos_gemv_grouped)          \
    X(trit5_gemv_grouped) X(bit2_gemv_grouped) X(bitcos_gemv_grouped_lists)

/* bind(name, address): where the library's function is */
static PyObject *bind(PyObject *self, PyObject *args) {
    const char *name;
    unsigned long long address;
    (void)self;
    if (!PyArg_ParseTuple(args, "sK", &name, &address)) return NULL;
#define SET(f)                                                      \
    if (!strcmp(name, #f)) {                                        \
        void *p = (void *)(uintptr_t)address;                       \
        memcpy(&p_##f, &p, sizeof p);                               \
        Py_RETURN_NONE;                                             \
    }
    EVERY(SET)
    PyErr_Format(PyExc_KeyError, "%s", name);
    return NULL;
}

#define ENTRY(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL},
static PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, NULL}, EVERY(ENTRY){NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) { return PyModule_Create(&module); }
