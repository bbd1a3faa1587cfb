/* CPython entry points of the two calls that sit inside a program's inner loop (sd_spmm and
 * sd_plan_update_values): argument marshalling only, like binding.py, which hands over the C addresses.
 *
 * What bounds a small product is the host: through ctypes and Python-level attribute look-ups one call cost
 * about 6 us on top of the launch itself (2,048 rows, 32 columns: 9.1 us per call, 4.0 us of kernel).  Here the
 * tensor's address and leading dimension are two vectorcalls each and the stream one more. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*spmm_fn)(const void *, const void *, int64_t, float *, int64_t, float, float, void *);
typedef int (*update_fn)(void *, const void *, void *);

static spmm_fn c_spmm;
static update_fn c_update;
static PyObject *current_device, *raw_stream;   /* torch's, set by bind() */
static PyObject *s_data_ptr, *s_stride, *s_cuda_stream, *s_ctypes, *s_data, *zero;

/* Address of None / int / torch tensor / numpy array.  0 with an exception set on failure. */
static int address(PyObject *o, void **out) {
    PyObject *v;
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return !(*out == NULL && PyErr_Occurred());
    }
    v = PyObject_VectorcallMethod(s_data_ptr, &o, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, NULL);
    if (!v) {   /* numpy */
        PyObject *c;
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return 0;
        PyErr_Clear();
        c = PyObject_GetAttr(o, s_ctypes);
        if (!c) return 0;
        v = PyObject_GetAttr(c, s_data);
        Py_DECREF(c);
        if (!v) return 0;
    }
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*out == NULL && PyErr_Occurred());
}

/* Row pitch in elements of a tensor. */
static int pitch(PyObject *o, int64_t *out) {
    PyObject *args[2] = {o, zero}, *v = PyObject_VectorcallMethod(s_stride, args, 2 | PY_VECTORCALL_ARGUMENTS_OFFSET, NULL);
    if (!v) return 0;
    *out = PyLong_AsLongLong(v);
    Py_DECREF(v);
    return !(*out == -1 && PyErr_Occurred());
}

static int stream_of(PyObject *o, void **out) {
    PyObject *v;
    if (o == Py_None) {   /* the current stream of the current device */
        PyObject *d = PyObject_CallNoArgs(current_device);
        if (!d) return 0;
        v = PyObject_CallOneArg(raw_stream, d);
        Py_DECREF(d);
    } else if (PyLong_Check(o)) {
        v = Py_NewRef(o);
    } else {
        v = PyObject_GetAttr(o, s_cuda_stream);
    }
    if (!v) return 0;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*out == NULL && PyErr_Occurred());
}

static int scalar(PyObject *o, float *out) {
    const double d = PyFloat_AsDouble(o);
    if (d == -1.0 && PyErr_Occurred()) return 0;
    *out = (float)d;
    return 1;
}

static int arity(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return 1;
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
    return 0;
}

static PyObject *call_spmm(void *plan, void *B, int64_t ldb, void *C, int64_t ldc, float alpha, float beta, void *st) {
    int rc;
    if (!c_spmm) {
        PyErr_SetString(PyExc_RuntimeError, "bind() has not been called");
        return NULL;
    }
    Py_BEGIN_ALLOW_THREADS
    rc = c_spmm(plan, B, ldb, (float *)C, ldc, alpha, beta, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* spmm(plan, B, ldb, C, ldc, alpha, beta, stream) -> status */
static PyObject *py_spmm(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *plan, *B, *C, *st;
    float alpha, beta;
    int64_t ldb, ldc;
    if (!arity(n, 8) || !address(a[0], &plan) || !address(a[1], &B) || !address(a[3], &C) || !scalar(a[5], &alpha) ||
        !scalar(a[6], &beta) || !stream_of(a[7], &st))
        return NULL;
    ldb = PyLong_AsLongLong(a[2]);
    ldc = PyLong_AsLongLong(a[4]);
    if (PyErr_Occurred()) return NULL;
    return call_spmm(plan, B, ldb, C, ldc, alpha, beta, st);
}

/* spmm_tensors(plan, B, C, alpha, beta, stream) -> status; the row pitches are the tensors' */
static PyObject *py_spmm_tensors(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *plan, *B, *C, *st;
    float alpha, beta;
    int64_t ldb, ldc;
    if (!arity(n, 6) || !address(a[0], &plan) || !address(a[1], &B) || !pitch(a[1], &ldb) || !address(a[2], &C) ||
        !pitch(a[2], &ldc) || !scalar(a[3], &alpha) || !scalar(a[4], &beta) || !stream_of(a[5], &st))
        return NULL;
    return call_spmm(plan, B, ldb, C, ldc, alpha, beta, st);
}

/* update_values(plan, vals, stream) -> status */
static PyObject *py_update_values(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *plan, *vals, *st;
    int rc;
    if (!arity(n, 3) || !address(a[0], &plan) || !address(a[1], &vals) || !stream_of(a[2], &st)) return NULL;
    if (!c_update) {
        PyErr_SetString(PyExc_RuntimeError, "bind() has not been called");
        return NULL;
    }
    Py_BEGIN_ALLOW_THREADS
    rc = c_update(plan, vals, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* bind(address of sd_spmm, address of sd_plan_update_values, device(), raw_stream(device)) */
static PyObject *py_bind(PyObject *self, PyObject *const *a, Py_ssize_t n) {
    void *f, *g;
    if (!arity(n, 4) || !address(a[0], &f) || !address(a[1], &g)) return NULL;
    c_spmm = (spmm_fn)(uintptr_t)f;
    c_update = (update_fn)(uintptr_t)g;
    Py_XSETREF(current_device, Py_NewRef(a[2]));
    Py_XSETREF(raw_stream, Py_NewRef(a[3]));
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, NULL},
                                {"spmm", (PyCFunction)(void (*)(void))py_spmm, METH_FASTCALL, NULL},
                                {"spmm_tensors", (PyCFunction)(void (*)(void))py_spmm_tensors, METH_FASTCALL, NULL},
                                {"update_values", (PyCFunction)(void (*)(void))py_update_values, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_stride = PyUnicode_InternFromString("stride");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_ctypes = PyUnicode_InternFromString("ctypes");
    s_data = PyUnicode_InternFromString("data");
    zero = PyLong_FromLong(0);
    if (!s_data_ptr || !s_stride || !s_cuda_stream || !s_ctypes || !s_data || !zero) return NULL;
    return PyModule_Create(&module);
}
