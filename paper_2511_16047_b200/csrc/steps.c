/* Python side of the calls of a generation step (amskv_append, amskv_attend, amskv_append_attend): takes addresses and strides
 * out of the tensors and calls the library, without the argument conversions of ctypes.  Marshalling only.
 *
 * These calls are made layers x scales times per image; through ctypes their Python side took 2.1 us with contiguous tensors
 * and 3.3 us with views, about what the launch itself takes; here 0.8 and 1.4.
 *
 * A tensor argument is anything with data_ptr(), is_contiguous() and stride() (a torch tensor), an address (int), or None.
 * The library's functions are handed over by bind() as addresses, so this module is independent of where it was loaded from.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*append_fn)(void*, int, int, const void*, const void*, const int64_t*, void*);
typedef int (*attend_fn)(void*, int, int, const void*, void*, const int64_t*, const int64_t*, void*);
typedef int (*append_attend_fn)(void*, int, int, const void*, const void*, const int64_t*, const void*, void*, const int64_t*,
                                const int64_t*, void*);
static append_fn f_append;
static attend_fn f_attend;
static append_attend_fn f_append_attend;
static PyObject *s_data_ptr, *s_is_contiguous, *s_stride, *s_cuda_stream;

static int as_pointer(PyObject* o, void** out) /* an int (or what __index__ makes one), or None */
{
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    PyObject* i = PyNumber_Long(o);
    if (!i) return -1;
    *out = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return PyErr_Occurred() ? -1 : 0;
}

/* address of a tensor argument; strides[3] and *strided = 1 when it is a view that is not contiguous */
static int tensor(PyObject* x, void** addr, int64_t* strides, int* strided)
{
    *strided = 0;
    if (x == Py_None || PyLong_CheckExact(x)) return as_pointer(x, addr);
    PyObject* r = PyObject_CallMethodNoArgs(x, s_data_ptr);
    if (!r) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
        PyErr_Clear();
        return as_pointer(x, addr);
    }
    int bad = as_pointer(r, addr);
    Py_DECREF(r);
    if (bad) return -1;
    r = PyObject_CallMethodNoArgs(x, s_is_contiguous);
    if (!r) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
        PyErr_Clear();   /* something with an address only */
        return 0;
    }
    const int contiguous = PyObject_IsTrue(r);
    Py_DECREF(r);
    if (contiguous) return contiguous < 0 ? -1 : 0;
    r = PyObject_CallMethodNoArgs(x, s_stride);
    if (!r) return -1;
    if (!PyTuple_Check(r) || PyTuple_GET_SIZE(r) != 4 || PyLong_AsLongLong(PyTuple_GET_ITEM(r, 3)) != 1) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_AssertionError, "expected [rows, heads, T, D] with contiguous channels");
        Py_DECREF(r);
        return -1;
    }
    for (int i = 0; i < 3; ++i) strides[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(r, i));
    Py_DECREF(r);
    *strided = 1;
    return PyErr_Occurred() ? -1 : 0;
}

static int stream_of(PyObject* s, void** out) /* None, an address, or something with .cuda_stream */
{
    if (s == Py_None || PyLong_CheckExact(s)) return as_pointer(s, out);
    PyObject* a = PyObject_GetAttr(s, s_cuda_stream);
    if (!a) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
        PyErr_Clear();
        return as_pointer(s, out);
    }
    const int bad = as_pointer(a, out);
    Py_DECREF(a);
    return bad;
}

static int head(PyObject* const* args, void** cache, int* layer, int* scale)
{
    if (as_pointer(args[0], cache)) return -1;
    const long l = PyLong_AsLong(args[1]), s = PyLong_AsLong(args[2]);
    if (PyErr_Occurred()) return -1;
    *layer = (int)l;
    *scale = (int)s;
    if (l != *layer || s != *scale) {
        PyErr_SetString(PyExc_OverflowError, "layer or scale out of range");
        return -1;
    }
    return 0;
}

static int key_value(PyObject* K, PyObject* V, void** k, void** v, int64_t* ks, int* strided)
{
    int64_t vs[3];
    int v_strided;
    if (tensor(K, k, ks, strided) || tensor(V, v, vs, &v_strided)) return -1;
    if (*strided != v_strided || (*strided && (ks[0] != vs[0] || ks[1] != vs[1] || ks[2] != vs[2]))) {
        PyErr_SetString(PyExc_ValueError, "K and V must share one stride triple");
        return -1;
    }
    return 0;
}

static int count(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want && f_append) return 0;
    PyErr_SetString(PyExc_TypeError, f_append ? "wrong number of arguments" : "bind() has not been called");
    return -1;
}

/* append(cache, layer, scale, K, V, stream) -> return code */
static PyObject* py_append(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void *cache, *k, *v, *stream;
    int layer, scale, kv, rc;
    int64_t ks[3];
    if (count(n, 6) || head(args, &cache, &layer, &scale) || key_value(args[3], args[4], &k, &v, ks, &kv) || stream_of(args[5], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_append(cache, layer, scale, k, v, kv ? ks : NULL, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* attend(cache, layer, scale, Q, out, stream) -> return code */
static PyObject* py_attend(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void *cache, *q, *o, *stream;
    int layer, scale, qv, ov, rc;
    int64_t qs[3], os[3];
    if (count(n, 6) || head(args, &cache, &layer, &scale) || tensor(args[3], &q, qs, &qv) || tensor(args[4], &o, os, &ov) ||
        stream_of(args[5], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_attend(cache, layer, scale, q, o, qv ? qs : NULL, ov ? os : NULL, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* append_attend(cache, layer, scale, K, V, Q, out, stream) -> return code */
static PyObject* py_append_attend(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void *cache, *k, *v, *q, *o, *stream;
    int layer, scale, kv, qv, ov, rc;
    int64_t ks[3], qs[3], os[3];
    if (count(n, 8) || head(args, &cache, &layer, &scale) || key_value(args[3], args[4], &k, &v, ks, &kv) ||
        tensor(args[5], &q, qs, &qv) || tensor(args[6], &o, os, &ov) || stream_of(args[7], &stream))
        return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_append_attend(cache, layer, scale, k, v, kv ? ks : NULL, q, o, qv ? qs : NULL, ov ? os : NULL, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* bind(append, attend, append_attend): addresses of the library's functions */
static PyObject* py_bind(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void* f[3];
    if (n != 3) {
        PyErr_SetString(PyExc_TypeError, "bind(append, attend, append_attend)");
        return NULL;
    }
    for (int i = 0; i < 3; ++i) {
        if (as_pointer(args[i], &f[i])) return NULL;
        if (!f[i]) {
            PyErr_SetString(PyExc_ValueError, "null function");
            return NULL;
        }
    }
    f_attend = (attend_fn)f[1];
    f_append_attend = (append_attend_fn)f[2];
    f_append = (append_fn)f[0];
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, NULL},
    {"append", (PyCFunction)(void (*)(void))py_append, METH_FASTCALL, NULL},
    {"attend", (PyCFunction)(void (*)(void))py_attend, METH_FASTCALL, NULL},
    {"append_attend", (PyCFunction)(void (*)(void))py_append_attend, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_steps", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__steps(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_stride = PyUnicode_InternFromString("stride");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (!s_data_ptr || !s_is_contiguous || !s_stride || !s_cuda_stream) return NULL;
    return PyModule_Create(&module);
}
