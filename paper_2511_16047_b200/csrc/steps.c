/* Python side of the calls of a generation step (amskv_append, amskv_attend, amskv_append_attend): takes addresses and strides
 * out of the tensors and calls the library, without the argument conversions of ctypes.  Marshalling only, and only of the
 * usual forms: a call with any other argument returns None without having called the library, and the binding makes it
 * through ctypes, which decides what is accepted and what the error is.
 *
 * These calls are made layers x scales times per image; through ctypes their Python side took 2.1 us with contiguous tensors
 * and 3.3 us with views, about what the launch itself takes; here 0.8 and 1.4.
 *
 * The usual forms: a handle, layer, scale or address that is exactly an int (None as an address), a tensor with data_ptr(),
 * is_contiguous() and stride() (a torch tensor), a stream that is None, an int or has an int as .cuda_stream.
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

/* The helpers below return 0, or -1 for an argument that is left to ctypes (with or without an error set). */

static int as_pointer(PyObject* o, void** out) /* an int, or None */
{
    if (o == Py_None) {
        *out = NULL;
        return 0;
    }
    if (!PyLong_CheckExact(o)) return -1;
    *out = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
    return 0;
}

/* address of a tensor argument; strides[3] and *strided = 1 when it is a view that is not contiguous */
static int tensor(PyObject* x, void** addr, int64_t* strides, int* strided)
{
    *strided = 0;
    if (x == Py_None || PyLong_CheckExact(x)) return as_pointer(x, addr);
    PyObject* r = PyObject_CallMethodNoArgs(x, s_data_ptr);
    if (!r) return -1;
    const int bad = as_pointer(r, addr);
    Py_DECREF(r);
    if (bad) return -1;
    r = PyObject_CallMethodNoArgs(x, s_is_contiguous);
    if (!r) return -1;
    const int contiguous = r == Py_True ? 1 : r == Py_False ? 0 : -1;
    Py_DECREF(r);
    if (contiguous) return contiguous < 0 ? -1 : 0;
    r = PyObject_CallMethodNoArgs(x, s_stride);
    if (!r) return -1;
    int ok = PyTuple_Check(r) && PyTuple_GET_SIZE(r) == 4;
    for (int i = 0; ok && i < 4; ++i) {
        const long long v = PyLong_AsLongLong(PyTuple_GET_ITEM(r, i));
        if (i < 3) strides[i] = v;
        ok = i < 3 ? !PyErr_Occurred() : v == 1;
    }
    Py_DECREF(r);
    *strided = 1;
    return ok ? 0 : -1;
}

static int stream_of(PyObject* s, void** out) /* None, an address, or something with .cuda_stream */
{
    if (s == Py_None || PyLong_CheckExact(s)) return as_pointer(s, out);
    PyObject* a = PyObject_GetAttr(s, s_cuda_stream);
    if (!a) return -1;
    const int bad = as_pointer(a, out);
    Py_DECREF(a);
    return bad;
}

static int head(PyObject* const* args, void** cache, int* layer, int* scale)
{
    if (as_pointer(args[0], cache) || !PyLong_CheckExact(args[1]) || !PyLong_CheckExact(args[2])) return -1;
    const long l = PyLong_AsLong(args[1]), s = PyLong_AsLong(args[2]);
    *layer = (int)l;
    *scale = (int)s;
    return PyErr_Occurred() || l != *layer || s != *scale ? -1 : 0;
}

static int key_value(PyObject* K, PyObject* V, void** k, void** v, int64_t* ks, int* strided)
{
    int64_t vs[3];
    int v_strided;
    if (tensor(K, k, ks, strided) || tensor(V, v, vs, &v_strided)) return -1;
    return *strided != v_strided || (*strided && (ks[0] != vs[0] || ks[1] != vs[1] || ks[2] != vs[2])) ? -1 : 0;
}

static int count(Py_ssize_t n, Py_ssize_t want)
{
    if (n == want && f_append) return 0;
    PyErr_SetString(PyExc_TypeError, f_append ? "wrong number of arguments" : "bind() has not been called");
    return -1;
}

static PyObject* left_to_ctypes(void)
{
    PyErr_Clear();
    Py_RETURN_NONE;
}

/* append(cache, layer, scale, K, V, stream) -> return code, or None */
static PyObject* py_append(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void *cache, *k, *v, *stream;
    int layer, scale, kv, rc;
    int64_t ks[3];
    if (count(n, 6)) return NULL;
    if (head(args, &cache, &layer, &scale) || key_value(args[3], args[4], &k, &v, ks, &kv) || stream_of(args[5], &stream))
        return left_to_ctypes();
    Py_BEGIN_ALLOW_THREADS
    rc = f_append(cache, layer, scale, k, v, kv ? ks : NULL, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* attend(cache, layer, scale, Q, out, stream) -> return code, or None */
static PyObject* py_attend(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void *cache, *q, *o, *stream;
    int layer, scale, qv, ov, rc;
    int64_t qs[3], os[3];
    if (count(n, 6)) return NULL;
    if (head(args, &cache, &layer, &scale) || tensor(args[3], &q, qs, &qv) || tensor(args[4], &o, os, &ov) ||
        stream_of(args[5], &stream))
        return left_to_ctypes();
    Py_BEGIN_ALLOW_THREADS
    rc = f_attend(cache, layer, scale, q, o, qv ? qs : NULL, ov ? os : NULL, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

/* append_attend(cache, layer, scale, K, V, Q, out, stream) -> return code, or None */
static PyObject* py_append_attend(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    void *cache, *k, *v, *q, *o, *stream;
    int layer, scale, kv, qv, ov, rc;
    int64_t ks[3], qs[3], os[3];
    if (count(n, 8)) return NULL;
    if (head(args, &cache, &layer, &scale) || key_value(args[3], args[4], &k, &v, ks, &kv) || tensor(args[5], &q, qs, &qv) ||
        tensor(args[6], &o, os, &ov) || stream_of(args[7], &stream))
        return left_to_ctypes();
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
        if (as_pointer(args[i], &f[i]) || !f[i]) {
            PyErr_SetString(PyExc_ValueError, "bind() wants addresses");
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
