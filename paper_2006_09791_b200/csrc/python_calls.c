/* Python entry points of the calls a program makes per layer and pass: argument marshalling only, in C.
 *
 * A forward of a small layer takes the GPU 2 to 3 us, and marshalling its five arguments through ctypes took the host
 * 1.8 us of every call (0.2 us per tensor for data_ptr() and the conversion, the argument array, the foreign call).  The
 * functions here do the same -- an argument is None, an integer, or an object with data_ptr() (stream: cuda_stream) -- and
 * call the library through the addresses that gconv.py hands over when it loads libgconv.so.  A status other than GCONV_OK
 * goes to gconv.py's `_check`, which raises.  The interpreter lock is released during the call, as ctypes does.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*forward_fn)(void *, const void *, const void *, void *, void *);
typedef int (*block_fn)(void *, int, const void *, const void *, void *, void *);
typedef int (*host_fn)(void *, const void *, const void *, void *, void *, void *, void *);

static forward_fn f_forward;
static block_fn f_block;
static host_fn f_host;
static PyObject *s_data_ptr, *s_cuda_stream, *o_load, *o_check;

static int to_pointer(PyObject *o, PyObject *attr, int call, void **out) {
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    PyObject *v = NULL;
    if (!PyLong_Check(o)) {
        v = call ? PyObject_CallMethodNoArgs(o, attr) : PyObject_GetAttr(o, attr);
        if (v == NULL) return 0;
        o = v;
    }
    const unsigned long long a = PyLong_AsUnsignedLongLongMask(o);
    Py_XDECREF(v);
    if (a == (unsigned long long)-1 && PyErr_Occurred()) return 0;
    *out = (void *)(uintptr_t)a;
    return 1;
}

/* positional and keyword arguments into out[0 .. count), borrowed; the last one defaults to None */
static int take(const char *name, const char *const *names, int count, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames, PyObject **out) {
    if (nargs == count && kwnames == NULL) {
        for (int i = 0; i < count; ++i) out[i] = args[i];
        return 1;
    }
    if (nargs > count) {
        PyErr_Format(PyExc_TypeError, "%s() takes %d arguments but %zd were given", name, count, nargs);
        return 0;
    }
    for (int i = 0; i < count; ++i) out[i] = i < nargs ? args[i] : NULL;
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
        PyObject *kw = PyTuple_GET_ITEM(kwnames, k);
        int i = 0;
        while (i < count && PyUnicode_CompareWithASCIIString(kw, names[i]) != 0) ++i;
        if (i == count || out[i] != NULL) {
            PyErr_Format(PyExc_TypeError, "%s() got %s argument '%U'", name, i == count ? "an unexpected keyword" : "multiple values for", kw);
            return 0;
        }
        out[i] = args[nargs + k];
    }
    for (int i = 0; i < count; ++i) {
        if (out[i] != NULL) continue;
        if (i != count - 1) {
            PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", name, names[i]);
            return 0;
        }
        out[i] = Py_None;
    }
    return 1;
}

static int loaded(void) {
    if (f_forward != NULL) return 1;
    PyObject *r = o_load ? PyObject_CallNoArgs(o_load) : NULL;      /* gconv.load(): opens the library and calls bind() */
    Py_XDECREF(r);
    if (r != NULL && f_forward == NULL) PyErr_SetString(PyExc_ImportError, "libgconv.so is not bound");
    return f_forward != NULL;
}

static PyObject *finish(int rc, const char *name) {
    if (rc == 0) Py_RETURN_NONE;
    return PyObject_CallFunction(o_check, "is", rc, name);
}

static PyObject *py_forward(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    static const char *const names[] = {"desc", "x_nchw", "w_packed", "y_nchw", "stream"};
    PyObject *a[5];
    void *p[5];
    int rc;
    if (!take("gconv_forward", names, 5, args, nargs, kwnames, a) || !loaded()) return NULL;
    for (int i = 0; i < 4; ++i)
        if (!to_pointer(a[i], s_data_ptr, 1, &p[i])) return NULL;
    if (!to_pointer(a[4], s_cuda_stream, 0, &p[4])) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_forward(p[0], p[1], p[2], p[3], p[4]);
    Py_END_ALLOW_THREADS
    return finish(rc, "gconv_forward");
}

static PyObject *py_block(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    static const char *const names[] = {"desc", "C2", "x_nchw", "w_packed", "y2_nchw", "stream"};
    PyObject *a[6];
    void *p[6];
    int rc;
    if (!take("gconv_block_forward", names, 6, args, nargs, kwnames, a) || !loaded()) return NULL;
    if (!to_pointer(a[0], s_data_ptr, 1, &p[0])) return NULL;
    const long c2 = PyLong_AsLong(a[1]);
    if (c2 == -1 && PyErr_Occurred()) return NULL;
    for (int i = 2; i < 5; ++i)
        if (!to_pointer(a[i], s_data_ptr, 1, &p[i])) return NULL;
    if (!to_pointer(a[5], s_cuda_stream, 0, &p[5])) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_block(p[0], (int)c2, p[2], p[3], p[4], p[5]);
    Py_END_ALLOW_THREADS
    return finish(rc, "gconv_block_forward");
}

static PyObject *py_host(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    static const char *const names[] = {"desc", "x_host", "w_packed", "y_host", "x_stage", "y_stage", "stream"};
    PyObject *a[7];
    void *p[7];
    int rc;
    if (!take("gconv_forward_host", names, 7, args, nargs, kwnames, a) || !loaded()) return NULL;
    for (int i = 0; i < 6; ++i)
        if (!to_pointer(a[i], s_data_ptr, 1, &p[i])) return NULL;
    if (!to_pointer(a[6], s_cuda_stream, 0, &p[6])) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_host(p[0], p[1], p[2], p[3], p[4], p[5], p[6]);
    Py_END_ALLOW_THREADS
    return finish(rc, "gconv_forward_host");
}

/* setup(load, check): the functions that open the library and turn a status into an exception */
static PyObject *py_setup(PyObject *self, PyObject *args) {
    PyObject *load, *check;
    if (!PyArg_ParseTuple(args, "OO", &load, &check)) return NULL;
    Py_INCREF(load);
    Py_INCREF(check);
    Py_XSETREF(o_load, load);
    Py_XSETREF(o_check, check);
    Py_RETURN_NONE;
}

/* bind(forward, block_forward, forward_host): addresses of the library's functions */
static PyObject *py_bind(PyObject *self, PyObject *args) {
    unsigned long long f, b, h;
    if (!PyArg_ParseTuple(args, "KKK", &f, &b, &h)) return NULL;
    f_block = (block_fn)(uintptr_t)b;
    f_host = (host_fn)(uintptr_t)h;
    f_forward = (forward_fn)(uintptr_t)f;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"gconv_forward", (PyCFunction)(void (*)(void))py_forward, METH_FASTCALL | METH_KEYWORDS,
     "gconv_forward($module, /, desc, x_nchw, w_packed, y_nchw, stream=None)\n--\n\nThe grouped convolution (asynchronous on `stream`)."},
    {"gconv_block_forward", (PyCFunction)(void (*)(void))py_block, METH_FASTCALL | METH_KEYWORDS,
     "gconv_block_forward($module, /, desc, C2, x_nchw, w_packed, y2_nchw, stream=None)\n--\n\n"
     "Grouped 3x3 convolution followed by the pointwise convolution, one kernel (asynchronous)."},
    {"gconv_forward_host", (PyCFunction)(void (*)(void))py_host, METH_FASTCALL | METH_KEYWORDS,
     "gconv_forward_host($module, /, desc, x_host, w_packed, y_host, x_stage, y_stage, stream=None)\n--\n\n"
     "The grouped convolution on host buffers: copies x in and y out around it (asynchronous with pinned buffers)."},
    {"setup", py_setup, METH_VARARGS, NULL},
    {"bind", py_bind, METH_VARARGS, NULL},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods};

PyMODINIT_FUNC PyInit__calls(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    if (s_data_ptr == NULL || s_cuda_stream == NULL) return NULL;
    return PyModule_Create(&module);
}
