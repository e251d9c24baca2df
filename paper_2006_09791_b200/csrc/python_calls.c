/* Python entry points of the calls a program makes per layer and pass: argument marshalling only, in C.
 *
 * A forward of a small layer takes the GPU 2 to 3 us, and marshalling its five arguments through ctypes took the host
 * 1.8 us of every call (0.2 us per tensor for data_ptr() and the conversion, the argument array, the foreign call).  The
 * functions here do the same for the usual arguments -- a descriptor and a C2 that are integers, tensors and a stream that are
 * None, an integer, or an object with data_ptr() (stream: cuda_stream) -- and call the library through the addresses that
 * gconv.py hands over when it loads libgconv.so.  Everything else, wrong arguments included, goes to gconv.py's own function
 * of the same name, so both accept and refuse the same.  A status other than GCONV_OK goes to gconv.py's `_check`, which
 * raises.  The interpreter lock is released during the call, as ctypes does.
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
static PyObject *s_data_ptr, *s_cuda_stream, *o_load, *o_check, *o_own[3];   /* o_own: gconv.py's functions, in the order of bind() */

/* None, an integer, or -- `attr` given -- what an object's method (`call`) or attribute of that name gives; 0: none of these */
static int to_pointer(PyObject *o, PyObject *attr, int call, void **out) {
    if (o == Py_None) {
        *out = NULL;
        return 1;
    }
    PyObject *v = NULL;
    if (!PyLong_Check(o)) {
        if (attr == NULL) return 0;
        v = call ? PyObject_CallMethodNoArgs(o, attr) : PyObject_GetAttr(o, attr);
        if (v == NULL || !PyLong_Check(v)) {
            Py_XDECREF(v);
            PyErr_Clear();                   /* (gconv.py's function raises it again) */
            return 0;
        }
        o = v;
    }
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
    Py_XDECREF(v);
    return 1;
}

/* positional and keyword arguments into out[0 .. count), borrowed; the last one defaults to None; 0: they do not fit */
static int take(const char *const *names, int count, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames, PyObject **out) {
    if (nargs > count) return 0;
    for (int i = 0; i < count; ++i) out[i] = i < nargs ? args[i] : NULL;
    const Py_ssize_t nkw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nkw; ++k) {
        PyObject *kw = PyTuple_GET_ITEM(kwnames, k);
        int i = 0;
        while (i < count && PyUnicode_CompareWithASCIIString(kw, names[i]) != 0) ++i;
        if (i == count || out[i] != NULL) return 0;
        out[i] = args[nargs + k];
    }
    for (int i = 0; i < count - 1; ++i)
        if (out[i] == NULL) return 0;
    if (out[count - 1] == NULL) out[count - 1] = Py_None;
    return 1;
}

static PyObject *own(int which, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) { return PyObject_Vectorcall(o_own[which], args, nargs, kwnames); }

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
    int rc, ok = take(names, 5, args, nargs, kwnames, a);
    for (int i = 0; ok && i < 4; ++i) ok = to_pointer(a[i], i > 0 ? s_data_ptr : NULL, 1, &p[i]);
    if (!ok || !to_pointer(a[4], s_cuda_stream, 0, &p[4])) return own(0, args, nargs, kwnames);
    if (!loaded()) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_forward(p[0], p[1], p[2], p[3], p[4]);
    Py_END_ALLOW_THREADS
    return finish(rc, "gconv_forward");
}

static PyObject *py_block(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    static const char *const names[] = {"desc", "C2", "x_nchw", "w_packed", "y2_nchw", "stream"};
    PyObject *a[6];
    void *p[6];
    int rc, ok = take(names, 6, args, nargs, kwnames, a) && PyLong_Check(a[1]) && to_pointer(a[0], NULL, 0, &p[0]);
    for (int i = 2; ok && i < 5; ++i) ok = to_pointer(a[i], s_data_ptr, 1, &p[i]);
    if (!ok || !to_pointer(a[5], s_cuda_stream, 0, &p[5])) return own(1, args, nargs, kwnames);
    const int c2 = (int)PyLong_AsUnsignedLongLongMask(a[1]);
    if (!loaded()) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_block(p[0], c2, p[2], p[3], p[4], p[5]);
    Py_END_ALLOW_THREADS
    return finish(rc, "gconv_block_forward");
}

static PyObject *py_host(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames) {
    static const char *const names[] = {"desc", "x_host", "w_packed", "y_host", "x_stage", "y_stage", "stream"};
    PyObject *a[7];
    void *p[7];
    int rc, ok = take(names, 7, args, nargs, kwnames, a);
    for (int i = 0; ok && i < 6; ++i) ok = to_pointer(a[i], i > 0 ? s_data_ptr : NULL, 1, &p[i]);
    if (!ok || !to_pointer(a[6], s_cuda_stream, 0, &p[6])) return own(2, args, nargs, kwnames);
    if (!loaded()) return NULL;
    Py_BEGIN_ALLOW_THREADS
    rc = f_host(p[0], p[1], p[2], p[3], p[4], p[5], p[6]);
    Py_END_ALLOW_THREADS
    return finish(rc, "gconv_forward_host");
}

/* setup(load, check, forward, block_forward, forward_host): the functions that open the library and turn a status into an
 * exception, and gconv.py's own functions */
static PyObject *py_setup(PyObject *self, PyObject *args) {
    PyObject *load, *check, *o[3];
    if (!PyArg_ParseTuple(args, "OOOOO", &load, &check, &o[0], &o[1], &o[2])) return NULL;
    Py_XSETREF(o_load, Py_NewRef(load));
    Py_XSETREF(o_check, Py_NewRef(check));
    for (int i = 0; i < 3; ++i) Py_XSETREF(o_own[i], Py_NewRef(o[i]));
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
