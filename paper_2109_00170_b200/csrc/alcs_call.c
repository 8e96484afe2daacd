// The calls that a program makes once per layer, marshalled in C: the same functions of libalcs.so that binding.py
// declares through ctypes, which spends about 2 us per call on a dozen arguments, a quarter of a small layer's pass.
// The addresses of the functions come from the library that binding.py has loaded (bind), so there is one library
// and one set of entry points.  Only the plain forms of arguments are taken here: Python integers, None, what has a
// data_ptr() or a cuda_stream that is such an integer.  For any other call (numpy integers, arrays, ctypes objects, what is
// wrong) the answer is None and nothing has been called: binding.py then makes it through ctypes, whose conversions
// and errors are the interface.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

typedef int (*spconv1x1_fn)(const void*, const void*, void*, int, int, int, const float*, unsigned, void*);
typedef int (*spconv1x1_ex_fn)(const void*, const void*, void*, int, int, int, int, const float*, const void*, unsigned, const void*, void*);
typedef int (*spconv2d_fn)(const void*, const void*, void*, int, int, int, int, int, int, int, int, const float*, unsigned, void*);
typedef int (*stack_run_fn)(void*, void*);

static spconv1x1_fn f_spconv1x1;
static spconv1x1_ex_fn f_spconv1x1_ex;
static spconv2d_fn f_spconv2d;
static stack_run_fn f_stack_run;
static PyObject *s_data_ptr, *s_cuda_stream, *s_value;

// An address of a Python integer that fits one.
static int to_ptr(PyObject* o, void** out)
{
    if (!PyLong_Check(o)) return 0;
    *out = PyLong_AsVoidPtr(o);
    return *out || !PyErr_Occurred();
}

// Of a ctypes.c_void_p that is not null.
static int handle(PyObject* o, void** out)
{
    PyObject* v = PyObject_GetAttr(o, s_value);
    const int ok = v && to_ptr(v, out) && *out;
    Py_XDECREF(v);
    return ok;
}

static int address(PyObject* o, void** out)
{
    if (o == Py_None) { *out = NULL; return 1; }
    if (PyLong_Check(o)) return to_ptr(o, out);
    PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    const int ok = v && to_ptr(v, out);
    Py_XDECREF(v);
    return ok;
}

static int stream_of(PyObject* o, void** out)
{
    if (o == Py_None) { *out = NULL; return 1; }
    if (PyLong_Check(o)) return to_ptr(o, out);
    PyObject* v = PyObject_GetAttr(o, s_cuda_stream);
    const int ok = v && (v == Py_None ? (*out = NULL, 1) : to_ptr(v, out));
    Py_XDECREF(v);
    return ok;
}

// C's int of a Python integer: the low bits, as ctypes takes them.
static int integer(PyObject* o, int* out)
{
    if (!PyLong_Check(o)) return 0;
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    if (v == (unsigned long)-1 && PyErr_Occurred()) return 0;
    *out = (int)v;
    return 1;
}

// Not a plain call: None, and whatever was raised on the way is raised again where ctypes meets it.
static PyObject* not_plain(void)
{
    if (PyErr_Occurred() && !PyErr_ExceptionMatches(PyExc_Exception)) return NULL;      // (an interrupt)
    PyErr_Clear();
    Py_RETURN_NONE;
}

static PyObject* bind(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void* f[4];
    (void)self;
    for (int i = 0; i < 4; ++i)
        if (n != 4 || !to_ptr(a[i], &f[i])) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "four addresses expected");
            return NULL;
        }
    f_spconv1x1 = (spconv1x1_fn)f[0];
    f_spconv1x1_ex = (spconv1x1_ex_fn)f[1];
    f_spconv2d = (spconv2d_fn)f[2];
    f_stack_run = (stack_run_fn)f[3];
    Py_RETURN_NONE;
}

// Each: the status, or None.  w, x, y, n, h, wd, bias, flags, stream
static PyObject* spconv1x1(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *w, *x, *y, *bias, *st;
    int d[3], flags, rc;
    (void)self;
    if (n != 9 || !handle(a[0], &w) || !address(a[1], &x) || !address(a[2], &y)) return not_plain();
    for (int i = 0; i < 3; ++i)
        if (!integer(a[3 + i], &d[i])) return not_plain();
    if (!address(a[6], &bias) || !integer(a[7], &flags) || !stream_of(a[8], &st)) return not_plain();
    Py_BEGIN_ALLOW_THREADS
    rc = f_spconv1x1(w, x, y, d[0], d[1], d[2], bias, (unsigned)flags, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// w, x, y, n, h, wd, stride, bias, residual, flags, stream
static PyObject* spconv1x1_ex(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *w, *x, *y, *bias, *res, *st;
    int d[4], flags, rc;
    (void)self;
    if (n != 11 || !handle(a[0], &w) || !address(a[1], &x) || !address(a[2], &y)) return not_plain();
    for (int i = 0; i < 4; ++i)
        if (!integer(a[3 + i], &d[i])) return not_plain();
    if (!address(a[7], &bias) || !address(a[8], &res) || !integer(a[9], &flags) || !stream_of(a[10], &st)) return not_plain();
    Py_BEGIN_ALLOW_THREADS
    rc = f_spconv1x1_ex(w, x, y, d[0], d[1], d[2], d[3], bias, res, (unsigned)flags, NULL, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// w, x, y, n, cin, h, wd, kh, kw, stride, pad, bias, flags, stream
static PyObject* spconv2d(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *w, *x, *y, *bias, *st;
    int d[8], flags, rc;
    (void)self;
    if (n != 14 || !handle(a[0], &w) || !address(a[1], &x) || !address(a[2], &y)) return not_plain();
    for (int i = 0; i < 8; ++i)
        if (!integer(a[3 + i], &d[i])) return not_plain();
    if (!address(a[11], &bias) || !integer(a[12], &flags) || !stream_of(a[13], &st)) return not_plain();
    Py_BEGIN_ALLOW_THREADS
    rc = f_spconv2d(w, x, y, d[0], d[1], d[2], d[3], d[4], d[5], d[6], d[7], bias, (unsigned)flags, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// stack, stream
static PyObject* stack_run(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *s, *st;
    int rc;
    (void)self;
    if (n != 2 || !handle(a[0], &s) || !stream_of(a[1], &st)) return not_plain();
    Py_BEGIN_ALLOW_THREADS
    rc = f_stack_run(s, st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {{"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, NULL},
                                {"spconv1x1", (PyCFunction)(void (*)(void))spconv1x1, METH_FASTCALL, NULL},
                                {"spconv1x1_ex", (PyCFunction)(void (*)(void))spconv1x1_ex, METH_FASTCALL, NULL},
                                {"spconv2d", (PyCFunction)(void (*)(void))spconv2d, METH_FASTCALL, NULL},
                                {"stack_run", (PyCFunction)(void (*)(void))stack_run, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_alcs_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__alcs_call(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_value = PyUnicode_InternFromString("value");
    if (!s_data_ptr || !s_cuda_stream || !s_value) return NULL;
    return PyModule_Create(&module);
}
