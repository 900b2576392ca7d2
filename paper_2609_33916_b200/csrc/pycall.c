/* Calls of the library's launch functions from Python: the marshalling of binding.py for the calls whose kernels can be shorter than it.
 *
 * invoke(entry, desc, pointer..., [workspace bytes,] stream) -> status.  `entry` is what add_entry() returned for a function's
 * address.  A pointer argument is None, an integer address, or an object with data_ptr() (a tensor); workspace bytes of None: the nbytes of
 * the last pointer argument, which is the workspace; a stream of None: the current one, an integer: its address, else an object with
 * cuda_stream. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#define MAX_ARGS 16 /* pointers, workspace bytes and stream */

static struct entry {
    uintptr_t fn;
    PyTypeObject *desc_type;
    Py_ssize_t npointers; /* pointer arguments, the workspace included */
    int has_ws;
} *entries; /* (grows: a reloaded binding registers its own descriptor types) */
static int nentries;
static PyObject *s_data_ptr, *s_nbytes, *s_cuda_stream;
static PyObject *stream_getter, *device_getter; /* stream_getter(device_getter()), or stream_getter() without the second */

static PyObject *add_entry(PyObject *self, PyObject *args)
{
    unsigned long long fn;
    PyObject *type;
    Py_ssize_t npointers;
    int has_ws;
    struct entry *more;
    (void)self;
    if (!PyArg_ParseTuple(args, "KO!np", &fn, &PyType_Type, &type, &npointers, &has_ws)) return NULL;
    if (npointers < 1 || npointers + 2 > MAX_ARGS) {
        PyErr_SetString(PyExc_ValueError, "too many arguments");
        return NULL;
    }
    more = PyMem_Realloc(entries, (size_t)(nentries + 1) * sizeof *entries);
    if (!more) return PyErr_NoMemory();
    entries = more;
    Py_INCREF(type);
    entries[nentries].fn = (uintptr_t)fn;
    entries[nentries].desc_type = (PyTypeObject *)type;
    entries[nentries].npointers = npointers;
    entries[nentries].has_ws = has_ws;
    return PyLong_FromLong(nentries++);
}

static PyObject *set_current_stream(PyObject *self, PyObject *args)
{
    PyObject *f, *device = NULL;
    (void)self;
    if (!PyArg_ParseTuple(args, "O|O", &f, &device)) return NULL;
    Py_INCREF(f);
    Py_XINCREF(device);
    Py_XSETREF(stream_getter, f);
    Py_XSETREF(device_getter, device);
    Py_RETURN_NONE;
}

static PyObject *current_stream(void)
{
    PyObject *f = stream_getter, *d = device_getter, *device, *v;
    if (!f) {
        PyErr_SetString(PyExc_RuntimeError, "no current stream");
        return NULL;
    }
    Py_INCREF(f); /* (the call may replace them) */
    Py_XINCREF(d);
    if (d) {
        device = PyObject_CallNoArgs(d);
        v = device ? PyObject_CallOneArg(f, device) : NULL;
        Py_XDECREF(device);
    } else {
        v = PyObject_CallNoArgs(f);
    }
    Py_DECREF(f);
    Py_XDECREF(d);
    return v;
}

/* v (a new reference or NULL) as an unsigned integer */
static int number(PyObject *v, uint64_t *out)
{
    if (!v) return -1;
    *out = PyLong_AsUnsignedLongLong(v);
    Py_DECREF(v);
    return *out == (uint64_t)-1 && PyErr_Occurred() ? -1 : 0;
}

/* the address an object stands for: a method (data_ptr) or an attribute (cuda_stream) gives it */
static int address(PyObject *o, PyObject *name, int method, uint64_t *out)
{
    if (o == Py_None) {
        *out = 0;
        return 0;
    }
    if (PyLong_Check(o)) {
        Py_INCREF(o);
        return number(o, out);
    }
    return number(method ? PyObject_CallMethodNoArgs(o, name) : PyObject_GetAttr(o, name), out);
}

static PyObject *invoke(PyObject *self, PyObject *const *args, Py_ssize_t nargs)
{
    uint64_t a[MAX_ARGS] = {0};
    Py_ssize_t np, i;
    Py_buffer desc;
    struct entry entry; /* (a copy: the table may move while other code runs) */
    int status;
    const long e = nargs > 0 ? PyLong_AsLong(args[0]) : -1;
    (void)self;
    if (e < 0 || e >= nentries) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "unknown entry");
        return NULL;
    }
    entry = entries[e];
    np = entry.npointers;
    if (nargs != 3 + np + (entry.has_ws ? 1 : 0)) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return NULL;
    }
    if (!PyObject_TypeCheck(args[1], entry.desc_type)) {
        PyErr_Format(PyExc_TypeError, "expected a %s", entry.desc_type->tp_name);
        return NULL;
    }
    for (i = 0; i < np; ++i)
        if (address(args[2 + i], s_data_ptr, 1, &a[i])) return NULL;
    if (entry.has_ws) {
        PyObject *ws = args[1 + np], *bytes = args[2 + np];
        if (bytes != Py_None) {
            Py_INCREF(bytes);
            if (number(bytes, &a[i])) return NULL;
        } else if (ws != Py_None && number(PyObject_GetAttr(ws, s_nbytes), &a[i])) {
            return NULL;
        }
        ++i;
    }
    if (args[nargs - 1] == Py_None ? number(current_stream(), &a[i]) : address(args[nargs - 1], s_cuda_stream, 0, &a[i])) return NULL;
    if (PyObject_GetBuffer(args[1], &desc, PyBUF_SIMPLE)) return NULL;
    Py_BEGIN_ALLOW_THREADS
    /* (every argument is a pointer, a size_t or a stream, an integer register or a stack slot each: one call with all the slots serves every
     * count, the callee reads as many as it has) */
    status = ((int (*)(void *, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t,
                       uint64_t, uint64_t, uint64_t, uint64_t, uint64_t))entry.fn)(
        desc.buf, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15]);
    Py_END_ALLOW_THREADS
    PyBuffer_Release(&desc);
    return PyLong_FromLong(status);
}

/* fill(struct, objects): the addresses of a tuple's objects, each as in invoke(), into the first words of a struct of pointers */
static PyObject *fill(PyObject *self, PyObject *const *args, Py_ssize_t nargs)
{
    Py_buffer to;
    Py_ssize_t i, n;
    (void)self;
    if (nargs != 2 || !PyTuple_Check(args[1])) {
        PyErr_SetString(PyExc_TypeError, "expected a struct and a tuple");
        return NULL;
    }
    if (PyObject_GetBuffer(args[0], &to, PyBUF_WRITABLE)) return NULL;
    n = PyTuple_GET_SIZE(args[1]);
    if (n * 8 > to.len) PyErr_SetString(PyExc_ValueError, "more objects than words");
    for (i = 0; i < n && !PyErr_Occurred(); ++i) address(PyTuple_GET_ITEM(args[1], i), s_data_ptr, 1, (uint64_t *)to.buf + i);
    PyBuffer_Release(&to);
    if (PyErr_Occurred()) return NULL;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"fill", (PyCFunction)(void (*)(void))fill, METH_FASTCALL, "fill(struct, objects): their addresses into its first words"},
    {"add_entry", add_entry, METH_VARARGS, "add_entry(address, descriptor type, pointer arguments, has a workspace) -> entry"},
    {"set_current_stream", set_current_stream, METH_VARARGS, "(f): f() is the current stream's address; (f, device): f(device()) is"},
    {"invoke", (PyCFunction)(void (*)(void))invoke, METH_FASTCALL, "invoke(entry, desc, pointers..., [ws_bytes,] stream) -> status"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_nbytes = PyUnicode_InternFromString("nbytes");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    return s_data_ptr && s_nbytes && s_cuda_stream ? PyModule_Create(&module) : NULL;
}
