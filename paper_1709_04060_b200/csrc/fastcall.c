/* The host path of a call from Python: descriptor, device pointers and stream handed to an entry point of
 * the C ABI without ctypes.
 *
 * A small product takes 2 to 5 us on the device, and the ctypes way to its launch took 2.2 us of host time
 * before the entry point was reached (argument objects, one Python frame per pointer, isinstance through
 * torch's metaclass); this takes 0.8.  Only the plain forms are handled here -- a descriptor of the
 * expected type, contiguous tensors, integers, None --; anything else goes to the ctypes function that
 * was given at binding, which converts or refuses it as it always did. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stddef.h>
#include <stdint.h>

#define MAX_ARGS 8

typedef struct {
    PyObject_HEAD
    vectorcallfunc vectorcall;
    uint64_t (*fn)(uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t);
    int n;
    char kinds[MAX_ARGS + 1];      /* d descriptor, p pointer, n number, s stream */
    PyTypeObject *desc_type, *tensor_type;
    PyObject *slow;                /* the ctypes way */
    PyObject *raw_stream, *device, *initialized;
} Entry;

static PyObject *s_data_ptr, *s_is_contiguous;

/* 1: converted, 0: not a plain form, -1: an exception is set */
static int pointer_of(Entry *e, PyObject *x, uint64_t *out) {
    if (x == Py_None) { *out = 0; return 1; }
    if (PyLong_CheckExact(x)) {
        *out = PyLong_AsUnsignedLongLongMask(x);
        return PyErr_Occurred() ? -1 : 1;
    }
    if (!PyObject_TypeCheck(x, e->tensor_type)) return 0;
    PyObject *r = PyObject_CallMethodNoArgs(x, s_is_contiguous);
    if (!r) return -1;
    const int contiguous = r == Py_True;
    Py_DECREF(r);
    if (!contiguous) return 0;
    r = PyObject_CallMethodNoArgs(x, s_data_ptr);
    if (!r) return -1;
    *out = PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 1;
}

static int stream_of(Entry *e, PyObject *x, uint64_t *out) {
    if (PyLong_CheckExact(x)) {
        *out = PyLong_AsUnsignedLongLongMask(x);
        return PyErr_Occurred() ? -1 : 1;
    }
    if (x != Py_None || e->raw_stream == Py_None || e->device == Py_None) return 0;
    PyObject *r = PyObject_CallNoArgs(e->initialized);
    if (!r) return -1;
    const int up = r == Py_True;
    Py_DECREF(r);
    if (!up) return 0;
    PyObject *dev = PyObject_CallNoArgs(e->device);
    if (!dev) return -1;
    r = PyObject_CallOneArg(e->raw_stream, dev);
    Py_DECREF(dev);
    if (!r) return -1;
    *out = PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 1;
}

static PyObject *entry_call(PyObject *self, PyObject *const *args, size_t nargsf, PyObject *kwnames) {
    Entry *e = (Entry *)self;
    uint64_t a[MAX_ARGS] = {0};
    Py_buffer view;
    int have_view = 0, ok = PyVectorcall_NARGS(nargsf) == e->n && (kwnames == NULL || PyTuple_GET_SIZE(kwnames) == 0);
    for (int i = 0; ok == 1 && i < e->n; ++i) {
        PyObject *x = args[i];
        switch (e->kinds[i]) {
            case 'd':
                /* the structure's own memory, held by the view until the call is over */
                ok = PyObject_TypeCheck(x, e->desc_type) ? 1 : 0;
                if (ok) {
                    if (PyObject_GetBuffer(x, &view, PyBUF_SIMPLE) != 0) { ok = -1; break; }
                    have_view = 1;
                    a[i] = (uint64_t)(uintptr_t)view.buf;
                }
                break;
            case 'p': ok = pointer_of(e, x, &a[i]); break;
            case 's': ok = stream_of(e, x, &a[i]); break;
            default:
                ok = PyLong_CheckExact(x) ? 1 : 0;
                if (ok) {
                    a[i] = PyLong_AsUnsignedLongLongMask(x);
                    if (PyErr_Occurred()) ok = -1;
                }
        }
    }
    PyObject *result = NULL;
    if (ok == 1) {
        uint64_t r;
        Py_BEGIN_ALLOW_THREADS
        r = e->fn(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7]);
        Py_END_ALLOW_THREADS
        result = PyLong_FromLong((int)r);
    }
    if (have_view) PyBuffer_Release(&view);
    if (ok == 0) result = PyObject_Vectorcall(e->slow, args, nargsf, kwnames);
    return result;
}

static void entry_dealloc(PyObject *self) {
    Entry *e = (Entry *)self;
    Py_XDECREF(e->desc_type); Py_XDECREF(e->tensor_type); Py_XDECREF(e->slow);
    Py_XDECREF(e->raw_stream); Py_XDECREF(e->device); Py_XDECREF(e->initialized);
    PyObject_Free(self);
}

static PyTypeObject EntryType = {
    PyVarObject_HEAD_INIT(NULL, 0)
    .tp_name = "_fastcall.Entry",
    .tp_basicsize = sizeof(Entry),
    .tp_dealloc = entry_dealloc,
    .tp_vectorcall_offset = offsetof(Entry, vectorcall),
    .tp_call = PyVectorcall_Call,
    .tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL,
};

/* bind(address, kinds, descriptor type, tensor type, slow, raw_stream, device, initialized) */
static PyObject *bind(PyObject *module, PyObject *args) {
    unsigned long long address;
    const char *kinds;
    Py_ssize_t n;
    PyObject *desc_type, *tensor_type, *slow, *raw_stream, *device, *initialized;
    (void)module;
    if (!PyArg_ParseTuple(args, "Ks#O!O!OOOO", &address, &kinds, &n, &PyType_Type, &desc_type, &PyType_Type, &tensor_type, &slow,
                          &raw_stream, &device, &initialized))
        return NULL;
    if (n > MAX_ARGS) { PyErr_SetString(PyExc_ValueError, "too many arguments"); return NULL; }
    Entry *e = PyObject_New(Entry, &EntryType);
    if (!e) return NULL;
    e->vectorcall = entry_call;
    e->fn = (uint64_t(*)(uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t))(uintptr_t)address;
    e->n = (int)n;
    for (Py_ssize_t i = 0; i < n; ++i) e->kinds[i] = kinds[i];
    e->kinds[n] = 0;
    e->desc_type = (PyTypeObject *)Py_NewRef(desc_type); e->tensor_type = (PyTypeObject *)Py_NewRef(tensor_type);
    e->slow = Py_NewRef(slow);
    e->raw_stream = Py_NewRef(raw_stream); e->device = Py_NewRef(device); e->initialized = Py_NewRef(initialized);
    return (PyObject *)e;
}

static PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, "A callable for one entry point."}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    if (!s_data_ptr || !s_is_contiguous || PyType_Ready(&EntryType) < 0) return NULL;
    return PyModule_Create(&module);
}
