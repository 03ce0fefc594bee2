/* Calls an entry point of libscap_b200.so from Python: call(address, arg, ...) -> status.
 *
 * An argument is None (null), an integer, or an object with data_ptr() (a tensor: its address).  Every parameter of the entry
 * points called this way is a pointer, an integer or a size, which the x86-64 calling convention passes alike, one 64-bit slot
 * each.  Why it is here: at one token a call is bound by the host, and the conversion of fifteen arguments by ctypes cost more
 * than the kernel launch (K = N = 1024, one row: 10.5 us a call, 5.3 with this). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#define MAX_ARGS 24
typedef long long slot;
typedef int (*entry)(slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot, slot,
                     slot, slot, slot, slot, slot);

static PyObject *s_data_ptr;

static int to_slot(PyObject *o, slot *out) {
    if (o == Py_None) {
        *out = 0;
        return 0;
    }
    if (PyLong_Check(o)) {
        *out = PyLong_AsLongLong(o);
        if (*out == -1 && PyErr_Occurred()) {  /* an address or a size beyond 2^63 */
            PyErr_Clear();
            *out = (slot)PyLong_AsUnsignedLongLong(o);
            if (PyErr_Occurred()) return -1;
        }
        return 0;
    }
    PyObject *r = PyObject_VectorcallMethod(s_data_ptr, &o, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, NULL);
    if (!r) return -1;
    *out = (slot)PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

static PyObject *call(PyObject *self, PyObject *const *args, Py_ssize_t n) {
    slot a[MAX_ARGS] = {0};
    (void)self;
    if (n < 1 || n - 1 > MAX_ARGS) {
        PyErr_SetString(PyExc_TypeError, "call(address, up to 24 arguments)");
        return NULL;
    }
    const entry f = (entry)PyLong_AsVoidPtr(args[0]);
    if (!f) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point");
        return NULL;
    }
    for (Py_ssize_t i = 1; i < n; ++i)
        if (to_slot(args[i], &a[i - 1])) return NULL;
    int status;
    Py_BEGIN_ALLOW_THREADS  /* as ctypes does: other threads run during the call */
    /* surplus slots are never read by the callee and removed by the caller */
    status = f(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17], a[18],
               a[19], a[20], a[21], a[22], a[23]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

static PyMethodDef methods[] = {{"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(address, arg, ...) -> status"}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_scap_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__scap_call(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return s_data_ptr ? PyModule_Create(&module) : NULL;
}
