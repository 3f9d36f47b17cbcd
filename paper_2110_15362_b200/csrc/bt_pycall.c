/* _pycall: calls of the C ABI from Python without ctypes' marshalling.
 *
 * native_call(address) wraps the address of an exported function that takes pointers, integers and at most one float, and
 * returns an int (an element of the ABI's status enumeration).  The wrapper is called with
 *   an integer        passed as it is (pointers, sizes, codes),
 *   None              a null pointer,
 *   a float           the function's one float argument, wherever it stands among the others,
 *   a buffer object   the address of its memory (the ctypes arrays of bt_batch_item),
 *   any other object  the result of its data_ptr() method (tensors).
 * What a small call costs is host work: ctypes took 2 to 3 us for the dozen arguments of a launch, this takes a few
 * tenths.
 *
 * On x86-64 integer and pointer arguments travel in one sequence (six registers, then the stack) and float arguments in
 * another, so one prototype -- a float and kMax integer words -- fits every such function: the callee does not look at
 * words behind its own, and the caller clears the stack.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stddef.h>
#include <stdint.h>

#if !defined(__x86_64__)
#error "the argument passing relied on here is that of x86-64"
#endif

enum { kMax = 18, kMaxBuffers = 4 };

typedef uint64_t W;
typedef int (*Function)(float, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W);

typedef struct {
    PyObject_HEAD
    vectorcallfunc vectorcall;
    Function       function;
} NativeCall;

static PyObject *s_data_ptr;

static PyObject *native_call_vectorcall(PyObject *self, PyObject *const *args, size_t nargsf, PyObject *kwnames)
{
    const Py_ssize_t n = PyVectorcall_NARGS(nargsf);
    W                a[kMax] = {0};
    float            f       = 0.0f;
    Py_buffer        buffers[kMaxBuffers];
    int              held = 0, k = 0, status = 0;
    if (kwnames != NULL && PyTuple_GET_SIZE(kwnames) != 0) {
        PyErr_SetString(PyExc_TypeError, "a native call takes no keyword arguments");
        return NULL;
    }
    if (n > kMax + 1) {
        PyErr_SetString(PyExc_TypeError, "too many arguments");
        return NULL;
    }
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject *const o = args[i];
        if (PyFloat_Check(o)) {
            f = (float)PyFloat_AS_DOUBLE(o);
            continue;
        }
        if (k == kMax) {
            PyErr_SetString(PyExc_TypeError, "too many arguments");
            goto fail;
        }
        if (o == Py_None) {
            a[k++] = 0;
        } else if (PyLong_Check(o)) {
            a[k] = PyLong_AsUnsignedLongLongMask(o);
            if (a[k++] == (W)-1 && PyErr_Occurred()) goto fail;
        } else if (PyObject_CheckBuffer(o) && !PyIndex_Check(o)) {
            if (held == kMaxBuffers) {
                PyErr_SetString(PyExc_TypeError, "too many buffer arguments");
                goto fail;
            }
            if (PyObject_GetBuffer(o, &buffers[held], PyBUF_SIMPLE) != 0) goto fail;
            a[k++] = (W)(uintptr_t)buffers[held++].buf;
        } else {
            PyObject *p = PyObject_CallMethodNoArgs(o, s_data_ptr);
            if (p == NULL && PyIndex_Check(o) && PyErr_ExceptionMatches(PyExc_AttributeError)) {      // other integer types
                PyErr_Clear();
                p = PyNumber_Index(o);
            }
            if (p == NULL) goto fail;
            a[k] = PyLong_AsUnsignedLongLongMask(p);
            Py_DECREF(p);
            if (a[k++] == (W)-1 && PyErr_Occurred()) goto fail;
        }
    }
    {
        const Function fn = ((NativeCall *)self)->function;
        Py_BEGIN_ALLOW_THREADS
        status = fn(f, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17]);
        Py_END_ALLOW_THREADS
    }
    while (held > 0) PyBuffer_Release(&buffers[--held]);
    return PyLong_FromLong(status);
fail:
    while (held > 0) PyBuffer_Release(&buffers[--held]);
    return NULL;
}

static PyMemberDef native_call_members[] = {
    {"__vectorcalloffset__", Py_T_PYSSIZET, offsetof(NativeCall, vectorcall), Py_READONLY, NULL},
    {NULL, 0, 0, 0, NULL},
};

static void native_call_dealloc(PyObject *self)
{
    PyTypeObject *const type = Py_TYPE(self);
    type->tp_free(self);
    Py_DECREF(type);
}

static PyType_Slot native_call_slots[] = {
    {Py_tp_members, native_call_members},
    {Py_tp_call, PyVectorcall_Call},
    {Py_tp_dealloc, native_call_dealloc},
    {0, NULL},
};
static PyType_Spec native_call_spec = {
    "_pycall.NativeCall", sizeof(NativeCall), 0, Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL | Py_TPFLAGS_DISALLOW_INSTANTIATION, native_call_slots,
};

static PyObject *s_type;

static PyObject *native_call(PyObject *module, PyObject *address)
{
    (void)module;
    const W at = PyLong_AsUnsignedLongLong(address);
    if (PyErr_Occurred()) return NULL;
    if (at == 0) {
        PyErr_SetString(PyExc_ValueError, "null function address");
        return NULL;
    }
    PyTypeObject *const type = (PyTypeObject *)s_type;
    NativeCall *const   c    = (NativeCall *)type->tp_alloc(type, 0);
    if (c == NULL) return NULL;
    c->vectorcall = native_call_vectorcall;
    c->function   = (Function)(uintptr_t)at;
    return (PyObject *)c;
}

static PyMethodDef methods[] = {
    {"native_call", native_call, METH_O, "A callable for the exported function at an address."},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_pycall", "Calls of the C ABI without ctypes.", -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_type     = PyType_FromSpec(&native_call_spec);
    if (s_data_ptr == NULL || s_type == NULL) return NULL;
    return PyModule_Create(&module_def);
}
