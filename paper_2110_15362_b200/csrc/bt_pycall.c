/* _pycall: calls of the C ABI from Python without ctypes' marshalling.
 *
 * native_call(address, kinds, otherwise, item) wraps the address of an exported function that takes pointers, integers and
 * at most one float, and returns an int (an element of the ABI's status enumeration).  `kinds` has a letter per parameter:
 *   p   a tensor: the result of the argument's data_ptr() method, or a null pointer for None,
 *   a   the same, or an address as an integer,
 *   s   a stream: an integer, or None,
 *   n   a count, a size or a code: an integer,
 *   f   the function's one float: a float,
 *   b   a ctypes array of `item` (bt_batch_item): the address of its memory.
 * A call whose arguments are not all of these very kinds, or not as many, is handed to `otherwise` as it is, which converts
 * or refuses them (the binding passes ctypes' own call of the same function): a float or a tensor given for a count must
 * neither move the arguments behind it nor become an address.  What a small call costs is host work: ctypes took 2 to 3 us
 * for the dozen arguments of a launch, this takes a few tenths.
 *
 * native_call(address) wraps a function without its parameters' kinds: every argument is taken for what it is itself, an
 * integer, None, a float, a buffer (its address) or a tensor, and the caller answers for their number and order.
 *
 * On x86-64 integer and pointer arguments travel in one sequence (six registers, then the stack) and float arguments in
 * another, so one prototype -- a float and kMax integer words -- fits every such function: the callee does not look at
 * words behind its own, and the caller clears the stack.  On other hosts the module is not built, and the binding calls
 * through ctypes alone.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <structmember.h>   /* T_PYSSIZET and READONLY: the names that Python versions before 3.12 have, too */
#include <stddef.h>
#include <stdint.h>
#include <string.h>

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
    char           kinds[kMax + 2];   /* a letter per parameter; empty: not given */
    Py_ssize_t     arity;
    PyObject      *otherwise, *item;
} NativeCall;

static PyObject *s_data_ptr, *s_item_type;

/* *out = the result of o.data_ptr() */
static int tensor_address(PyObject *o, W *out)
{
    PyObject *p = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (p == NULL) return -1;
    *out = PyLong_AsUnsignedLongLongMask(p);
    Py_DECREF(p);
    return *out == (W)-1 && PyErr_Occurred() ? -1 : 0;
}

/* Is o a ctypes array of `item`? */
static int is_item_array(PyObject *o, PyObject *item)
{
    PyObject *t = PyObject_GetAttr((PyObject *)Py_TYPE(o), s_item_type);
    if (t == NULL) PyErr_Clear();
    Py_XDECREF(t);
    return t != NULL && t == item && PyObject_CheckBuffer(o);
}

/* The call with checked arguments.  (An integer, here and below, is an int: its value modulo 2^64 is taken, as ctypes does.) */
static PyObject *checked_vectorcall(PyObject *self, PyObject *const *args, size_t nargsf, PyObject *kwnames)
{
    NativeCall *const c = (NativeCall *)self;
    const Py_ssize_t  n = PyVectorcall_NARGS(nargsf);
    W                 a[kMax] = {0};
    float             f       = 0.0f;
    Py_buffer         items;
    int               held = 0, k = 0, status = 0;
    if (n != c->arity || (kwnames != NULL && PyTuple_GET_SIZE(kwnames) != 0)) return PyObject_Vectorcall(c->otherwise, args, (size_t)n, kwnames);
    for (Py_ssize_t i = 0; i < n; ++i) {
        PyObject *const o = args[i];
        int             other = 0;
        switch (c->kinds[i]) {
        case 'n':
            if (PyLong_Check(o)) a[k++] = PyLong_AsUnsignedLongLongMask(o);
            else other = 1;
            break;
        case 'f':
            if (PyFloat_Check(o)) f = (float)PyFloat_AS_DOUBLE(o);
            else other = 1;
            break;
        case 'b':
            if (!held && is_item_array(o, c->item)) {
                if (PyObject_GetBuffer(o, &items, PyBUF_SIMPLE) != 0) return NULL;
                held   = 1;
                a[k++] = (W)(uintptr_t)items.buf;
            } else other = 1;
            break;
        default:
            if (o == Py_None) a[k++] = 0;
            else if (c->kinds[i] != 'p' && PyLong_Check(o)) a[k++] = PyLong_AsUnsignedLongLongMask(o);
            else if (c->kinds[i] == 's') other = 1;
            else if (tensor_address(o, &a[k++]) != 0) {
                if (held) PyBuffer_Release(&items);
                return NULL;
            }
        }
        if (other) {
            if (held) PyBuffer_Release(&items);
            return PyObject_Vectorcall(c->otherwise, args, (size_t)n, NULL);
        }
    }
    {
        const Function fn = c->function;
        Py_BEGIN_ALLOW_THREADS
        status = fn(f, a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17]);
        Py_END_ALLOW_THREADS
    }
    if (held) PyBuffer_Release(&items);
    return PyLong_FromLong(status);
}

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
    {"__vectorcalloffset__", T_PYSSIZET, offsetof(NativeCall, vectorcall), READONLY, NULL},
    {NULL, 0, 0, 0, NULL},
};

static void native_call_dealloc(PyObject *self)
{
    PyTypeObject *const type = Py_TYPE(self);
    Py_XDECREF(((NativeCall *)self)->otherwise);
    Py_XDECREF(((NativeCall *)self)->item);
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

static PyObject *native_call(PyObject *module, PyObject *args)
{
    PyObject   *address, *otherwise = NULL, *item = NULL;
    const char *kinds = NULL;
    (void)module;
    if (!PyArg_ParseTuple(args, "O|sOO", &address, &kinds, &otherwise, &item)) return NULL;
    const W at = PyLong_AsUnsignedLongLong(address);
    if (PyErr_Occurred()) return NULL;
    if (at == 0) {
        PyErr_SetString(PyExc_ValueError, "null function address");
        return NULL;
    }
    if (kinds != NULL) {
        size_t words = 0, floats = 0, batches = 0;
        for (const char *q = kinds; *q; ++q) {
            if (strchr("pasnfb", *q) == NULL) words = kMax + 1;
            *q == 'f' ? ++floats : ++words;
            batches += *q == 'b';
        }
        if (words > kMax || floats > 1 || batches > 1 || !*kinds || otherwise == NULL || !PyCallable_Check(otherwise) || (batches && item == NULL)) {
            PyErr_SetString(PyExc_ValueError, "not the parameters of a native call");
            return NULL;
        }
    }
    PyTypeObject *const type = (PyTypeObject *)s_type;
    NativeCall *const   c    = (NativeCall *)type->tp_alloc(type, 0);
    if (c == NULL) return NULL;
    c->vectorcall = kinds ? checked_vectorcall : native_call_vectorcall;
    c->function   = (Function)(uintptr_t)at;
    if (kinds) {
        c->arity = (Py_ssize_t)strlen(kinds);
        memcpy(c->kinds, kinds, (size_t)c->arity + 1);
        c->otherwise = Py_NewRef(otherwise);
        c->item      = Py_XNewRef(item);
    }
    return (PyObject *)c;
}

static PyMethodDef methods[] = {
    {"native_call", native_call, METH_VARARGS, "A callable for the exported function at an address."},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_pycall", "Calls of the C ABI without ctypes.", -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void)
{
    s_data_ptr  = PyUnicode_InternFromString("data_ptr");
    s_item_type = PyUnicode_InternFromString("_type_");
    s_type      = PyType_FromSpec(&native_call_spec);
    if (s_data_ptr == NULL || s_item_type == NULL || s_type == NULL) return NULL;
    return PyModule_Create(&module_def);
}
