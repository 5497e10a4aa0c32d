/* Calls of the C ABI from Python without ctypes' per-argument objects: bind(address) returns a builtin
 * that takes integers (device or host addresses, sizes, handles), None (a null pointer) and tuples
 * or lists of numbers (passed as int arrays that live for the call), and returns the status code.  What counts as an
 * integer is what the ctypes declarations take.
 * Marshalling only, like the ctypes declarations in binding.py, which are used where this module has not
 * been built; a decode call's share of host time goes from 1.0 to 0.3 us.
 *
 * Every parameter of the entry points is an integer or a pointer, so one prototype with as many
 * 64-bit integers as the longest of them serves them all (x86-64 and AArch64 calling conventions: the
 * first ones in registers, the rest in eight-byte stack slots; what a callee does not take it ignores).
 * The interpreter lock is released during the call (the host-buffer pass waits for the device). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

enum { kMaxArgs = 26, kMaxInts = 256 };
typedef uint64_t u;
typedef int (*entry)(u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u);

/* What ctypes makes of an int argument: anything with an index (numpy and torch integers too), its low bits. */
static int take_scalar(PyObject* x, u* out)
{
    if (PyLong_Check(x)) {
        *out = PyLong_AsUnsignedLongLongMask(x);
    } else {
        PyObject* v = PyNumber_Index(x);
        if (!v) return -1;
        *out = PyLong_AsUnsignedLongLongMask(v);
        Py_DECREF(v);
    }
    return PyErr_Occurred() ? -1 : 0;
}

/* What c_int makes of int(x). */
static int take_element(PyObject* x, int* out)
{
    PyObject* v = PyLong_Check(x) ? Py_NewRef(x) : PyNumber_Long(x);
    if (!v) return -1;
    *out = (int)(unsigned)PyLong_AsUnsignedLongMask(v);
    Py_DECREF(v);
    return PyErr_Occurred() ? -1 : 0;
}

static PyObject* invoke(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    u a[kMaxArgs] = {0};
    int stack[kMaxInts], *ints = stack;
    PyObject* seq[kMaxArgs] = {0};                     /* sequence arguments as tuples of this call's own */
    PyObject* result = NULL;
    Py_ssize_t used = 0;
    if (n > kMaxArgs) return PyErr_Format(PyExc_TypeError, "%zd arguments, at most %d", n, kMaxArgs);
    for (Py_ssize_t i = 0; i < n; ++i)
        if (PyTuple_Check(args[i]) || PyList_Check(args[i])) {
            seq[i] = PySequence_Tuple(args[i]);
            if (!seq[i]) goto done;
            used += PyTuple_GET_SIZE(seq[i]);
        }
    if (used > kMaxInts && !(ints = PyMem_Malloc(used * sizeof(int)))) {
        PyErr_NoMemory();
        goto done;
    }
    used = 0;
    for (Py_ssize_t i = 0; i < n; ++i) {
        if (seq[i]) {
            a[i] = (u)(uintptr_t)(ints + used);
            for (Py_ssize_t k = 0; k < PyTuple_GET_SIZE(seq[i]); ++k)
                if (take_element(PyTuple_GET_ITEM(seq[i], k), ints + used++) < 0) goto done;
        } else if (args[i] != Py_None && take_scalar(args[i], &a[i]) < 0) {
            goto done;
        }
    }
    const entry f = (entry)(uintptr_t)PyLong_AsUnsignedLongLong(self);
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17],
           a[18], a[19], a[20], a[21], a[22], a[23], a[24], a[25]);
    Py_END_ALLOW_THREADS
    result = PyLong_FromLong(rc);
done:
    for (Py_ssize_t i = 0; i < n; ++i) Py_XDECREF(seq[i]);
    if (ints != stack) PyMem_Free(ints);
    return result;
}

static PyMethodDef invoke_def = {"entry", (PyCFunction)(void (*)(void))invoke, METH_FASTCALL, "calls one entry point of the C ABI"};

static PyObject* bind(PyObject* module, PyObject* address)
{
    (void)module;
    if (!PyLong_Check(address)) return PyErr_Format(PyExc_TypeError, "an address");
    return PyCFunction_New(&invoke_def, address);
}

/* A decoding step is one short call per layer, and most of its host time is Python's: bind_decode(address) returns a builtin
 * that takes the tensors themselves, (params, q, k_cache, v_cache, n_valid, out, lse, ws, stream), and asks them for what
 * sablock_decode_attention wants to know. */
static PyObject *s_data_ptr, *s_shape, *s_numel;

static int take_method(PyObject* t, PyObject* name, u* out)
{
    if (t == Py_None) return 0;                        /* a null pointer */
    PyObject* v = PyObject_CallMethodNoArgs(t, name);
    if (!v) return -1;
    const int rc = take_scalar(v, out);
    Py_DECREF(v);
    return rc;
}

/* Extent `dim` of a tensor; it has `rank` dimensions (0: any number). */
static int take_extent(PyObject* t, Py_ssize_t rank, Py_ssize_t dim, u* out)
{
    PyObject* shape = PyObject_GetAttr(t, s_shape);
    if (!shape) return -1;
    int rc = -1;
    if (!PyTuple_Check(shape)) PyErr_SetString(PyExc_TypeError, "a tensor");
    else if (rank && PyTuple_GET_SIZE(shape) != rank) PyErr_Format(PyExc_ValueError, "%zd dimensions, not %zd", PyTuple_GET_SIZE(shape), rank);
    else if (dim >= PyTuple_GET_SIZE(shape)) PyErr_SetString(PyExc_IndexError, "too few dimensions");
    else rc = take_scalar(PyTuple_GET_ITEM(shape, dim), out);
    Py_DECREF(shape);
    return rc;
}

static PyObject* invoke_decode(PyObject* self, PyObject* const* args, Py_ssize_t n)
{
    typedef int (*decode)(u, u, u, u, u, u, u, u, u, u, u, u);
    u p = 0, q = 0, k = 0, v = 0, valid = 0, out = 0, lse = 0, ws = 0, ws_bytes = 0, stream = 0, n_prob = 0, n_rows = 0;
    if (n != 9) return PyErr_Format(PyExc_TypeError, "%zd arguments, not 9", n);
    if (take_scalar(args[0], &p) < 0 || take_extent(args[1], 3, 0, &n_prob) < 0 || take_extent(args[2], 0, 1, &n_rows) < 0 ||
        take_method(args[1], s_data_ptr, &q) < 0 || take_method(args[2], s_data_ptr, &k) < 0 || take_method(args[3], s_data_ptr, &v) < 0 ||
        take_method(args[4], s_data_ptr, &valid) < 0 || take_method(args[5], s_data_ptr, &out) < 0 || take_method(args[6], s_data_ptr, &lse) < 0 ||
        take_method(args[7], s_data_ptr, &ws) < 0 || take_method(args[7], s_numel, &ws_bytes) < 0 || take_scalar(args[8], &stream) < 0)
        return NULL;
    const decode f = (decode)(uintptr_t)PyLong_AsUnsignedLongLong(self);
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f(p, n_prob, q, k, v, n_rows, valid, out, lse, ws, ws_bytes, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

static PyMethodDef invoke_decode_def = {"decode", (PyCFunction)(void (*)(void))invoke_decode, METH_FASTCALL, "calls sablock_decode_attention"};

static PyObject* bind_decode(PyObject* module, PyObject* address)
{
    (void)module;
    if (!PyLong_Check(address)) return PyErr_Format(PyExc_TypeError, "an address");
    return PyCFunction_New(&invoke_decode_def, address);
}

static PyMethodDef methods[] = {{"bind_decode", bind_decode, METH_O, "bind_decode(address): sablock_decode_attention for tensors"},
                                {"bind", bind, METH_O, "bind(address): a callable for the entry point at that address"}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__fastcall(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_numel = PyUnicode_InternFromString("numel");
    return s_data_ptr && s_shape && s_numel ? PyModule_Create(&module) : NULL;
}
