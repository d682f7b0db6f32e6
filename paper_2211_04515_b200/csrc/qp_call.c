/* Call path from Python into the C ABI (the module _qpcall, built beside libquantpipe.so).
 *
 * A small-tensor call is bound by the host: the receiver of one ViT-Base image spends under 3 us on
 * the GPU, and through ctypes (argument objects for 9 to 14 parameters, five method calls per tensor)
 * the call took 14 us.  Here the arguments go from the vectorcall array straight into registers:
 * about 1 us per call beside the launch itself.
 *
 *   bind(address, kinds)    makes the function at `address` callable; returns its number for call / call64.  kinds: a
 *                           letter per parameter,
 *                             i  an integer: int, or an object that can stand for one (a numpy integer, a tensor of one
 *                                integer); passed as its low 64 bits
 *                             p  a buffer: a tensor (its data_ptr()) or None (NULL)
 *                             a  an address: an int, a tensor or None
 *   call(number, *args)     calls the function; returns its int32 status
 *   call64(number, *args)   the same for functions that return uint64
 *   tensor_in(x)            (numel, dtype code) of a contiguous CUDA tensor; AssertionError for others,
 *                           dtype code -1 for a dtype the library does not take
 *   setup(float32, bfloat16)  the two dtype objects that have a code; empties the table of bound functions
 *
 * A tensor of one integer has an address and a value, so which of them is meant has to come from the parameter.
 * Every parameter of the functions called this way is an integer or a pointer, which the 64-bit C
 * calling conventions pass alike, so one function type per argument count covers them all.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#define MAX_ARGS 16

static PyObject *s_data_ptr, *s_numel, *s_is_contiguous, *s_is_cuda, *s_dtype;
static PyObject *t_float32, *t_bfloat16;

#define MAX_FUNCS 64
static struct { uint64_t f; Py_ssize_t n; char kinds[MAX_ARGS + 1]; } funcs[MAX_FUNCS];
static int n_funcs;

static int word_of(PyObject* o, char kind, uint64_t* out)
{
    if (PyLong_Check(o) && kind != 'p') {                /* bool is an int */
        *out = PyLong_AsUnsignedLongLongMask(o);
    } else if (o == Py_None && kind != 'i') {
        *out = 0;
    } else {
        PyObject* p = kind == 'i' ? PyNumber_Index(o) : PyObject_CallMethodNoArgs(o, s_data_ptr);
        if (!p) return -1;
        *out = PyLong_AsUnsignedLongLongMask(p);
        Py_DECREF(p);
    }
    return (*out == (uint64_t)-1 && PyErr_Occurred()) ? -1 : 0;
}

typedef uint64_t u;
#define A1 a[0]
#define A4 a[0], a[1], a[2], a[3]
#define A8 A4, a[4], a[5], a[6], a[7]
#define A12 A8, a[8], a[9], a[10], a[11]

static u jump(u f, const u* a, Py_ssize_t n)
{
    switch (n) {
        case 1: return ((u(*)(u))f)(A1);
        case 2: return ((u(*)(u, u))f)(A1, a[1]);
        case 3: return ((u(*)(u, u, u))f)(A1, a[1], a[2]);
        case 4: return ((u(*)(u, u, u, u))f)(A4);
        case 5: return ((u(*)(u, u, u, u, u))f)(A4, a[4]);
        case 6: return ((u(*)(u, u, u, u, u, u))f)(A4, a[4], a[5]);
        case 7: return ((u(*)(u, u, u, u, u, u, u))f)(A4, a[4], a[5], a[6]);
        case 8: return ((u(*)(u, u, u, u, u, u, u, u))f)(A8);
        case 9: return ((u(*)(u, u, u, u, u, u, u, u, u))f)(A8, a[8]);
        case 10: return ((u(*)(u, u, u, u, u, u, u, u, u, u))f)(A8, a[8], a[9]);
        case 11: return ((u(*)(u, u, u, u, u, u, u, u, u, u, u))f)(A8, a[8], a[9], a[10]);
        case 12: return ((u(*)(u, u, u, u, u, u, u, u, u, u, u, u))f)(A12);
        case 13: return ((u(*)(u, u, u, u, u, u, u, u, u, u, u, u, u))f)(A12, a[12]);
        case 14: return ((u(*)(u, u, u, u, u, u, u, u, u, u, u, u, u, u))f)(A12, a[12], a[13]);
        case 15: return ((u(*)(u, u, u, u, u, u, u, u, u, u, u, u, u, u, u))f)(A12, a[12], a[13], a[14]);
        default: return ((u(*)(u, u, u, u, u, u, u, u, u, u, u, u, u, u, u, u))f)(A12, a[12], a[13], a[14], a[15]);
    }
}

static int invoke(PyObject* const* args, Py_ssize_t n, u* r)
{
    u a[MAX_ARGS];
    const long i = n > 0 ? PyLong_AsLong(args[0]) : -1;
    if (i == -1 && PyErr_Occurred()) return -1;
    if (i < 0 || i >= n_funcs || n - 1 != funcs[i].n) {
        PyErr_SetString(PyExc_TypeError, "the number of a bound function and its arguments");
        return -1;
    }
    for (Py_ssize_t k = 1; k < n; ++k)
        if (word_of(args[k], funcs[i].kinds[k - 1], &a[k - 1])) return -1;
    Py_BEGIN_ALLOW_THREADS                               /* a launch may wait for room in the queue */
    *r = jump(funcs[i].f, a, n - 1);
    Py_END_ALLOW_THREADS
    return 0;
}

static PyObject* py_bind(PyObject* m, PyObject* args)
{
    unsigned long long f;
    const char* kinds;
    Py_ssize_t n;
    (void)m;
    if (!PyArg_ParseTuple(args, "Ks#", &f, &kinds, &n)) return NULL;
    if (!f || n < 1 || n > MAX_ARGS || strspn(kinds, "ipa") != (size_t)n || n_funcs == MAX_FUNCS) {
        PyErr_SetString(PyExc_ValueError, "an address, 1 to 16 kinds of i, p and a, and room in the table");
        return NULL;
    }
    funcs[n_funcs].f = f;
    funcs[n_funcs].n = n;
    memcpy(funcs[n_funcs].kinds, kinds, (size_t)n + 1);
    return PyLong_FromLong(n_funcs++);
}

static PyObject* py_call(PyObject* m, PyObject* const* args, Py_ssize_t n)
{
    u r;
    (void)m;
    return invoke(args, n, &r) ? NULL : PyLong_FromLong((int32_t)(uint32_t)r);
}

static PyObject* py_call64(PyObject* m, PyObject* const* args, Py_ssize_t n)
{
    u r;
    (void)m;
    return invoke(args, n, &r) ? NULL : PyLong_FromUnsignedLongLong(r);
}

static int is_true(PyObject* o)                          /* steals the reference; -1 on an error */
{
    if (!o) return -1;
    const int r = PyObject_IsTrue(o);
    Py_DECREF(o);
    return r;
}

static PyObject* py_tensor_in(PyObject* m, PyObject* x)
{
    (void)m;
    const int cuda = is_true(PyObject_GetAttr(x, s_is_cuda));
    if (cuda < 0) return NULL;
    const int contiguous = is_true(PyObject_CallMethodNoArgs(x, s_is_contiguous));
    if (contiguous < 0) return NULL;
    if (!cuda || !contiguous) {
        PyErr_SetString(PyExc_AssertionError, "a contiguous CUDA tensor is required");
        return NULL;
    }
    PyObject* dtype = PyObject_GetAttr(x, s_dtype);
    if (!dtype) return NULL;
    const long code = dtype == t_float32 ? 0 : dtype == t_bfloat16 ? 1 : -1;
    Py_DECREF(dtype);
    PyObject* numel = PyObject_CallMethodNoArgs(x, s_numel);
    if (!numel) return NULL;
    PyObject* c = PyLong_FromLong(code);
    PyObject* r = c ? PyTuple_New(2) : NULL;
    if (!r) { Py_DECREF(numel); Py_XDECREF(c); return NULL; }
    PyTuple_SET_ITEM(r, 0, numel);
    PyTuple_SET_ITEM(r, 1, c);
    return r;
}

static PyObject* py_setup(PyObject* m, PyObject* args)
{
    PyObject *f, *b;
    (void)m;
    if (!PyArg_ParseTuple(args, "OO", &f, &b)) return NULL;
    Py_INCREF(f);
    Py_INCREF(b);
    Py_XSETREF(t_float32, f);
    Py_XSETREF(t_bfloat16, b);
    n_funcs = 0;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", py_bind, METH_VARARGS, "bind(address, kinds) -> number"},
    {"call", (PyCFunction)(void (*)(void))py_call, METH_FASTCALL, "call(number, *args) -> int32 status"},
    {"call64", (PyCFunction)(void (*)(void))py_call64, METH_FASTCALL, "call64(number, *args) -> uint64"},
    {"tensor_in", py_tensor_in, METH_O, "tensor_in(x) -> (numel, dtype code)"},
    {"setup", py_setup, METH_VARARGS, "setup(float32, bfloat16)"},
    {NULL, NULL, 0, NULL},
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_qpcall", "Calls into the quantpipe C ABI.", -1, methods,
                                    NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__qpcall(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_dtype = PyUnicode_InternFromString("dtype");
    if (!s_data_ptr || !s_numel || !s_is_contiguous || !s_is_cuda || !s_dtype) return NULL;
    return PyModule_Create(&module);
}
