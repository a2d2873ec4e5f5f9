/* The calls of the binding that enqueue work, without ctypes: a foreign call with five to nine arguments costs the host about a microsecond there, as much as
 * half of a launch, and a product of a few microseconds is bound by what the host pays for it: 256 x 256 x 256 in a row of calls 3.97 us through ctypes, 3.07 this way.
 *
 * Every function returns the library's status, or -1 if an argument is anything but a plain int (a float where the C function takes one; None for a null
 * pointer): the caller then goes through ctypes, which converts or refuses it as ever.  The interpreter's lock is released around the call, as ctypes does. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

static int (*matmul)(void*, const void*, const void*, void*, void*);
static int (*addmm)(void*, const void*, const void*, const void*, int, float, float, void*, void*);
static int (*strided)(void*, const void*, int64_t, const void*, int64_t, void*, int64_t, int64_t, void*);

static int pointer(PyObject* o, void** out)
{
    if (o == Py_None) { *out = NULL; return 1; }
    if (!PyLong_CheckExact(o)) return 0;
    *out = (void*)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
    return 1;
}
static int integer(PyObject* o, long long* out)
{
    int overflow = 0;
    if (!PyLong_CheckExact(o)) return 0;
    *out = PyLong_AsLongLongAndOverflow(o, &overflow);
    return !overflow;
}
static int number(PyObject* o, float* out)
{
    if (PyFloat_CheckExact(o)) *out = (float)PyFloat_AS_DOUBLE(o);
    else return 0;
    return 1;
}

static PyObject* py_bind(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void* p[3];
    if (n != 3 || !pointer(a[0], &p[0]) || !pointer(a[1], &p[1]) || !pointer(a[2], &p[2])) {
        PyErr_SetString(PyExc_TypeError, "three addresses are wanted");
        return NULL;
    }
    matmul = (int (*)(void*, const void*, const void*, void*, void*))p[0];
    addmm = (int (*)(void*, const void*, const void*, const void*, int, float, float, void*, void*))p[1];
    strided = (int (*)(void*, const void*, int64_t, const void*, int64_t, void*, int64_t, int64_t, void*))p[2];
    Py_RETURN_NONE;
}

static PyObject* py_matmul(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *plan, *A, *B, *C, *stream;
    int r;
    if (!matmul || n != 5 || !pointer(a[0], &plan) || !pointer(a[1], &A) || !pointer(a[2], &B) || !pointer(a[3], &C) || !pointer(a[4], &stream)) return PyLong_FromLong(-1);
    Py_BEGIN_ALLOW_THREADS
    r = matmul(plan, A, B, C, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(r);
}

static PyObject* py_addmm(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *plan, *A, *B, *D, *C, *stream;
    long long vector;
    float alpha, beta;
    int r;
    if (!addmm || n != 9 || !pointer(a[0], &plan) || !pointer(a[1], &A) || !pointer(a[2], &B) || !pointer(a[3], &D) || !integer(a[4], &vector) ||
        !number(a[5], &alpha) || !number(a[6], &beta) || !pointer(a[7], &C) || !pointer(a[8], &stream)) return PyLong_FromLong(-1);
    Py_BEGIN_ALLOW_THREADS
    r = addmm(plan, A, B, D, vector != 0, alpha, beta, C, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(r);
}

static PyObject* py_strided(PyObject* self, PyObject* const* a, Py_ssize_t n)
{
    void *plan, *A, *B, *C, *stream;
    long long sa, sb, sc, batch;
    int r;
    if (!strided || n != 9 || !pointer(a[0], &plan) || !pointer(a[1], &A) || !integer(a[2], &sa) || !pointer(a[3], &B) || !integer(a[4], &sb) ||
        !pointer(a[5], &C) || !integer(a[6], &sc) || !integer(a[7], &batch) || !pointer(a[8], &stream)) return PyLong_FromLong(-1);
    Py_BEGIN_ALLOW_THREADS
    r = strided(plan, A, sa, B, sb, C, sc, batch, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(r);
}

static PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))py_bind, METH_FASTCALL, "addresses of adapt_matmul, adapt_addmm, adapt_matmul_strided_batch"},
    {"matmul", (PyCFunction)(void (*)(void))py_matmul, METH_FASTCALL, "adapt_matmul"},
    {"addmm", (PyCFunction)(void (*)(void))py_addmm, METH_FASTCALL, "adapt_addmm"},
    {"strided", (PyCFunction)(void (*)(void))py_strided, METH_FASTCALL, "adapt_matmul_strided_batch"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods};
PyMODINIT_FUNC PyInit__fastcall(void) { return PyModule_Create(&module); }
