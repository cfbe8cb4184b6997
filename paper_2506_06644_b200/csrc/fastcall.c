/* Calls an entry point of libspark_b200.so from Python: marshalling only.
 *
 * call(address, arguments...) turns every argument into a 64-bit word -- None is a null pointer, an integer itself, a torch
 * tensor its device pointer (ValueError unless it is a contiguous CUDA tensor) -- appends the current CUDA stream and returns the
 * function's status.  Every parameter of the entry points called this way is a pointer or an integer, which the x86-64 calling
 * convention passes in full words, so one function type serves them all.  ctypes took 6 to 8 us for such a call, as long as the
 * smaller kernels run (64 x 1024 top-k: 10 us a call with 5.5 us on the GPU). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#define MAX_ARGS 32
typedef int (*entry_fn)(int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t,
                        int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t,
                        int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t);

static PyObject *s_is_cuda, *s_is_contiguous, *s_data_ptr;
static PyObject *get_device, *get_stream; /* torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream */

static int word(PyObject* v, int64_t* out) {
    if (v == Py_None) {
        *out = 0;
        return 0;
    }
    if (PyLong_Check(v)) {
        const unsigned long long u = PyLong_AsUnsignedLongLongMask(v);
        if (u == (unsigned long long)-1 && PyErr_Occurred()) return -1;
        *out = (int64_t)u;
        return 0;
    }
    PyObject* cuda = PyObject_GetAttr(v, s_is_cuda);
    if (cuda == NULL) { /* not a tensor: anything that is an integer */
        PyErr_Clear();
        PyObject* i = PyNumber_Index(v);
        if (i == NULL) return -1;
        const int rc = word(i, out);
        Py_DECREF(i);
        return rc;
    }
    const int on_gpu = cuda == Py_True;
    Py_DECREF(cuda);
    int contiguous = 0;
    if (on_gpu) {
        PyObject* c = PyObject_CallMethodNoArgs(v, s_is_contiguous);
        if (c == NULL) return -1;
        contiguous = c == Py_True;
        Py_DECREF(c);
    }
    if (!contiguous) {
        PyErr_SetString(PyExc_ValueError, "tensors passed to the library must be contiguous CUDA tensors");
        return -1;
    }
    PyObject* p = PyObject_CallMethodNoArgs(v, s_data_ptr);
    if (p == NULL) return -1;
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(p);
    Py_DECREF(p);
    return 0;
}

static PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    if (n < 1 || n > MAX_ARGS) {
        PyErr_SetString(PyExc_TypeError, "call(address, up to 31 arguments)");
        return NULL;
    }
    int64_t a[MAX_ARGS] = {0};
    const entry_fn fn = (entry_fn)(uintptr_t)PyLong_AsUnsignedLongLongMask(args[0]);
    for (Py_ssize_t i = 1; i < n; ++i)
        if (word(args[i], &a[i - 1]) != 0) return NULL;
    PyObject* dev = PyObject_CallNoArgs(get_device);
    if (dev == NULL) return NULL;
    PyObject* st = PyObject_CallOneArg(get_stream, dev);
    Py_DECREF(dev);
    if (st == NULL) return NULL;
    const int bad = word(st, &a[n - 1]);
    Py_DECREF(st);
    if (bad) return NULL;
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = fn(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17],
                a[18], a[19], a[20], a[21], a[22], a[23], a[24], a[25], a[26], a[27], a[28], a[29], a[30], a[31]);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

static PyObject* init(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    (void)self;
    if (n != 2) {
        PyErr_SetString(PyExc_TypeError, "init(get_device, get_stream)");
        return NULL;
    }
    Py_INCREF(args[0]);
    Py_INCREF(args[1]);
    Py_XSETREF(get_device, args[0]);
    Py_XSETREF(get_stream, args[1]);
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call an entry point on the current stream"},
                                {"init", (PyCFunction)(void (*)(void))init, METH_FASTCALL, "torch's functions for the current device and stream"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    return PyModule_Create(&module);
}
