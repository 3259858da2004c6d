/* The checks and the call of the two sampling entry points that a host makes once per decision, from Python.
 *
 * A lone decision keeps the GPU busy for 8 us; checking seven tensors in Python and a call through ctypes took the host 10.5.  Here
 * the same questions are asked of the same objects (is_cuda, dtype, is_contiguous(), shape, data_ptr()) from C, and the library
 * is called through its address: 4 x 8192 logits, call after call, 10.5 -> 9.6 us, 7.7 where the GPU
 * need not wait between two of them.
 * Whatever is not the plain case - another type, a missing tensor, a shape that does not fit - is answered with None and
 * nothing done: binding.py then makes the call itself and says what is wrong. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*verify_fn)(const float*, const float*, const int32_t*, const float*, int, int, int, float, float, int, float, int32_t*,
                         int32_t*, void*, size_t, void*);
typedef int (*sample_fn)(const float*, const float*, int, int, float, int32_t*, void*);

static verify_fn g_verify;
static sample_fn g_sample;
static PyObject *g_float32, *g_int32, *g_uint8;
static PyObject *s_is_cuda, *s_dtype, *s_is_contiguous, *s_shape, *s_data_ptr, *s_numel;

/* The address of a contiguous CUDA tensor of this type; its sizes in dims[n] (n < 0: not asked for).  0: something else. */
static int tensor(PyObject* t, PyObject* dtype, int n, Py_ssize_t* dims, void** address) {
    PyObject* v = PyObject_GetAttr(t, s_is_cuda);
    if (!v) return 0;
    Py_DECREF(v);
    if (v != Py_True) return 0;
    if (!(v = PyObject_GetAttr(t, s_dtype))) return 0;
    Py_DECREF(v);
    if (v != dtype) return 0;
    if (!(v = PyObject_CallMethodNoArgs(t, s_is_contiguous))) return 0;
    Py_DECREF(v);
    if (v != Py_True) return 0;
    if (n >= 0) {
        int fits;
        if (!(v = PyObject_GetAttr(t, s_shape))) return 0;
        fits = PyTuple_Check(v) && PyTuple_GET_SIZE(v) == n;
        for (int i = 0; fits && i < n; ++i) {
            dims[i] = PyLong_AsSsize_t(PyTuple_GET_ITEM(v, i));
            if (dims[i] < 0 || dims[i] > INT32_MAX) fits = 0;
        }
        Py_DECREF(v);
        if (!fits) return 0;
    }
    if (!(v = PyObject_CallMethodNoArgs(t, s_data_ptr))) return 0;
    *address = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}

static int number(PyObject* o, double* out) {
    if (!PyFloat_Check(o) && !PyLong_Check(o)) return 0;
    *out = PyFloat_AsDouble(o);
    return !PyErr_Occurred();
}

static PyObject* not_plain(void) {
    PyErr_Clear();
    Py_RETURN_NONE;
}

/* verify(target, draft, tokens, uniforms, n_accepted, next_token, workspace, temperature, lenience, top_k, top_p, stream) -> status */
static PyObject* verify(PyObject* self, PyObject* const* a, Py_ssize_t count) {
    void *target, *draft, *tokens, *uniforms, *accepted, *next, *workspace, *stream;
    Py_ssize_t t[3], q[3], x[2], u[2];
    double temperature, lenience, top_p;
    long top_k;
    size_t bytes;
    PyObject* v;
    int status;
    (void)self;
    if (count != 12 || !g_verify) return not_plain();
    if (!tensor(a[0], g_float32, 3, t, &target) || !tensor(a[1], g_float32, 3, q, &draft) || !tensor(a[2], g_int32, 2, x, &tokens) ||
        !tensor(a[3], g_float32, 2, u, &uniforms) || !tensor(a[4], g_int32, -1, NULL, &accepted) ||
        !tensor(a[5], g_int32, -1, NULL, &next) || !tensor(a[6], g_uint8, -1, NULL, &workspace))
        return not_plain();
    if (t[1] < 2 || q[0] != t[0] || q[1] != t[1] - 1 || q[2] != t[2] || x[0] != t[0] || x[1] != t[1] - 1 || u[0] != t[0] || u[1] != t[1])
        return not_plain();
    if (!number(a[7], &temperature) || !number(a[8], &lenience) || !PyLong_Check(a[9]) || !number(a[10], &top_p)) return not_plain();
    top_k = PyLong_AsLong(a[9]);
    if (PyErr_Occurred() || top_k < INT32_MIN || top_k > INT32_MAX) return not_plain();
    if (!(v = PyObject_CallMethodNoArgs(a[6], s_numel))) return not_plain();
    bytes = PyLong_AsSize_t(v);
    Py_DECREF(v);
    stream = PyLong_AsVoidPtr(a[11]);
    if (PyErr_Occurred()) return not_plain();
    Py_BEGIN_ALLOW_THREADS
    status = g_verify((const float*)target, (const float*)draft, (const int32_t*)tokens, (const float*)uniforms, (int)t[0], (int)t[1] - 1,
                      (int)t[2], (float)temperature, (float)lenience, (int)top_k, (float)top_p, (int32_t*)accepted, (int32_t*)next,
                      workspace, bytes, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

/* sample(logits, uniforms, temperature, tokens, stream) -> status */
static PyObject* sample(PyObject* self, PyObject* const* a, Py_ssize_t count) {
    void *logits, *uniforms, *tokens, *stream;
    Py_ssize_t l[2];
    double temperature;
    int status;
    (void)self;
    if (count != 5 || !g_sample) return not_plain();
    if (!tensor(a[0], g_float32, 2, l, &logits) || !tensor(a[1], g_float32, -1, NULL, &uniforms) || !number(a[2], &temperature) ||
        !tensor(a[3], g_int32, -1, NULL, &tokens))
        return not_plain();
    stream = PyLong_AsVoidPtr(a[4]);
    if (PyErr_Occurred()) return not_plain();
    Py_BEGIN_ALLOW_THREADS
    status = g_sample((const float*)logits, (const float*)uniforms, (int)l[0], (int)l[1], (float)temperature, (int32_t*)tokens, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(status);
}

/* bind(address of spec_verify_sample_truncated, of spec_sample, torch.float32, torch.int32, torch.uint8) */
static PyObject* bind(PyObject* self, PyObject* args) {
    PyObject *verify_at, *sample_at, *f, *i, *u;
    (void)self;
    if (!PyArg_ParseTuple(args, "OOOOO", &verify_at, &sample_at, &f, &i, &u)) return NULL;
    g_verify = (verify_fn)(uintptr_t)PyLong_AsVoidPtr(verify_at);
    g_sample = (sample_fn)(uintptr_t)PyLong_AsVoidPtr(sample_at);
    if (PyErr_Occurred()) return NULL;
    Py_INCREF(f);
    Py_INCREF(i);
    Py_INCREF(u);
    g_float32 = f;
    g_int32 = i;
    g_uint8 = u;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, NULL},
    {"verify", (PyCFunction)(void (*)(void))verify, METH_FASTCALL, NULL},
    {"sample", (PyCFunction)(void (*)(void))sample, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL},
};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_dtype = PyUnicode_InternFromString("dtype");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    s_shape = PyUnicode_InternFromString("shape");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    if (!s_is_cuda || !s_dtype || !s_is_contiguous || !s_shape || !s_data_ptr || !s_numel) return NULL;
    return PyModule_Create(&module);
}
