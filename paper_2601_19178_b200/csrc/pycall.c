/*
 * CPython helper of binding.py: marshals the arguments of the calls a request makes.  A decode call of a few users takes the
 * GPU about 6 us; taking two array addresses, two tensor addresses and going through ctypes took Python another 4.
 * Marshalling only: the call itself is the C-ABI function whose address is passed in.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

static PyObject *s_data_ptr, *s_is_contiguous;

/* Address and length of a C-contiguous host array of whole numbers of `size` bytes; 0 if `o` is something else. */
static int host_array(PyObject* o, Py_ssize_t size, Py_buffer* b)
{
    if (PyObject_GetBuffer(o, b, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT) != 0) {
        PyErr_Clear();
        return 0;
    }
    const char* f = b->format ? b->format : "B";
    if (b->ndim == 1 && b->itemsize == size && (f[0] == 'l' || f[0] == 'i' || f[0] == 'q') && f[1] == 0) return 1;
    PyBuffer_Release(b);
    return 0;
}

/* Address of a contiguous tensor; 0 if `o` is something else (an exception of the tensor's own stays set). */
static int tensor_address(PyObject* o, void** p)
{
    PyObject* c = PyObject_CallMethodNoArgs(o, s_is_contiguous);
    if (!c) {
        if (PyErr_ExceptionMatches(PyExc_AttributeError)) PyErr_Clear();
        return 0;
    }
    const int yes = c == Py_True;
    Py_DECREF(c);
    if (!yes) return 0;
    PyObject* a = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!a) return 0;
    *p = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
    return !PyErr_Occurred();
}

typedef int32_t (*attend_fn)(void*, int32_t, const void*, const void*, const void*, void*, void*);
typedef int32_t (*attend_visible_fn)(void*, int32_t, const void*, const void*, const void*, const void*, void*, void*);

/* attend(function address, context, users int64[n], q_off int32[n + 1], vis tensor | None, queries, out, stream):
 * the status of the call, or None if an argument is not of the plain kind (binding.py then converts it). */
static PyObject* attend(PyObject* self, PyObject* const* args, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 8) {
        PyErr_SetString(PyExc_TypeError, "attend takes 8 arguments");
        return NULL;
    }
    void* fn = PyLong_AsVoidPtr(args[0]);
    void* ctx = PyLong_AsVoidPtr(args[1]);
    void* stream = PyLong_AsVoidPtr(args[7]);
    if (PyErr_Occurred()) return NULL;
    Py_buffer users, q_off;
    if (!host_array(args[2], 8, &users)) Py_RETURN_NONE;
    if (!host_array(args[3], 4, &q_off)) {
        PyBuffer_Release(&users);
        Py_RETURN_NONE;
    }
    const Py_ssize_t n = users.len / 8;
    void *vis = NULL, *q = NULL, *out = NULL;
    const int with_vis = args[4] != Py_None;
    int32_t status = 0;
    const int plain = q_off.len / 4 == n + 1 && n <= INT32_MAX && (!with_vis || tensor_address(args[4], &vis)) &&
                      tensor_address(args[5], &q) && tensor_address(args[6], &out);
    if (plain) {
        Py_BEGIN_ALLOW_THREADS;
        status = with_vis ? ((attend_visible_fn)fn)(ctx, (int32_t)n, users.buf, q_off.buf, vis, q, out, stream)
                          : ((attend_fn)fn)(ctx, (int32_t)n, users.buf, q_off.buf, q, out, stream);
        Py_END_ALLOW_THREADS;
    }
    PyBuffer_Release(&users);
    PyBuffer_Release(&q_off);
    if (PyErr_Occurred()) return NULL;
    if (!plain) Py_RETURN_NONE;
    return PyLong_FromLong(status);
}

typedef int32_t (*append_fn)(void*, int64_t, int32_t, const void*, const void*, const void*, const void*, int32_t, void*);

/* append(function address, context, user, L_new, idx_K, idx_V, user_K, user_V, d_user, stream): as attend, every array a
 * contiguous tensor. */
static PyObject* append(PyObject* self, PyObject* const* args, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 10) {
        PyErr_SetString(PyExc_TypeError, "append takes 10 arguments");
        return NULL;
    }
    void* fn = PyLong_AsVoidPtr(args[0]);
    void* ctx = PyLong_AsVoidPtr(args[1]);
    const long long user = PyLong_AsLongLong(args[2]);
    const long L_new = PyLong_AsLong(args[3]), d_user = PyLong_AsLong(args[8]);
    void* stream = PyLong_AsVoidPtr(args[9]);
    if (PyErr_Occurred()) return NULL;
    void* p[4];
    for (int i = 0; i < 4; ++i)
        if (!tensor_address(args[4 + i], &p[i])) {
            if (PyErr_Occurred()) return NULL;
            Py_RETURN_NONE;
        }
    if (L_new != (int32_t)L_new || d_user != (int32_t)d_user) Py_RETURN_NONE;
    int32_t status;
    Py_BEGIN_ALLOW_THREADS;
    status = ((append_fn)fn)(ctx, user, (int32_t)L_new, p[0], p[1], p[2], p[3], (int32_t)d_user, stream);
    Py_END_ALLOW_THREADS;
    return PyLong_FromLong(status);
}

/* Like tensor_address, with None for a null pointer. */
static int optional_address(PyObject* o, void** p)
{
    *p = NULL;
    return o == Py_None || tensor_address(o, p);
}

static int whole_numbers(PyObject* const* args, int n, int32_t* v)
{
    for (int i = 0; i < n; ++i) {
        const long x = PyLong_AsLong(args[i]);
        if ((x == -1 && PyErr_Occurred()) || x != (int32_t)x) return 0;
        v[i] = (int32_t)x;
    }
    return 1;
}

typedef int32_t (*project_fn)(int32_t, int32_t, int32_t, int32_t, int32_t, const void*, const void*, const void*, void*, void*);
typedef int32_t (*route_fn)(int32_t, int32_t, int32_t, int32_t, int32_t, const void*, const void*, const void*, void*, int32_t,
                            void*);

/* prefill(function address, five whole numbers, x, W, bias | None, output, variant | None, stream): ckv_project without a
 * variant, ckv_route with one; None as above. */
static PyObject* prefill(PyObject* self, PyObject* const* args, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 12) {
        PyErr_SetString(PyExc_TypeError, "prefill takes 12 arguments");
        return NULL;
    }
    void* fn = PyLong_AsVoidPtr(args[0]);
    void* stream = PyLong_AsVoidPtr(args[11]);
    if (PyErr_Occurred()) return NULL;
    int32_t v[5], variant = 0, status;
    void* p[4];
    const int route = args[10] != Py_None;
    if (!whole_numbers(args + 1, 5, v) || (route && !whole_numbers(args + 10, 1, &variant)) || !tensor_address(args[6], &p[0]) ||
        !tensor_address(args[7], &p[1]) || !optional_address(args[8], &p[2]) || !tensor_address(args[9], &p[3])) {
        if (PyErr_Occurred()) return NULL;
        Py_RETURN_NONE;
    }
    Py_BEGIN_ALLOW_THREADS;
    status = route ? ((route_fn)fn)(v[0], v[1], v[2], v[3], v[4], p[0], p[1], p[2], p[3], variant, stream)
                   : ((project_fn)fn)(v[0], v[1], v[2], v[3], v[4], p[0], p[1], p[2], p[3], stream);
    Py_END_ALLOW_THREADS;
    return PyLong_FromLong(status);
}

typedef int32_t (*put_fn)(void*, int32_t, const void*, const void*, const void*, const void*, const void*, const void*, int32_t,
                          void*);

/* put(function address, context, users int64[n], hist_off int64[n + 1], idx_K, idx_V, user_K, user_V (tensor | None each),
 * d_user, stream): as attend. */
static PyObject* put(PyObject* self, PyObject* const* args, Py_ssize_t n_args)
{
    (void)self;
    if (n_args != 10) {
        PyErr_SetString(PyExc_TypeError, "put takes 10 arguments");
        return NULL;
    }
    void* fn = PyLong_AsVoidPtr(args[0]);
    void* ctx = PyLong_AsVoidPtr(args[1]);
    void* stream = PyLong_AsVoidPtr(args[9]);
    if (PyErr_Occurred()) return NULL;
    int32_t d_user, status = 0;
    void* p[4];
    int plain = whole_numbers(args + 8, 1, &d_user);
    for (int i = 0; plain && i < 4; ++i) plain = optional_address(args[4 + i], &p[i]);
    if (PyErr_Occurred()) return NULL;
    Py_buffer users, off;
    if (!plain || !host_array(args[2], 8, &users)) Py_RETURN_NONE;
    if (!host_array(args[3], 8, &off)) {
        PyBuffer_Release(&users);
        Py_RETURN_NONE;
    }
    const Py_ssize_t n = users.len / 8;
    plain = off.len / 8 == n + 1 && n <= INT32_MAX;
    if (plain) {
        Py_BEGIN_ALLOW_THREADS;
        status = ((put_fn)fn)(ctx, (int32_t)n, users.buf, off.buf, p[0], p[1], p[2], p[3], d_user, stream);
        Py_END_ALLOW_THREADS;
    }
    PyBuffer_Release(&users);
    PyBuffer_Release(&off);
    if (!plain) Py_RETURN_NONE;
    return PyLong_FromLong(status);
}

static PyMethodDef methods[] = {{"attend", (PyCFunction)(void (*)(void))attend, METH_FASTCALL, "one decode call"},
                                {"append", (PyCFunction)(void (*)(void))append, METH_FASTCALL, "one append"},
                                {"put", (PyCFunction)(void (*)(void))put, METH_FASTCALL, "one put of several users"},
                                {"prefill", (PyCFunction)(void (*)(void))prefill, METH_FASTCALL, "one router or projection call"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void)
{
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
    return s_data_ptr && s_is_contiguous ? PyModule_Create(&module) : NULL;
}
