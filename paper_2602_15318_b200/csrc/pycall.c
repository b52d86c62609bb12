/* Argument marshalling of the Python binding in C.  A decoder's step is dozens of short calls (row
 * movers of 1-2 us of GPU time each), so what the interpreter spends per call bounds it: converting the
 * arguments through ctypes and asking torch for a Stream object took 8 us of an 11 us append.
 *
 * bind(address, signature, name, on_error) -> callable.  One signature letter per C argument:
 *   c  the context: attribute `address` (an int)
 *   t  a tensor (its data_ptr()) or None (NULL)
 *   i  an int, passed as int32
 *   l  a sequence of ints -> int32 array, valid during the call;  L  the same, or None -> NULL
 *   s  a stream: None (the current one), an object with `cuda_stream`, an int handle, or one in a ctypes.c_void_p
 * Every argument is an integer or a pointer, i.e. one 64-bit slot of the calling convention.  A non-zero
 * status calls on_error(status, name), which raises.  The interpreter lock is released during the
 * call.  set_stream_functions(get_device, get_raw_stream) says how to ask for the current stream, if not torch. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#define MAX_ARGS 16
#define STACK_INTS 256

typedef struct {
    void* fn;
    int n;
    char sig[MAX_ARGS + 1];
    PyObject* name;
    PyObject* on_error;
} Bound;

/* pycall_torch.cpp */
int sparrow_tensor_address(PyObject* o, int64_t* out);
int sparrow_current_stream(int64_t* out);

static PyObject *s_address, *s_data_ptr, *s_cuda_stream, *s_value, *g_void_p, *g_get_device, *g_get_raw_stream;

static const char kCapsule[] = "sparrow.bound";

static void bound_free(PyObject* cap)
{
    Bound* b = (Bound*)PyCapsule_GetPointer(cap, kCapsule);
    if (!b) { PyErr_Clear(); return; }
    Py_XDECREF(b->name);
    Py_XDECREF(b->on_error);
    PyMem_Free(b);
}

/* An int object's value as a 64-bit slot (pointers included). */
static int as_slot(PyObject* o, int64_t* out)
{
    PyObject* i = PyNumber_Index(o);
    if (!i) return -1;
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(i);
    Py_DECREF(i);
    return PyErr_Occurred() ? -1 : 0;
}

static int stolen_slot(PyObject* o, int64_t* out)      /* the same, dropping the reference */
{
    if (!o) return -1;
    const int r = as_slot(o, out);
    Py_DECREF(o);
    return r;
}

static int stream_slot(PyObject* o, int64_t* out)
{
    if (o == Py_None) {
        if (!g_get_device && sparrow_current_stream(out)) return 0;
        if (!g_get_device || !g_get_raw_stream) { PyErr_SetString(PyExc_RuntimeError, "no current stream"); return -1; }
        PyObject* dev = PyObject_CallNoArgs(g_get_device);
        if (!dev) return -1;
        PyObject* st = PyObject_CallOneArg(g_get_raw_stream, dev);
        Py_DECREF(dev);
        return stolen_slot(st, out);
    }
    if (PyLong_Check(o)) return as_slot(o, out);
    const int is_handle = PyObject_IsInstance(o, g_void_p);
    if (is_handle < 0) return -1;
    if (!is_handle) return stolen_slot(PyObject_GetAttr(o, s_cuda_stream), out);
    PyObject* v = PyObject_GetAttr(o, s_value);
    if (v != Py_None) return stolen_slot(v, out);
    Py_DECREF(v);                                               /* (a null handle: the default stream) */
    return 0;
}

/* Sequence of ints -> int32 array in *buf (STACK_INTS entries) or on the heap (*heap). */
static int int_array(PyObject* o, int32_t* buf, int32_t** heap, int64_t* out)
{
    PyObject* seq = PySequence_Fast(o, "expected a sequence of ints");
    if (!seq) return -1;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    int32_t* dst = buf;
    if (n > STACK_INTS) {
        dst = *heap = (int32_t*)PyMem_Malloc((size_t)n * sizeof(int32_t));
        if (!dst) { Py_DECREF(seq); PyErr_NoMemory(); return -1; }
    }
    for (Py_ssize_t k = 0; k < n; ++k) {
        PyObject* item = PySequence_Fast_GET_ITEM(seq, k);      /* borrowed */
        int64_t v;
        if (PyLong_Check(item) ? as_slot(item, &v) : stolen_slot(PyNumber_Long(item), &v)) { Py_DECREF(seq); return -1; }
        dst[k] = (int32_t)v;
    }
    Py_DECREF(seq);
    *out = (int64_t)(intptr_t)dst;
    return 0;
}

static PyObject* bound_call(PyObject* self, PyObject* const* args, Py_ssize_t nargs)
{
    Bound* b = (Bound*)PyCapsule_GetPointer(self, kCapsule);
    if (!b) return NULL;
    if (nargs != b->n) return PyErr_Format(PyExc_TypeError, "%U takes %d arguments (%zd given)", b->name, b->n, nargs);
    int64_t a[MAX_ARGS] = {0};
    int32_t ints[2][STACK_INTS];
    int32_t* heap[2] = {NULL, NULL};
    int n_arrays = 0, bad = 0;
    for (int k = 0; k < b->n && !bad; ++k) {
        PyObject* o = args[k];
        switch (b->sig[k]) {
            case 'c': bad = stolen_slot(PyObject_GetAttr(o, s_address), &a[k]); break;
            case 't':
                if (o != Py_None && !sparrow_tensor_address(o, &a[k])) bad = stolen_slot(PyObject_CallMethodNoArgs(o, s_data_ptr), &a[k]);
                break;
            case 'i': bad = as_slot(o, &a[k]); a[k] = (int64_t)(int32_t)a[k]; break;
            case 'L': if (o == Py_None) break; /* fall through */
            case 'l': bad = int_array(o, ints[n_arrays], &heap[n_arrays], &a[k]); ++n_arrays; break;
            default: bad = stream_slot(o, &a[k]); break;
        }
    }
    int status = 0;
    if (!bad) {
        typedef int (*Fn)(int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t, int64_t,
                          int64_t, int64_t, int64_t, int64_t);
        Py_BEGIN_ALLOW_THREADS
        status = ((Fn)b->fn)(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15]);
        Py_END_ALLOW_THREADS
    }
    PyMem_Free(heap[0]);
    PyMem_Free(heap[1]);
    if (bad) return NULL;
    if (status != 0) return PyObject_CallFunction(b->on_error, "iO", status, b->name);
    Py_RETURN_NONE;
}

static PyMethodDef bound_def = {"bound", (PyCFunction)(void (*)(void))bound_call, METH_FASTCALL, NULL};

static PyObject* py_bind(PyObject* self, PyObject* args)
{
    unsigned long long address;
    const char* sig;
    PyObject *name, *on_error;
    (void)self;
    if (!PyArg_ParseTuple(args, "KsUO", &address, &sig, &name, &on_error)) return NULL;
    const size_t n = strlen(sig);
    int arrays = 0;
    for (size_t k = 0; k < n; ++k) arrays += sig[k] == 'l' || sig[k] == 'L';
    if (!address || n > MAX_ARGS || arrays > 2 || strspn(sig, "ctilLs") != n) return PyErr_Format(PyExc_ValueError, "bad signature %s", sig);
    Bound* b = (Bound*)PyMem_Calloc(1, sizeof *b);
    if (!b) return PyErr_NoMemory();
    b->fn = (void*)(uintptr_t)address;
    b->n = (int)n;
    memcpy(b->sig, sig, n);
    b->name = Py_NewRef(name);
    b->on_error = Py_NewRef(on_error);
    PyObject* cap = PyCapsule_New(b, kCapsule, bound_free);
    if (!cap) { Py_DECREF(name); Py_DECREF(on_error); PyMem_Free(b); return NULL; }
    PyObject* f = PyCFunction_NewEx(&bound_def, cap, NULL);
    Py_DECREF(cap);
    return f;
}

static PyObject* py_set_stream_functions(PyObject* self, PyObject* args)
{
    PyObject *dev, *raw;
    (void)self;
    if (!PyArg_ParseTuple(args, "OO", &dev, &raw)) return NULL;
    Py_XSETREF(g_get_device, dev == Py_None ? NULL : Py_NewRef(dev));
    Py_XSETREF(g_get_raw_stream, raw == Py_None ? NULL : Py_NewRef(raw));
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"bind", py_bind, METH_VARARGS, "bind(address, signature, name, on_error) -> callable"},
                                {"set_stream_functions", py_set_stream_functions, METH_VARARGS, "set_stream_functions(get_device, get_raw_stream)"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void)
{
    s_address = PyUnicode_InternFromString("address");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_value = PyUnicode_InternFromString("value");
    PyObject* ctypes = PyImport_ImportModule("ctypes");
    g_void_p = ctypes ? PyObject_GetAttrString(ctypes, "c_void_p") : NULL;
    Py_XDECREF(ctypes);
    if (!s_address || !s_data_ptr || !s_cuda_stream || !s_value || !g_void_p) return NULL;
    return PyModule_Create(&module);
}
