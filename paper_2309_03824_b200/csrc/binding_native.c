/* Argument marshalling of the launch calls in C: what binding.py's device entry points do per call.
 *
 * A step of a small layer is a few launches of some ten microseconds each, and marshalling a call through ctypes objects
 * took the interpreter 7 to 9 microseconds (linear_fwd / linear_bwd) -- as long as the GPU takes for a launch.  Here a
 * call costs 1.0 / 2.3: tensors are asked for their data_ptr(), descriptors (ctypes structures) are read through the
 * buffer protocol, the current stream comes from torch's own lookup.  Nothing of a call is kept for the next;
 * the two stream functions of torch are looked up once.  The GIL is released around the library call, as ctypes does.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <string.h>

#include "../../include/lrd.h"

static PyObject *s_data_ptr, *s_numel, *s_element_size;      /* interned method names */
static PyObject* stream_source;                              /* () -> (current device, device -> its current raw stream) */
static PyObject *fn_device, *fn_stream;
static PyTypeObject *linear_type, *tucker2_type;             /* the binding's two descriptor structures */

typedef struct {
    PyObject* const* v;      /* the call's arguments */
    int bad;                 /* a Python exception is set */
} Args;

static void* pointer(Args* a, PyObject* t) {
    if (a->bad || t == Py_None) return NULL;
    PyObject* r = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!r) { a->bad = 1; return NULL; }
    void* p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    if (!p && PyErr_Occurred()) a->bad = 1;
    return p;
}
static void* ptr(Args* a, int i) { return pointer(a, a->v[i]); }

static long long integer(Args* a, PyObject* o) {
    if (a->bad) return 0;
    const long long x = PyLong_AsLongLong(o);
    if (x == -1 && PyErr_Occurred()) a->bad = 1;
    return x;
}
static long long num(Args* a, int i) { return integer(a, a->v[i]); }

static size_t bytes_of(Args* a, PyObject* t) {               /* of a workspace tensor; 0 for None */
    if (a->bad || t == Py_None) return 0;
    PyObject* n = PyObject_CallMethodNoArgs(t, s_numel);
    PyObject* e = n ? PyObject_CallMethodNoArgs(t, s_element_size) : NULL;
    size_t r = 0;
    if (e) r = (size_t)integer(a, n) * (size_t)integer(a, e);
    else a->bad = 1;
    Py_XDECREF(n);
    Py_XDECREF(e);
    return r;
}
static size_t nbytes(Args* a, int i) { return bytes_of(a, a->v[i]); }

static void* stream(Args* a, int i) {
    if (a->bad) return NULL;
    if (a->v[i] != Py_None) {
        PyObject* o = PyNumber_Long(a->v[i]);
        void* p = o ? PyLong_AsVoidPtr(o) : NULL;
        Py_XDECREF(o);
        if (!p && PyErr_Occurred()) a->bad = 1;
        return p;
    }
    if (!fn_stream) {
        PyObject *device = NULL, *raw = NULL, *pair = PyObject_CallNoArgs(stream_source);
        if (!pair || !PyArg_ParseTuple(pair, "OO", &device, &raw)) {
            Py_XDECREF(pair);
            a->bad = 1;
            return NULL;
        }
        if (!fn_stream) {                                    /* (the call above may have let another thread in) */
            fn_device = Py_NewRef(device);
            fn_stream = Py_NewRef(raw);
        }
        Py_DECREF(pair);
    }
    PyObject* dev = PyObject_CallNoArgs(fn_device);
    PyObject* s = dev ? PyObject_CallOneArg(fn_stream, dev) : NULL;
    Py_XDECREF(dev);
    void* p = s ? PyLong_AsVoidPtr(s) : NULL;
    if (!s || (!p && PyErr_Occurred())) a->bad = 1;
    Py_XDECREF(s);
    return p;
}

static void descriptor(Args* a, PyObject* o, PyTypeObject* type, void* out, size_t size) {
    Py_buffer b;
    if (a->bad) return;
    if (!PyObject_TypeCheck(o, type)) {
        PyErr_Format(PyExc_TypeError, "expected %s, not %s", type->tp_name, Py_TYPE(o)->tp_name);
        a->bad = 1;
        return;
    }
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) { a->bad = 1; return; }
    if ((size_t)b.len == size) {
        memcpy(out, b.buf, size);
    } else {
        PyErr_SetString(PyExc_TypeError, "not a descriptor of this call");
        a->bad = 1;
    }
    PyBuffer_Release(&b);
}

#define ENTRY(name, count)                                                                      \
    static PyObject* py_##name(PyObject* self, PyObject* const* v, Py_ssize_t n) {              \
        Args args = {v, 0}, *a = &args;                                                         \
        lrd_status_t st = LRD_OK;                                                               \
        (void)self;                                                                             \
        if (n != (count)) return PyErr_Format(PyExc_TypeError, #name ": %d arguments", (count));
#define CALL(expr)                         \
        if (a->bad) return NULL;           \
        Py_BEGIN_ALLOW_THREADS             \
        st = (expr);                       \
        Py_END_ALLOW_THREADS               \
        return PyLong_FromLong((long)st);  \
    }

ENTRY(linear_fwd, 10)      /* desc X V U bias Y Z_save freeze workspace stream */
    lrd_linear_desc_t d;
    descriptor(a, v[0], linear_type, &d, sizeof d);
    void *X = ptr(a, 1), *V = ptr(a, 2), *U = ptr(a, 3), *bias = ptr(a, 4), *Y = ptr(a, 5), *Z = ptr(a, 6), *w = ptr(a, 8), *s = stream(a, 9);
    const lrd_freeze_t f = (lrd_freeze_t)num(a, 7);
    const size_t nb = nbytes(a, 8);
CALL(lrd_linear_fwd(&d, X, V, U, bias, Y, Z, f, w, nb, s))

#define BACKWARD(name)     /* desc dY X V U Z_save dX dU dV dbias freeze workspace stream */                                   \
    ENTRY(name, 13)                                                                                                            \
    lrd_linear_desc_t d;                                                                                                       \
    descriptor(a, v[0], linear_type, &d, sizeof d);                                                                            \
    void *dY = ptr(a, 1), *X = ptr(a, 2), *V = ptr(a, 3), *U = ptr(a, 4), *Z = ptr(a, 5), *dX = ptr(a, 6), *dU = ptr(a, 7),     \
         *dV = ptr(a, 8), *db = ptr(a, 9), *w = ptr(a, 11), *s = stream(a, 12);                                                \
    const lrd_freeze_t f = (lrd_freeze_t)num(a, 10);                                                                           \
    const size_t nb = nbytes(a, 11);                                                                                           \
    CALL(lrd_##name(&d, dY, X, V, U, Z, dX, dU, dV, db, f, w, nb, s))
BACKWARD(linear_bwd)
BACKWARD(linear_bwd_accumulate)

ENTRY(linear_bwd_data, 8)  /* desc dY V U dX freeze workspace stream */
    lrd_linear_desc_t d;
    descriptor(a, v[0], linear_type, &d, sizeof d);
    void *dY = ptr(a, 1), *V = ptr(a, 2), *U = ptr(a, 3), *dX = ptr(a, 4), *w = ptr(a, 6), *s = stream(a, 7);
    const lrd_freeze_t f = (lrd_freeze_t)num(a, 5);
    const size_t nb = nbytes(a, 6);
CALL(lrd_linear_bwd_data(&d, dY, V, U, dX, f, w, nb, s))

ENTRY(linear_bwd_weights, 10)      /* desc dY X Z_save dU dV dbias freeze workspace stream */
    lrd_linear_desc_t d;
    descriptor(a, v[0], linear_type, &d, sizeof d);
    void *dY = ptr(a, 1), *X = ptr(a, 2), *Z = ptr(a, 3), *dU = ptr(a, 4), *dV = ptr(a, 5), *db = ptr(a, 6), *w = ptr(a, 8), *s = stream(a, 9);
    const lrd_freeze_t f = (lrd_freeze_t)num(a, 7);
    const size_t nb = nbytes(a, 8);
CALL(lrd_linear_bwd_weights(&d, dY, X, Z, dU, dV, db, f, w, nb, s))

ENTRY(dense_fwd, 7)        /* desc X W bias Y workspace stream */
    lrd_linear_desc_t d;
    descriptor(a, v[0], linear_type, &d, sizeof d);
    void *X = ptr(a, 1), *W = ptr(a, 2), *bias = ptr(a, 3), *Y = ptr(a, 4), *w = ptr(a, 5), *s = stream(a, 6);
    const size_t nb = nbytes(a, 5);
CALL(lrd_dense_fwd(&d, X, W, bias, Y, w, nb, s))

ENTRY(dense_bwd, 9)        /* desc dY X W dX dW dbias workspace stream */
    lrd_linear_desc_t d;
    descriptor(a, v[0], linear_type, &d, sizeof d);
    void *dY = ptr(a, 1), *X = ptr(a, 2), *W = ptr(a, 3), *dX = ptr(a, 4), *dW = ptr(a, 5), *db = ptr(a, 6), *w = ptr(a, 7), *s = stream(a, 8);
    const size_t nb = nbytes(a, 7);
CALL(lrd_dense_bwd(&d, dY, X, W, dX, dW, db, w, nb, s))

ENTRY(tucker2_fwd, 12)     /* desc X A G Bm bias Y Z1_save Z2_save freeze workspace stream */
    lrd_tucker2_desc_t d;
    descriptor(a, v[0], tucker2_type, &d, sizeof d);
    void *X = ptr(a, 1), *A = ptr(a, 2), *G = ptr(a, 3), *B = ptr(a, 4), *bias = ptr(a, 5), *Y = ptr(a, 6), *Z1 = ptr(a, 7), *Z2 = ptr(a, 8),
         *w = ptr(a, 10), *s = stream(a, 11);
    const lrd_tucker_freeze_t f = (lrd_tucker_freeze_t)num(a, 9);
    const size_t nb = nbytes(a, 10);
CALL(lrd_tucker2_fwd(&d, X, A, G, B, bias, Y, Z1, Z2, f, w, nb, s))

ENTRY(tucker2_bwd, 16)     /* desc dY X A G Bm Z1_save Z2_save dX dA dG dB dbias freeze workspace stream */
    lrd_tucker2_desc_t d;
    descriptor(a, v[0], tucker2_type, &d, sizeof d);
    void *dY = ptr(a, 1), *X = ptr(a, 2), *A = ptr(a, 3), *G = ptr(a, 4), *B = ptr(a, 5), *Z1 = ptr(a, 6), *Z2 = ptr(a, 7), *dX = ptr(a, 8),
         *dA = ptr(a, 9), *dG = ptr(a, 10), *dB = ptr(a, 11), *db = ptr(a, 12), *w = ptr(a, 14), *s = stream(a, 15);
    const lrd_tucker_freeze_t f = (lrd_tucker_freeze_t)num(a, 13);
    const size_t nb = nbytes(a, 14);
CALL(lrd_tucker2_bwd(&d, dY, X, A, G, B, Z1, Z2, dX, dA, dG, dB, db, f, w, nb, s))

/* ---- groups: every argument but freeze and stream is a list with one entry per layer (or None as a whole) ----------- */
#define MAX_LISTS 9
typedef struct {
    int n;
    lrd_linear_desc_t* descs;
    void** p[MAX_LISTS];
    void** ws;
    size_t* ws_bytes;
    void* block;
} Group;

/* v[0] = descriptors, v[1 .. lists] = tensor lists, workspaces in v[at_ws] */
static void group_parse(Args* a, Group* g, int lists, int at_ws) {
    memset(g, 0, sizeof *g);
    PyObject* ds = PySequence_Fast(a->v[0], "a list of descriptors");
    if (!ds) { a->bad = 1; return; }
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(ds);
    g->n = (int)n;
    g->block = PyMem_Calloc(1, (size_t)n * (sizeof(lrd_linear_desc_t) + (size_t)(lists + 1) * sizeof(void*) + sizeof(size_t)) + 1);
    if (!g->block) { PyErr_NoMemory(); a->bad = 1; Py_DECREF(ds); return; }
    g->descs = (lrd_linear_desc_t*)g->block;
    void** at = (void**)(g->descs + n);
    for (Py_ssize_t i = 0; i < n; ++i) descriptor(a, PySequence_Fast_GET_ITEM(ds, i), linear_type, &g->descs[i], sizeof g->descs[i]);
    Py_DECREF(ds);
    for (int k = 0; k <= lists && !a->bad; ++k, at += n) {
        PyObject* arg = a->v[k < lists ? k + 1 : at_ws];
        if (k < lists && arg == Py_None) continue;
        PyObject* l = PySequence_Fast(arg, "a list with one entry per layer");
        if (!l) { a->bad = 1; return; }
        if (PySequence_Fast_GET_SIZE(l) != n) {
            PyErr_SetString(PyExc_ValueError, "every per-layer list of a group has one entry per layer");
            a->bad = 1;
        }
        for (Py_ssize_t i = 0; i < n && !a->bad; ++i) at[i] = pointer(a, PySequence_Fast_GET_ITEM(l, i));
        if (k < lists) {
            g->p[k] = at;
        } else {
            g->ws = at;
            g->ws_bytes = (size_t*)(at + n);
            for (Py_ssize_t i = 0; i < n && !a->bad; ++i) g->ws_bytes[i] = bytes_of(a, PySequence_Fast_GET_ITEM(l, i));
        }
        Py_DECREF(l);
    }
}

#define GROUP_CALL(expr)                                    \
        if (a->bad) { PyMem_Free(g.block); return NULL; }   \
        Py_BEGIN_ALLOW_THREADS                              \
        st = (expr);                                        \
        Py_END_ALLOW_THREADS                                \
        PyMem_Free(g.block);                                \
        return PyLong_FromLong((long)st);                   \
    }
#define IN(k) ((const void* const*)g.p[k])

ENTRY(linear_group_fwd, 10)        /* descs X V U bias Y Z_save | freeze workspaces stream */
    Group g;
    group_parse(a, &g, 6, 8);
    const lrd_freeze_t f = (lrd_freeze_t)num(a, 7);
    void* s = stream(a, 9);
GROUP_CALL(lrd_linear_group_fwd(g.n, g.descs, IN(0), IN(1), IN(2), IN(3), g.p[4], g.p[5], f, g.ws, g.ws_bytes, s))

ENTRY(linear_group_bwd, 13)        /* descs dY X V U Z_save dX dU dV dbias | freeze workspaces stream */
    Group g;
    group_parse(a, &g, 9, 11);
    const lrd_freeze_t f = (lrd_freeze_t)num(a, 10);
    void* s = stream(a, 12);
GROUP_CALL(lrd_linear_group_bwd(g.n, g.descs, IN(0), IN(1), IN(2), IN(3), IN(4), g.p[5], g.p[6], g.p[7], g.p[8], f, g.ws, g.ws_bytes, s))

static PyObject* py_set_stream_source(PyObject* self, PyObject* f) {
    (void)self;
    Py_XSETREF(stream_source, Py_NewRef(f));
    Py_RETURN_NONE;
}

static PyObject* py_set_descriptor_types(PyObject* self, PyObject* args) {
    PyTypeObject *linear, *tucker2;
    (void)self;
    if (!PyArg_ParseTuple(args, "O!O!", &PyType_Type, &linear, &PyType_Type, &tucker2)) return NULL;
    Py_XSETREF(linear_type, (PyTypeObject*)Py_NewRef(linear));
    Py_XSETREF(tucker2_type, (PyTypeObject*)Py_NewRef(tucker2));
    Py_RETURN_NONE;
}

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {METHOD(linear_fwd), METHOD(linear_bwd), METHOD(linear_bwd_accumulate), METHOD(linear_bwd_data),
                                METHOD(linear_bwd_weights), METHOD(dense_fwd), METHOD(dense_bwd), METHOD(tucker2_fwd), METHOD(tucker2_bwd),
                                METHOD(linear_group_fwd), METHOD(linear_group_bwd),
                                {"set_stream_source", py_set_stream_source, METH_O, NULL},
                                {"set_descriptor_types", py_set_descriptor_types, METH_VARARGS, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_numel = PyUnicode_InternFromString("numel");
    s_element_size = PyUnicode_InternFromString("element_size");
    return s_data_ptr && s_numel && s_element_size ? PyModule_Create(&module) : NULL;
}
