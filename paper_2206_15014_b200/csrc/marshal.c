/* Argument marshalling of the entry points that programs call once per layer, without ctypes.
 *
 * A small layer runs for 4-6 us on the device, and ctypes took up to 2.5 us of the host's time to convert the eleven arguments
 * of a call (0.8 us here; nm_absmax 1.1 -> 0.3).  Every entry has the name, the arguments and the defaults of its Python twin in
 * __init__.py and calls the same C entry point.  Whatever it does not recognise at once (an argument of another type, an unknown
 * keyword, a value outside its C type) goes to that twin unchanged, which converts it or raises as it always did; so does the
 * error report. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <limits.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>
#include "../../include/nmsparse.h"

/* Kinds of arguments: tensor or None; C int; float; size_t; packed-weight descriptor; stream handle or None. */
enum { PTR = 'p', INT = 'i', FLT = 'f', SIZE = 'z', PACKED = 'W', STREAM = 's' };
#define MAX_ARGS 12
typedef union { void* p; int i; float f; size_t z; } Arg;

typedef struct {
    const char* name;
    const char* kinds;                 /* one letter per argument */
    int required;
    const char* args[MAX_ARGS];
    PyObject* names[MAX_ARGS];         /* the same, interned */
} Spec;

enum { LINEAR, LINEAR_DSX, LINEAR_Q8, LINEAR_BF16, ABSMAX, QUANTIZE, NSPECS };
static Spec specs[NSPECS] = {
    {"nm_int_linear", "piWfppppzps", 7, {"X", "tokens", "W", "sx", "sw", "bias", "Y", "ws", "ws_bytes", "status", "stream"}, {0}},
    {"nm_int_linear_dsx", "piWppppppzps", 7, {"X", "tokens", "W", "sx_dev", "sw", "bias", "Y", "absmax_out", "ws", "ws_bytes", "status", "stream"}, {0}},
    {"nm_int_linear_q8", "piWfppfppzps", 8, {"X", "tokens", "W", "sx", "sw", "bias", "sy", "Yq", "ws", "ws_bytes", "status", "stream"}, {0}},
    {"nm_int_linear_bf16", "piWfppppzps", 7, {"X", "tokens", "W", "sx", "sw", "bias", "Ybf16", "ws", "ws_bytes", "status", "stream"}, {0}},
    {"nm_absmax", "pzps", 3, {"Y", "count", "absmax", "stream"}, {0}},
    {"nm_quantize_act", "pzppps", 4, {"Y", "count", "absmax", "Xq", "sx_out", "stream"}, {0}},
};

/* One entry point of one loaded library. */
typedef struct {
    PyObject_HEAD
    vectorcallfunc vectorcall;
    const Spec* spec;
    void* fn;                          /* C entry point */
    PyObject* twin;                    /* the Python function */
    PyObject* packed_type;             /* class of the weight descriptor */
    PyObject* check;                   /* check(code, name) raises the library's error */
    PyObject *dict, *weakrefs;
} Entry;

static PyObject *s_data_ptr, *current_device, *raw_stream;

/* The stream of the current device, as __init__._stream finds it. */
static int current_stream(void** out) {
    if (!raw_stream) {
        PyObject* cuda = PyImport_ImportModule("torch.cuda");
        PyObject* c = cuda ? PyImport_ImportModule("torch._C") : NULL;
        if (c) {
            if (!current_device) current_device = PyObject_GetAttrString(cuda, "current_device");
            if (current_device) raw_stream = PyObject_GetAttrString(c, "_cuda_getCurrentRawStream");
        }
        Py_XDECREF(cuda);
        Py_XDECREF(c);
        if (!raw_stream) return 0;
    }
    PyObject* dev = PyObject_CallNoArgs(current_device);
    if (!dev) return 0;
    PyObject* h = PyObject_CallOneArg(raw_stream, dev);
    Py_DECREF(dev);
    if (!h) return 0;
    *out = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

/* 1 when `o` is a plain value of its kind, converted into *out; 0 (perhaps with an exception set) otherwise. */
static int convert(const Entry* e, char kind, PyObject* o, Arg* out) {
    switch (kind) {
        case PTR: {
            if (o == Py_None) { out->p = NULL; return 1; }
            PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
            if (!v) return 0;
            const int ok = PyLong_CheckExact(v);
            out->p = ok ? PyLong_AsVoidPtr(v) : NULL;
            Py_DECREF(v);
            return ok && !PyErr_Occurred();
        }
        case INT: {
            if (!PyLong_CheckExact(o)) return 0;
            int over = 0;
            const long v = PyLong_AsLongAndOverflow(o, &over);
            if (over || v < INT_MIN || v > INT_MAX) return 0;
            out->i = (int)v;
            return 1;
        }
        case FLT:
            if (!PyFloat_CheckExact(o)) return 0;
            out->f = (float)PyFloat_AS_DOUBLE(o);
            return 1;
        case SIZE: {
            if (!PyLong_CheckExact(o)) return 0;
            out->z = PyLong_AsSize_t(o);
            return !PyErr_Occurred();
        }
        case PACKED: {
            if ((PyObject*)Py_TYPE(o) != e->packed_type) return 0;
            Py_buffer b;
            if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return 0;
            const int ok = b.len == (Py_ssize_t)sizeof(nm_packed_t);
            out->p = b.buf;  /* the argument keeps the structure alive during the call */
            PyBuffer_Release(&b);
            return ok;
        }
        default:  /* STREAM */
            if (o == Py_None) return current_stream(&out->p);
            if (!PyLong_CheckExact(o)) return 0;
            out->p = PyLong_AsVoidPtr(o);
            return !PyErr_Occurred();
    }
}

static PyObject* call(PyObject* self, PyObject* const* argv, size_t nargsf, PyObject* kwnames) {
    const Entry* e = (const Entry*)self;
    const Spec* s = e->spec;
    const Py_ssize_t npos = PyVectorcall_NARGS(nargsf);
    const int n = (int)strlen(s->kinds);
    PyObject* given[MAX_ARGS] = {NULL};
    Arg a[MAX_ARGS];
    if (npos > n) goto twin;
    for (Py_ssize_t i = 0; i < npos; ++i) given[i] = argv[i];
    if (kwnames) {
        const Py_ssize_t nkw = PyTuple_GET_SIZE(kwnames);
        for (Py_ssize_t k = 0; k < nkw; ++k) {
            PyObject* name = PyTuple_GET_ITEM(kwnames, k);
            int i = (int)npos;
            while (i < n && s->names[i] != name) ++i;  /* keywords in a call are interned; another string goes to the twin */
            if (i == n || given[i]) goto twin;
            given[i] = argv[npos + k];
        }
    }
    for (int i = 0; i < n; ++i) {
        if (!given[i]) {
            if (i < s->required) goto twin;
            if (s->kinds[i] == SIZE) { a[i].z = 0; continue; }
            given[i] = Py_None;
        }
        if (!convert(e, s->kinds[i], given[i], &a[i])) goto twin;
    }
    int rc = 0;
    Py_BEGIN_ALLOW_THREADS
    switch (s - specs) {
        case LINEAR:
            rc = ((int (*)(const int8_t*, int, const nm_packed_t*, float, const float*, const float*, float*, void*, size_t, uint32_t*, void*))e->fn)(
                a[0].p, a[1].i, a[2].p, a[3].f, a[4].p, a[5].p, a[6].p, a[7].p, a[8].z, a[9].p, a[10].p);
            break;
        case LINEAR_DSX:
            rc = ((int (*)(const int8_t*, int, const nm_packed_t*, const float*, const float*, const float*, float*, float*, void*, size_t, uint32_t*, void*))e->fn)(
                a[0].p, a[1].i, a[2].p, a[3].p, a[4].p, a[5].p, a[6].p, a[7].p, a[8].p, a[9].z, a[10].p, a[11].p);
            break;
        case LINEAR_Q8:
            rc = ((int (*)(const int8_t*, int, const nm_packed_t*, float, const float*, const float*, float, int8_t*, void*, size_t, uint32_t*, void*))e->fn)(
                a[0].p, a[1].i, a[2].p, a[3].f, a[4].p, a[5].p, a[6].f, a[7].p, a[8].p, a[9].z, a[10].p, a[11].p);
            break;
        case LINEAR_BF16:
            rc = ((int (*)(const int8_t*, int, const nm_packed_t*, float, const float*, const float*, uint16_t*, void*, size_t, uint32_t*, void*))e->fn)(
                a[0].p, a[1].i, a[2].p, a[3].f, a[4].p, a[5].p, a[6].p, a[7].p, a[8].z, a[9].p, a[10].p);
            break;
        case ABSMAX:
            rc = ((int (*)(const float*, size_t, float*, void*))e->fn)(a[0].p, a[1].z, a[2].p, a[3].p);
            break;
        default:
            rc = ((int (*)(const float*, size_t, const float*, int8_t*, float*, void*))e->fn)(a[0].p, a[1].z, a[2].p, a[3].p, a[4].p, a[5].p);
    }
    Py_END_ALLOW_THREADS
    if (rc == NM_OK) Py_RETURN_NONE;
    return PyObject_CallFunction(e->check, "is", rc, s->name);
twin:
    PyErr_Clear();
    return PyObject_Vectorcall(e->twin, argv, (size_t)npos, kwnames);
}

static int entry_traverse(PyObject* self, visitproc visit, void* arg) {
    Entry* e = (Entry*)self;
    Py_VISIT(e->twin); Py_VISIT(e->packed_type); Py_VISIT(e->check); Py_VISIT(e->dict);
    return 0;
}
/* The cycle through the twin's globals is broken there: an entry that a finaliser calls late still has all it needs. */
static int entry_clear(PyObject* self) {
    Py_CLEAR(((Entry*)self)->dict);
    return 0;
}
static void entry_dealloc(PyObject* self) {
    Entry* e = (Entry*)self;
    PyObject_GC_UnTrack(self);
    if (e->weakrefs) PyObject_ClearWeakRefs(self);
    Py_CLEAR(e->dict);
    Py_DECREF(e->twin); Py_DECREF(e->packed_type); Py_DECREF(e->check);
    PyObject_GC_Del(self);
}
/* Everything else that a Python function can do: __name__, __doc__ and the signature (through __wrapped__) are the twin's, and so is
 * every attribute not set here; an entry pickles and copies by its name, binds as a method and takes attributes and weak references. */
static PyObject* entry_getattro(PyObject* self, PyObject* name) {
    PyObject* v = PyObject_GenericGetAttr(self, name);
    if (v || !PyErr_ExceptionMatches(PyExc_AttributeError)) return v;
    PyErr_Clear();
    return PyObject_GetAttr(((Entry*)self)->twin, name);
}
static PyObject* entry_repr(PyObject* self) { return PyObject_Repr(((Entry*)self)->twin); }
static PyObject* entry_bind(PyObject* self, PyObject* obj, PyObject* type) {
    (void)type;
    return obj ? PyMethod_New(self, obj) : Py_NewRef(self);
}
static PyObject* entry_reduce(PyObject* self, PyObject* none) { (void)none; return PyObject_GetAttrString(((Entry*)self)->twin, "__qualname__"); }
static PyMethodDef entry_methods[] = {{"__reduce__", entry_reduce, METH_NOARGS, NULL}, {NULL, NULL, 0, NULL}};
static PyObject* get_wrapped(PyObject* self, void* c) { (void)c; return Py_NewRef(((Entry*)self)->twin); }
static PyObject* get_of_twin(PyObject* self, void* attr) { return PyObject_GetAttrString(((Entry*)self)->twin, (const char*)attr); }
static PyGetSetDef entry_getset[] = {{"__wrapped__", get_wrapped, NULL, NULL, NULL},
                                     {"__name__", get_of_twin, NULL, NULL, "__name__"},
                                     {"__qualname__", get_of_twin, NULL, NULL, "__qualname__"},
                                     {"__module__", get_of_twin, NULL, NULL, "__module__"},
                                     {"__doc__", get_of_twin, NULL, NULL, "__doc__"},
                                     {"__dict__", PyObject_GenericGetDict, PyObject_GenericSetDict, NULL, NULL},
                                     {NULL, NULL, NULL, NULL, NULL}};
static PyTypeObject EntryType = {
    PyVarObject_HEAD_INIT(NULL, 0).tp_name = "_marshal.Entry",
    .tp_basicsize = sizeof(Entry),
    .tp_flags = Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_GC | Py_TPFLAGS_HAVE_VECTORCALL,
    .tp_vectorcall_offset = offsetof(Entry, vectorcall),
    .tp_call = PyVectorcall_Call,
    .tp_dealloc = entry_dealloc,
    .tp_traverse = entry_traverse,
    .tp_clear = entry_clear,
    .tp_getset = entry_getset,
    .tp_methods = entry_methods,
    .tp_getattro = entry_getattro,
    .tp_setattro = PyObject_GenericSetAttr,
    .tp_repr = entry_repr,
    .tp_descr_get = entry_bind,
    .tp_dictoffset = offsetof(Entry, dict),
    .tp_weaklistoffset = offsetof(Entry, weakrefs),
};

/* entry(name, address of the C entry point, Python twin, weight descriptor class, check) */
static PyObject* entry(PyObject* self, PyObject* args) {
    const char* name;
    unsigned long long address;
    PyObject *twin, *cls, *check;
    (void)self;
    if (!PyArg_ParseTuple(args, "sKOOO", &name, &address, &twin, &cls, &check)) return NULL;
    for (int i = 0; i < NSPECS; ++i) {
        if (strcmp(specs[i].name, name)) continue;
        Entry* e = PyObject_GC_New(Entry, &EntryType);
        if (!e) return NULL;
        e->vectorcall = call;
        e->spec = &specs[i];
        e->fn = (void*)(uintptr_t)address;
        e->twin = Py_NewRef(twin);
        e->packed_type = Py_NewRef(cls);
        e->check = Py_NewRef(check);
        e->dict = e->weakrefs = NULL;
        PyObject_GC_Track((PyObject*)e);
        return (PyObject*)e;
    }
    return PyErr_Format(PyExc_KeyError, "%s", name);
}

static PyMethodDef methods[] = {{"entry", entry, METH_VARARGS, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) {
    if (PyType_Ready(&EntryType) < 0) return NULL;
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    if (!s_data_ptr) return NULL;
    for (int i = 0; i < NSPECS; ++i)
        for (int k = 0; specs[i].kinds[k]; ++k)
            if (!(specs[i].names[k] = PyUnicode_InternFromString(specs[i].args[k]))) return NULL;
    return PyModule_Create(&module);
}
