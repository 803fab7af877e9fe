/* Argument marshalling of the hot entry points (dbspmspv_run, dbspmspv_run_masked, dbspmspv_decode,
 * dbspmspv_decode_batch, db_bfs, db_sssp) as a CPython extension: the same names, arguments,
 * defaults and errors as a ctypes wrapper, at a tenth of its cost.
 *
 * What bounds a short call is the host.  Through ctypes the marshalling alone took 6 us of a 10 us
 * call: 3.4 us to ask torch.cuda.current_stream() for the stream (0.17 us from the two raw
 * getters used here), the rest argument conversion.
 *
 * The extension links neither the library nor torch: binding.py hands it the addresses of the
 * entry points (whichever build of the library was loaded) on first use, and the stream getters when
 * the first call without a stream argument asks for them: a call that names its stream needs no torch. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

enum { F_RUN, F_RUN_MASKED, F_DECODE, F_DECODE_BATCH, F_BFS, F_SSSP, N_FUNCS };

static void *g_addr[N_FUNCS];
static PyObject *g_load;          /* called once: loads the library and calls setup() */
static PyObject *g_plain;         /* (object) -> what stands behind a ctypes instance or an object with _as_parameter_ */
static PyObject *g_raise;         /* (status, name) -> raises DbSpmspvError */
static PyObject *g_bind_streams;  /* called once, by the first call without a stream argument: calls streams() */
static PyObject *g_get_device;    /* () -> int */
static PyObject *g_get_stream;    /* (device) -> int, the raw current stream */
static PyObject *s_data_ptr, *s_ctypes, *s_data;

static int ready(void) {
    if (g_addr[F_RUN]) return 1;
    if (!g_load) { PyErr_SetString(PyExc_RuntimeError, "the binding has not been set up"); return 0; }
    PyObject *r = PyObject_CallNoArgs(g_load);
    if (!r) return 0;
    Py_DECREF(r);
    if (!g_addr[F_RUN]) { PyErr_SetString(PyExc_RuntimeError, "the library's entry points are not bound"); return 0; }
    return 1;
}

/* address of a tensor (data_ptr()) or a numpy array (ctypes.data); None is NULL */
static int as_pointer(PyObject *o, void **out) {
    if (o == Py_None) { *out = NULL; return 1; }
    PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return 0;
        PyErr_Clear();
        PyObject *c = PyObject_GetAttr(o, s_ctypes);
        if (!c) return 0;
        v = PyObject_GetAttr(c, s_data);
        Py_DECREF(c);
        if (!v) return 0;
    }
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*out == NULL && PyErr_Occurred());
}

/* an argument as a Python integer (or None): as a ctypes prototype, it takes a ctypes instance or an object with _as_parameter_ too */
static PyObject *plain(PyObject *o) {
    if (PyLong_Check(o) || o == Py_None) { Py_INCREF(o); return o; }
    return PyObject_CallOneArg(g_plain, o);
}

/* a handle or a stream: an integer, or None for NULL */
static int as_opaque(PyObject *o, void **out) {
    PyObject *v = plain(o);
    if (!v) return 0;
    *out = NULL;
    if (v != Py_None) {
        if (!PyLong_Check(v)) PyErr_Format(PyExc_TypeError, "an integer or None is wanted, not %.80s", Py_TYPE(v)->tp_name);
        else *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(v);
    }
    Py_DECREF(v);
    return !PyErr_Occurred();
}

/* (an integer that does not fit keeps its low bits, as it does through ctypes) */
static int as_i64(PyObject *o, int64_t *out) {
    PyObject *p = plain(o), *v = p ? PyNumber_Index(p) : NULL;
    Py_XDECREF(p);
    if (!v) return 0;
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(v);
    Py_DECREF(v);
    return !PyErr_Occurred();
}
static int as_i32(PyObject *o, int32_t *out) {
    int64_t v = 0;
    if (!as_i64(o, &v)) return 0;
    *out = (int32_t)v;
    return 1;
}

/* the stream argument: None (or absent) is torch's current stream on the current device */
static int as_stream(PyObject *o, void **out) {
    if (o && o != Py_None) return as_opaque(o, out);
    if (!g_get_stream) {
        PyObject *r = PyObject_CallNoArgs(g_bind_streams);
        if (!r) return 0;
        Py_DECREF(r);
        if (!g_get_stream) { PyErr_SetString(PyExc_RuntimeError, "the stream getters have not been set"); return 0; }
    }
    PyObject *dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return 0;
    PyObject *s = PyObject_CallOneArg(g_get_stream, dev);
    Py_DECREF(dev);
    if (!s) return 0;
    const int ok = as_opaque(s, out);
    Py_DECREF(s);
    return ok;
}

/* positional and keyword arguments -> slots, in the order of `names`; the last one (stream) may be absent */
static int unpack(const char *fn, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames, const char *const *names, int n, PyObject **slot) {
    if (nargs > n) { PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", fn, n, nargs); return 0; }
    for (int i = 0; i < n; ++i) slot[i] = i < nargs ? args[i] : NULL;
    const Py_ssize_t nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nk; ++k) {
        PyObject *name = PyTuple_GET_ITEM(kwnames, k);
        int i = 0;
        while (i < n && PyUnicode_CompareWithASCIIString(name, names[i]) != 0) ++i;
        if (i == n) { PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", fn, name); return 0; }
        if (slot[i]) { PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", fn, names[i]); return 0; }
        slot[i] = args[nargs + k];
    }
    for (int i = 0; i < n - 1; ++i)
        if (!slot[i]) { PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", fn, names[i]); return 0; }
    return 1;
}

static PyObject *finish(int status, const char *name) {
    if (status == 0) Py_RETURN_NONE;
    PyObject *r = PyObject_CallFunction(g_raise, "is", status, name);
    Py_XDECREF(r);
    if (!PyErr_Occurred()) PyErr_Format(PyExc_RuntimeError, "%s: status %d", name, status);
    return NULL;
}

typedef int (*run_fn)(void *, const void *, const void *, int32_t, int, void *, void *, int64_t, void *, void *);
typedef int (*run_masked_fn)(void *, const void *, const void *, int32_t, int, const void *, int, void *, void *, int64_t, void *, void *);
typedef int (*decode_fn)(void *, const void *, void *, void *);
typedef int (*decode_batch_fn)(void *, const void *, int64_t, void *, int64_t, int32_t, void *);
typedef int (*bfs_fn)(void *, int32_t, void *, void *);
typedef int (*sssp_fn)(void *, int32_t, void *, int32_t *, void *);

static PyObject *f_run(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kw) {
    static const char *const names[] = {"h", "x_idx", "x_val", "nnz_x", "semiring", "y_idx", "y_val", "y_capacity", "y_nnz", "stream"};
    PyObject *a[10];
    void *h, *xi, *xv, *yi, *yv, *yn, *st;
    int32_t nnz, semiring;
    int64_t cap;
    if (!ready() || !unpack("dbspmspv_run", args, nargs, kw, names, 10, a)) return NULL;
    if (!as_opaque(a[0], &h) || !as_pointer(a[1], &xi) || !as_pointer(a[2], &xv) || !as_i32(a[3], &nnz) || !as_i32(a[4], &semiring) ||
        !as_pointer(a[5], &yi) || !as_pointer(a[6], &yv) || !as_i64(a[7], &cap) || !as_pointer(a[8], &yn) || !as_stream(a[9], &st)) return NULL;
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = ((run_fn)g_addr[F_RUN])(h, xi, xv, nnz, semiring, yi, yv, cap, yn, st);
    Py_END_ALLOW_THREADS
    return finish(s, "dbspmspv_run");
}

static PyObject *f_run_masked(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kw) {
    static const char *const names[] = {"h", "x_idx", "x_val", "nnz_x", "semiring", "row_mask", "complement", "y_idx", "y_val", "y_capacity", "y_nnz", "stream"};
    PyObject *a[12];
    void *h, *xi, *xv, *rm, *yi, *yv, *yn, *st;
    int32_t nnz, semiring, comp;
    int64_t cap;
    if (!ready() || !unpack("dbspmspv_run_masked", args, nargs, kw, names, 12, a)) return NULL;
    if (!as_opaque(a[0], &h) || !as_pointer(a[1], &xi) || !as_pointer(a[2], &xv) || !as_i32(a[3], &nnz) || !as_i32(a[4], &semiring) ||
        !as_pointer(a[5], &rm) || !as_i32(a[6], &comp) || !as_pointer(a[7], &yi) || !as_pointer(a[8], &yv) || !as_i64(a[9], &cap) ||
        !as_pointer(a[10], &yn) || !as_stream(a[11], &st)) return NULL;
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = ((run_masked_fn)g_addr[F_RUN_MASKED])(h, xi, xv, nnz, semiring, rm, comp, yi, yv, cap, yn, st);
    Py_END_ALLOW_THREADS
    return finish(s, "dbspmspv_run_masked");
}

static PyObject *f_decode(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kw) {
    static const char *const names[] = {"h", "x", "y", "stream"};
    PyObject *a[4];
    void *h, *x, *y, *st;
    if (!ready() || !unpack("dbspmspv_decode", args, nargs, kw, names, 4, a)) return NULL;
    if (!as_opaque(a[0], &h) || !as_pointer(a[1], &x) || !as_pointer(a[2], &y) || !as_stream(a[3], &st)) return NULL;
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = ((decode_fn)g_addr[F_DECODE])(h, x, y, st);
    Py_END_ALLOW_THREADS
    return finish(s, "dbspmspv_decode");
}

static PyObject *f_decode_batch(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kw) {
    static const char *const names[] = {"h", "x", "ldx", "y", "ldy", "batch", "stream"};
    PyObject *a[7];
    void *h, *x, *y, *st;
    int64_t ldx, ldy;
    int32_t batch;
    if (!ready() || !unpack("dbspmspv_decode_batch", args, nargs, kw, names, 7, a)) return NULL;
    if (!as_opaque(a[0], &h) || !as_pointer(a[1], &x) || !as_i64(a[2], &ldx) || !as_pointer(a[3], &y) || !as_i64(a[4], &ldy) || !as_i32(a[5], &batch) ||
        !as_stream(a[6], &st)) return NULL;
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = ((decode_batch_fn)g_addr[F_DECODE_BATCH])(h, x, ldx, y, ldy, batch, st);
    Py_END_ALLOW_THREADS
    return finish(s, "dbspmspv_decode_batch");
}

static PyObject *f_bfs(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kw) {
    static const char *const names[] = {"h", "src", "levels", "stream"};
    PyObject *a[4];
    void *h, *lv, *st;
    int32_t src;
    if (!ready() || !unpack("db_bfs", args, nargs, kw, names, 4, a)) return NULL;
    if (!as_opaque(a[0], &h) || !as_i32(a[1], &src) || !as_pointer(a[2], &lv) || !as_stream(a[3], &st)) return NULL;
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = ((bfs_fn)g_addr[F_BFS])(h, src, lv, st);
    Py_END_ALLOW_THREADS
    return finish(s, "db_bfs");
}

static PyObject *f_sssp(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kw) {
    static const char *const names[] = {"h", "src", "dist", "stream"};
    PyObject *a[4];
    void *h, *dist, *st;
    int32_t src, steps = 0;
    if (!ready() || !unpack("db_sssp", args, nargs, kw, names, 4, a)) return NULL;
    if (!as_opaque(a[0], &h) || !as_i32(a[1], &src) || !as_pointer(a[2], &dist) || !as_stream(a[3], &st)) return NULL;
    int s;
    Py_BEGIN_ALLOW_THREADS
    s = ((sssp_fn)g_addr[F_SSSP])(h, src, dist, &steps, st);
    Py_END_ALLOW_THREADS
    if (s != 0) return finish(s, "db_sssp");
    return PyLong_FromLong(steps);
}

/* set_loader(load, plain) */
static PyObject *f_set_loader(PyObject *self, PyObject *args) {
    PyObject *load, *pl;
    if (!PyArg_ParseTuple(args, "OO", &load, &pl)) return NULL;
    Py_INCREF(load); Py_XSETREF(g_load, load);
    Py_INCREF(pl); Py_XSETREF(g_plain, pl);
    Py_RETURN_NONE;
}

/* setup(addresses, raise, bind_streams) */
static PyObject *f_setup(PyObject *self, PyObject *args) {
    PyObject *addr, *rs, *bs;
    if (!PyArg_ParseTuple(args, "O!OO", &PyTuple_Type, &addr, &rs, &bs)) return NULL;
    if (PyTuple_GET_SIZE(addr) != N_FUNCS) { PyErr_SetString(PyExc_ValueError, "wrong number of addresses"); return NULL; }
    void *p[N_FUNCS];
    for (int i = 0; i < N_FUNCS; ++i)
        if (!as_opaque(PyTuple_GET_ITEM(addr, i), &p[i])) return NULL;
    Py_INCREF(rs); Py_XSETREF(g_raise, rs);
    Py_INCREF(bs); Py_XSETREF(g_bind_streams, bs);
    for (int i = 0; i < N_FUNCS; ++i) g_addr[i] = p[i];
    Py_RETURN_NONE;
}

/* streams(get_device, get_stream) */
static PyObject *f_streams(PyObject *self, PyObject *args) {
    PyObject *gd, *gs;
    if (!PyArg_ParseTuple(args, "OO", &gd, &gs)) return NULL;
    Py_INCREF(gd); Py_XSETREF(g_get_device, gd);
    Py_INCREF(gs); Py_XSETREF(g_get_stream, gs);
    Py_RETURN_NONE;
}

#define FAST(name, f) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL | METH_KEYWORDS, NULL}
static PyMethodDef methods[] = {
    FAST("dbspmspv_run", f_run), FAST("dbspmspv_run_masked", f_run_masked), FAST("dbspmspv_decode", f_decode),
    FAST("dbspmspv_decode_batch", f_decode_batch), FAST("db_bfs", f_bfs), FAST("db_sssp", f_sssp),
    {"set_loader", f_set_loader, METH_VARARGS, NULL}, {"setup", f_setup, METH_VARARGS, NULL}, {"streams", f_streams, METH_VARARGS, NULL}, {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_ctypes = PyUnicode_InternFromString("ctypes");
    s_data = PyUnicode_InternFromString("data");
    if (!s_data_ptr || !s_ctypes || !s_data) return NULL;
    return PyModule_Create(&module);
}
