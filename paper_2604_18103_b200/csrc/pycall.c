/* The binding's path of a decoding call, which on a short cache the host bounds (28 calls on 8192 and 2728 rows in a row: 220 us of GPU time, 280 before and 246
 * with this): what dash.py does with ctypes for the other entry points --
 * pointers, strides and sizes read from the tensors, one call of the C ABI without the interpreter's lock -- in C.  Per call: 2.9 us of attribute reads
 * in bytecode and 1.8 us of argument conversion in ctypes, 2.0 together here.  Tensors are asked through their Python methods (no torch header: nothing here depends
 * on a version of it, and subclasses and tracing tensors answer, or raise, as they do in Python).  Not needed: where it is not built for the running interpreter dash.py takes ctypes here too. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <math.h>
#include <stdint.h>

typedef int (*decode_fn)(const void*, const void*, const void*, void*, float*, int64_t, int64_t, int64_t, int64_t, const int32_t*, int, int64_t, int, int, int,
                         float, int, void*, size_t, void*);
static decode_fn g_decode;
static PyObject *g_bf16, *g_f32, *g_zero;
static PyObject *s_data_ptr, *s_stride, *s_numel, *s_is_cuda, *s_shape, *s_dtype;

/* object.name() as an integer; -1 with an exception set on failure */
static long long call_int(PyObject* o, PyObject* name, PyObject* arg, int* bad) {
    PyObject* args[2] = {o, arg};
    PyObject* r = PyObject_VectorcallMethod(name, args, arg ? 2 : 1, NULL);
    if (!r) { *bad = 1; return -1; }
    const unsigned long long v = PyLong_AsUnsignedLongLongMask(r);
    Py_DECREF(r);
    if (v == (unsigned long long)-1 && PyErr_Occurred()) { *bad = 1; return -1; }
    return (long long)v;
}
static void* ptr_of(PyObject* o, int* bad) { return o == Py_None ? NULL : (void*)(uintptr_t)call_int(o, s_data_ptr, NULL, bad); }
static int on_device(PyObject* o) {
    PyObject* r = PyObject_GetAttr(o, s_is_cuda);
    if (!r) return 0;
    const int yes = PyObject_IsTrue(r);
    Py_DECREF(r);
    if (yes == 0) PyErr_SetString(PyExc_ValueError, "device tensor expected");
    return yes > 0;
}
/* first `want` sizes (exactly that many dimensions if `exact`) */
static int sizes_of(PyObject* o, Py_ssize_t want, int exact, long long* out) {
    PyObject* sh = PyObject_GetAttr(o, s_shape);
    if (!sh) return 0;
    PyObject* seq = PySequence_Fast(sh, "a tensor's shape");
    Py_DECREF(sh);
    if (!seq) return 0;
    const Py_ssize_t dims = PySequence_Fast_GET_SIZE(seq);
    int ok = exact ? dims == want : dims >= want;
    if (!ok) PyErr_Format(PyExc_ValueError, "tensor of %zd dimensions where %zd are expected", dims, want);
    for (Py_ssize_t i = 0; ok && i < want; ++i) {
        PyObject* n = PyNumber_Index(PySequence_Fast_GET_ITEM(seq, i));
        out[i] = n ? PyLong_AsLongLong(n) : -1;
        Py_XDECREF(n);
        if (PyErr_Occurred()) ok = 0;
    }
    Py_DECREF(seq);
    return ok;
}

/* decode(q, K, V, cu_seqlens, scale or None, out, lse or None, ws, stream) -> status */
static PyObject* py_decode(PyObject* self, PyObject* const* a, Py_ssize_t n_args) {
    (void)self;
    if (n_args != 9 || !g_decode) { PyErr_SetString(PyExc_TypeError, "decode(q, K, V, cu_seqlens, scale, out, lse, ws, stream), after setup()"); return NULL; }
    PyObject *q = a[0], *K = a[1], *V = a[2], *cu = a[3], *out = a[5], *ws = a[7];
    if (!on_device(q) || !on_device(K) || !on_device(V) || !on_device(cu)) return NULL;
    long long qs[3], ks[2];
    if (!sizes_of(q, 3, 1, qs) || !sizes_of(K, 2, 0, ks)) return NULL;
    const long long n = ks[0], Hkv = ks[1], D = qs[2];
    const double scale = a[4] == Py_None ? 1.0 / pow((double)D, 0.5) : PyFloat_AsDouble(a[4]);
    if (PyErr_Occurred()) return NULL;
    PyObject* dt = PyObject_GetAttr(q, s_dtype);
    if (!dt) return NULL;
    const int code = dt == g_bf16 ? 1 : dt == g_f32 ? 0 : -1;
    if (code < 0) PyErr_Format(PyExc_TypeError, "unsupported dtype %S", dt);
    Py_DECREF(dt);
    if (code < 0) return NULL;
    int bad = 0;
    const void *qp = ptr_of(q, &bad), *kp = bad ? NULL : ptr_of(K, &bad), *vp = bad ? NULL : ptr_of(V, &bad);
    void *op = bad ? NULL : ptr_of(out, &bad), *lp = bad ? NULL : ptr_of(a[6], &bad), *wp = bad ? NULL : ptr_of(ws, &bad);
    const void* cp = bad ? NULL : ptr_of(cu, &bad);
    const long long ldq = bad ? 0 : call_int(q, s_stride, g_zero, &bad), ldo = bad ? 0 : call_int(out, s_stride, g_zero, &bad);
    const long long ldk = bad || !n ? Hkv * D : call_int(K, s_stride, g_zero, &bad), ldv = bad || !n ? Hkv * D : call_int(V, s_stride, g_zero, &bad);
    const long long ws_n = bad ? 0 : call_int(ws, s_numel, NULL, &bad);
    if (bad) return NULL;
    const unsigned long long stream = PyLong_AsUnsignedLongLongMask(a[8]);
    if (stream == (unsigned long long)-1 && PyErr_Occurred()) return NULL;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = g_decode(qp, kp, vp, op, (float*)lp, ldq, ldk, ldv, ldo, (const int32_t*)cp, (int)qs[0], n, (int)qs[1], (int)Hkv, (int)D, (float)scale, code, wp,
                  (size_t)ws_n, (void*)(uintptr_t)stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

/* setup(address of dash_decode_attention, torch.bfloat16, torch.float32) */
static PyObject* py_setup(PyObject* self, PyObject* args) {
    (void)self;
    unsigned long long fn;
    PyObject *bf, *f;
    if (!PyArg_ParseTuple(args, "KOO", &fn, &bf, &f)) return NULL;
    Py_INCREF(bf); Py_INCREF(f);
    Py_XSETREF(g_bf16, bf);
    Py_XSETREF(g_f32, f);
    g_decode = (decode_fn)(uintptr_t)fn;
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"decode", (PyCFunction)(void (*)(void))py_decode, METH_FASTCALL, NULL}, {"setup", py_setup, METH_VARARGS, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__pycall(void) {
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_stride = PyUnicode_InternFromString("stride");
    s_numel = PyUnicode_InternFromString("numel");
    s_is_cuda = PyUnicode_InternFromString("is_cuda");
    s_shape = PyUnicode_InternFromString("shape");
    s_dtype = PyUnicode_InternFromString("dtype");
    g_zero = PyLong_FromLong(0);
    if (!s_data_ptr || !s_stride || !s_numel || !s_is_cuda || !s_shape || !s_dtype || !g_zero) return NULL;
    return PyModule_Create(&module);
}
