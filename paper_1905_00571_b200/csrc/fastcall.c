/*
 * Native argument marshalling of the calls a program makes per layer or per image (cadnn_conv2d, cadnn_fc, cadnn_forward,
 * cadnn_forward_host): reads pointers and shapes off the tensor objects and calls the C ABI.  Through ctypes the
 * marshalling of one layer call took about 6 microseconds, more than the smallest kernels run; here it takes under one.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <limits.h>
#include "cadnn.h"

static PyObject *g_check, *g_act, *g_dtype;            /* binding._check, binding.ACT, binding.DTYPE */
static PyObject *g_get_device, *g_raw_stream;          /* torch._C._cuda_getDevice / _cuda_getCurrentRawStream */
static PyObject *s_dtype, *s_data_ptr, *s_shape, *s_cuda_stream, *s_handle, *s_value, *s_ctypes, *s_data;

/* args / keywords -> out[0 .. n), NULL where not given */
static int parse(PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames, const char *const *names, int n, int required, PyObject **out)
{
    if (nargs > n) {
        PyErr_Format(PyExc_TypeError, "takes at most %d arguments (%zd given)", n, nargs);
        return -1;
    }
    for (int i = 0; i < n; ++i) out[i] = i < nargs ? args[i] : NULL;
    const Py_ssize_t nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
    for (Py_ssize_t k = 0; k < nk; ++k) {
        PyObject *name = PyTuple_GET_ITEM(kwnames, k);
        int i = 0;
        while (i < n && PyUnicode_CompareWithASCIIString(name, names[i]) != 0) ++i;
        if (i == n || out[i]) {
            PyErr_Format(PyExc_TypeError, i == n ? "unexpected keyword argument '%U'" : "multiple values for argument '%U'", name);
            return -1;
        }
        out[i] = args[nargs + k];
    }
    for (int i = 0; i < required; ++i)
        if (!out[i]) {
            PyErr_Format(PyExc_TypeError, "missing argument '%s'", names[i]);
            return -1;
        }
    return 0;
}

/* (the C ABI takes int: what does not fit is refused, not cut) */
static int as_int(PyObject *o, int dflt, int *v)
{
    if (!o) { *v = dflt; return 0; }
    const long l = PyLong_AsLong(o);
    if (l == -1 && PyErr_Occurred()) return -1;
    if (l < INT_MIN || l > INT_MAX) {
        PyErr_Format(PyExc_OverflowError, "%ld does not fit a C int", l);
        return -1;
    }
    *v = (int)l;
    return 0;
}

/* device pointer of a tensor (None = NULL) */
static int tensor_ptr(PyObject *t, void **p)
{
    *p = NULL;
    if (!t || t == Py_None) return 0;
    PyObject *r = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!r) return -1;
    *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

/* the handle of a Weights / Net object (NULL once freed) */
static int handle_ptr(PyObject *w, void **p)
{
    *p = NULL;
    PyObject *h = PyObject_GetAttr(w, s_handle);
    if (!h) return -1;
    if (h != Py_None) {
        PyObject *v = PyObject_GetAttr(h, s_value);
        if (!v) { Py_DECREF(h); return -1; }
        if (v != Py_None) *p = PyLong_AsVoidPtr(v);
        Py_DECREF(v);
    }
    Py_DECREF(h);
    return PyErr_Occurred() ? -1 : 0;
}

static int shape_dims(PyObject *t, int *d, int want)
{
    PyObject *s = PyObject_GetAttr(t, s_shape);
    if (!s) return -1;
    PyObject *f = PySequence_Fast(s, "shape is not a sequence");
    Py_DECREF(s);
    if (!f) return -1;
    if (PySequence_Fast_GET_SIZE(f) < want) {
        PyErr_SetString(PyExc_IndexError, "tensor has too few dimensions");
        Py_DECREF(f);
        return -1;
    }
    for (int i = 0; i < want; ++i)
        if (as_int(PySequence_Fast_GET_ITEM(f, i), 0, &d[i])) { Py_DECREF(f); return -1; }
    Py_DECREF(f);
    return 0;
}

static int stream_ptr(PyObject *o, void **p)
{
    if (o && o != Py_None) {
        PyObject *v = PyObject_GetAttr(o, s_cuda_stream);
        if (!v) {
            if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
            PyErr_Clear();
            v = PyNumber_Long(o);
            if (!v) return -1;
        }
        *p = PyLong_AsVoidPtr(v);
        Py_DECREF(v);
        return PyErr_Occurred() ? -1 : 0;
    }
    if (!g_raw_stream) {   /* torch's current stream on the current device */
        PyObject *torch = PyImport_ImportModule("torch");   /* the public module: initialises torch._C */
        PyObject *m = torch ? PyImport_ImportModule("torch._C") : NULL;
        PyObject *cuda = m ? PyImport_ImportModule("torch.cuda") : NULL;
        PyObject *r = cuda ? PyObject_CallMethod(cuda, "current_stream", NULL) : NULL;   /* initialises CUDA */
        if (r) {
            Py_DECREF(r);
            g_get_device = PyObject_GetAttrString(m, "_cuda_getDevice");
            if (g_get_device) g_raw_stream = PyObject_GetAttrString(m, "_cuda_getCurrentRawStream");
        }
        Py_XDECREF(cuda); Py_XDECREF(m); Py_XDECREF(torch);
        if (!g_raw_stream) return -1;
    }
    PyObject *dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return -1;
    PyObject *r = PyObject_CallOneArg(g_raw_stream, dev);
    Py_DECREF(dev);
    if (!r) return -1;
    *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

/* dictionary code of a name (or the number itself) */
static int code_of(PyObject *dict, PyObject *o, int *v)
{
    if (PyLong_Check(o)) return as_int(o, 0, v);
    PyObject *c = PyObject_GetItem(dict, o);
    if (!c) return -1;
    const int rc = as_int(c, 0, v);
    Py_DECREF(c);
    return rc;
}

/* y on success; raises through binding._check otherwise */
static PyObject *result(int st, const char *where, PyObject *y)
{
    if (st != CADNN_OK) {
        PyObject *r = PyObject_CallFunction(g_check, "is", st, where);
        Py_XDECREF(r);
        if (!r) return NULL;
    }
    Py_INCREF(y);
    return y;
}

/* the epilogue's part of a layer call: scale, bias, residual, act, out_dtype at a[0 .. 5) */
static int epilogue_of(PyObject *w, PyObject **a, cadnn_epilogue *ep)
{
    void *p;
    if (tensor_ptr(a[0], &p)) return -1;
    ep->scale = (const float *)p;
    if (tensor_ptr(a[1], &p)) return -1;
    ep->bias = (const float *)p;
    if (tensor_ptr(a[2], &p)) return -1;
    ep->residual = p;
    ep->act = CADNN_ACT_NONE;
    if (a[3] && code_of(g_act, a[3], &ep->act)) return -1;
    if (a[4] && a[4] != Py_None) return code_of(g_dtype, a[4], &ep->out_dtype);
    PyObject *d = PyObject_GetAttrString(w, "desc");   /* the layer's own type */
    if (!d) return -1;
    PyObject *t = PyObject_GetAttr(d, s_dtype);
    Py_DECREF(d);
    if (!t) return -1;
    const int rc = as_int(t, 0, &ep->out_dtype);
    Py_DECREF(t);
    return rc;
}

static PyObject *conv2d(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    static const char *const names[] = {"w", "x", "y", "scale", "bias", "residual", "act", "out_dtype", "stream", "out_c_total",
                                        "out_c_off", "residual_scale"};
    PyObject *a[12];
    void *w, *x, *y, *st;
    int d[3];
    cadnn_epilogue ep = {0};
    if (parse(args, nargs, kwnames, names, 12, 3, a) || shape_dims(a[1], d, 3) || handle_ptr(a[0], &w) || tensor_ptr(a[1], &x) ||
        tensor_ptr(a[2], &y) || epilogue_of(a[0], a + 3, &ep) || stream_ptr(a[8], &st) || as_int(a[9], 0, &ep.out_c_total) ||
        as_int(a[10], 0, &ep.out_c_off))
        return NULL;
    if (a[11]) {
        const double r = PyFloat_AsDouble(a[11]);
        if (r == -1.0 && PyErr_Occurred()) return NULL;
        ep.residual_scale = (float)r;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = cadnn_conv2d((const cadnn_weights *)w, x, d[0], d[1], d[2], y, &ep, st);
    Py_END_ALLOW_THREADS
    return result(rc, "cadnn_conv2d", a[2]);
}

static PyObject *fc(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    static const char *const names[] = {"w", "x", "y", "scale", "bias", "residual", "act", "out_dtype", "stream"};
    PyObject *a[9];
    void *w, *x, *y, *st;
    int n;
    cadnn_epilogue ep = {0};
    if (parse(args, nargs, kwnames, names, 9, 3, a) || shape_dims(a[1], &n, 1) || handle_ptr(a[0], &w) || tensor_ptr(a[1], &x) ||
        tensor_ptr(a[2], &y) || epilogue_of(a[0], a + 3, &ep) || stream_ptr(a[8], &st))
        return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = cadnn_fc((const cadnn_weights *)w, x, n, y, &ep, st);
    Py_END_ALLOW_THREADS
    return result(rc, "cadnn_fc", a[2]);
}

static PyObject *forward(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    static const char *const names[] = {"net", "x", "y", "use_graph", "stream"};
    PyObject *a[5];
    void *net, *x, *y, *st;
    if (parse(args, nargs, kwnames, names, 5, 3, a) || handle_ptr(a[0], &net) || tensor_ptr(a[1], &x) || tensor_ptr(a[2], &y) ||
        stream_ptr(a[4], &st))
        return NULL;
    const int graph = a[3] ? PyObject_IsTrue(a[3]) : 1;
    if (graph < 0) return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = cadnn_forward((cadnn_net *)net, x, y, graph, st);
    Py_END_ALLOW_THREADS
    return result(rc, "cadnn_forward", a[2]);
}

/* host buffer of a CPU torch tensor or a numpy array */
static int host_ptr(PyObject *t, void **p)
{
    PyObject *r = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (!r) {
        if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return -1;
        PyErr_Clear();
        PyObject *c = PyObject_GetAttr(t, s_ctypes);
        if (!c) return -1;
        r = PyObject_GetAttr(c, s_data);
        Py_DECREF(c);
        if (!r) return -1;
    }
    *p = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return PyErr_Occurred() ? -1 : 0;
}

static PyObject *forward_host(PyObject *self, PyObject *const *args, Py_ssize_t nargs, PyObject *kwnames)
{
    static const char *const names[] = {"net", "x_host", "y_host", "use_graph", "stream"};
    PyObject *a[5];
    void *net, *x, *y, *st;
    if (parse(args, nargs, kwnames, names, 5, 3, a) || handle_ptr(a[0], &net) || host_ptr(a[1], &x) || host_ptr(a[2], &y) ||
        stream_ptr(a[4], &st))
        return NULL;
    const int graph = a[3] ? PyObject_IsTrue(a[3]) : 1;
    if (graph < 0) return NULL;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = cadnn_forward_host((cadnn_net *)net, x, y, graph, st);
    Py_END_ALLOW_THREADS
    return result(rc, "cadnn_forward_host", a[2]);
}

static PyObject *setup(PyObject *self, PyObject *args)
{
    PyObject *check, *act, *dtype;
    if (!PyArg_ParseTuple(args, "OOO", &check, &act, &dtype)) return NULL;
    Py_INCREF(check); Py_INCREF(act); Py_INCREF(dtype);
    Py_XSETREF(g_check, check);
    Py_XSETREF(g_act, act);
    Py_XSETREF(g_dtype, dtype);
    Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"cadnn_conv2d", (PyCFunction)(void (*)(void))conv2d, METH_FASTCALL | METH_KEYWORDS,
     "cadnn_conv2d(w, x, y, scale=None, bias=None, residual=None, act='none', out_dtype=None, stream=None, out_c_total=0, out_c_off=0, "
     "residual_scale=0.0)\n\nx, y: torch CUDA tensors, NHWC contiguous; y is written in place (channels [out_c_off, out_c_off + c_out)\n"
     "of it when out_c_total > 0) and returned."},
    {"cadnn_fc", (PyCFunction)(void (*)(void))fc, METH_FASTCALL | METH_KEYWORDS,
     "cadnn_fc(w, x, y, scale=None, bias=None, residual=None, act='none', out_dtype=None, stream=None)\n\nx [n, c_in], y [n, c_out]: torch "
     "CUDA tensors; y is written in place and returned."},
    {"cadnn_forward", (PyCFunction)(void (*)(void))forward, METH_FASTCALL | METH_KEYWORDS,
     "cadnn_forward(net, x, y, use_graph=True, stream=None)\n\nRuns the network on CUDA tensor x into y; returns y."},
    {"cadnn_forward_host", (PyCFunction)(void (*)(void))forward_host, METH_FASTCALL | METH_KEYWORDS,
     "cadnn_forward_host(net, x_host, y_host, use_graph=True, stream=None)\n\nx_host, y_host: CPU torch tensors (pinned recommended) or numpy "
     "arrays; blocks until y_host is filled."},
    {"setup", setup, METH_VARARGS, "setup(check, act_codes, dtype_codes): called once by the binding."},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", "Native marshalling of the per-call entry points.", -1, methods};

PyMODINIT_FUNC PyInit__fastcall(void)
{
    s_dtype = PyUnicode_InternFromString("dtype");
    s_data_ptr = PyUnicode_InternFromString("data_ptr");
    s_shape = PyUnicode_InternFromString("shape");
    s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
    s_handle = PyUnicode_InternFromString("handle");
    s_value = PyUnicode_InternFromString("value");
    s_ctypes = PyUnicode_InternFromString("ctypes");
    s_data = PyUnicode_InternFromString("data");
    return PyModule_Create(&module);
}
