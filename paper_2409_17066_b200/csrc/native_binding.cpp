// Argument marshalling of the calls a decode loop makes for every projection, as a CPython extension: tensors to pointers,
// the checks of binding.py, torch's current stream, and the C ABI call.  No arithmetic and no kernels.
//
// Why native: a small projection takes the GPU 2.6 us (256 x 512) and took the host 9.8 us per call, nearly all of it Python
// attribute look-ups, ctypes conversions and torch.cuda.current_stream().
#include <Python.h>

#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/vptq.h"

namespace {

PyObject *g_error_class = nullptr;       // binding.VptqError

// The memory of a ctypes structure (or array of them) of at least `bytes` bytes; it stays valid while the object lives.
template <typename T>
const T *struct_of(PyObject *o, Py_ssize_t count = 1)
{
    Py_buffer v;
    if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) != 0) return nullptr;
    const T *p = static_cast<const T *>(v.buf);
    const Py_ssize_t len = v.len;
    PyBuffer_Release(&v);
    if (len < count * (Py_ssize_t)sizeof(T)) {
        PyErr_SetString(PyExc_TypeError, "descriptor or pointer structure too small");
        return nullptr;
    }
    return p;
}

const at::Tensor *tensor_of(PyObject *o)
{
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "a torch tensor was expected");
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

PyObject *fail(int code)
{
    if (PyErr_Occurred()) return nullptr;
    PyObject *arg = PyLong_FromLong(code);
    PyObject *e = arg && g_error_class ? PyObject_CallOneArg(g_error_class, arg) : nullptr;
    if (e) {
        PyErr_SetObject(g_error_class, e);
        Py_DECREF(e);
    } else if (!PyErr_Occurred()) {
        PyErr_Format(PyExc_RuntimeError, "libvptq error %d", code);
    }
    Py_XDECREF(arg);
    return nullptr;
}

PyObject *assertion(const char *what)
{
    PyErr_SetString(PyExc_AssertionError, what);
    return nullptr;
}

at::ScalarType dtype_of(int32_t code)
{
    return code == VPTQ_DTYPE_FP16 ? at::kHalf : code == VPTQ_DTYPE_BF16 ? at::kBFloat16 : at::kFloat;
}

void *current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// workspace argument: a tensor or None
bool workspace_of(PyObject *o, void **p, size_t *bytes)
{
    *p = nullptr; *bytes = 0;
    if (o == Py_None) return true;
    const at::Tensor *t = tensor_of(o);
    if (!t) return false;
    *p = t->data_ptr();
    *bytes = (size_t)t->nbytes();
    return true;
}

// out = x * W^T for one layer; the checks are those binding.vptq_linear documents
PyObject *call_linear(const vptq_layer_desc *d, const at::Tensor &x, const vptq_layer_ptrs *p, const at::Tensor &out,
                      PyObject *out_obj, void *ws, size_t ws_bytes)
{
    if (!x.is_cuda() || !x.is_contiguous() || !out.is_cuda() || !out.is_contiguous()) return assertion("contiguous CUDA tensors");
    if (x.scalar_type() != dtype_of(d->x_dtype) || out.scalar_type() != dtype_of(d->out_dtype)) return assertion("dtypes of the descriptor");
    if (x.dim() != 2 || out.dim() != 2 || x.size(1) != d->N || out.size(0) != x.size(0) || out.size(1) != d->M)
        return assertion("x [B][N] and out [B][M]");
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = vptq_linear(d, x.data_ptr(), (int32_t)x.size(0), p, out.data_ptr(), ws, ws_bytes, current_stream());
    Py_END_ALLOW_THREADS
    if (rc != VPTQ_OK) return fail(rc);
    Py_INCREF(out_obj);
    return out_obj;
}

// linear(desc, x, ptrs, out, workspace) -> out
PyObject *py_linear(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 5) { PyErr_SetString(PyExc_TypeError, "linear takes 5 arguments"); return nullptr; }
    const vptq_layer_desc *d = struct_of<vptq_layer_desc>(a[0]);
    const at::Tensor *x = d ? tensor_of(a[1]) : nullptr;
    const vptq_layer_ptrs *p = x ? struct_of<vptq_layer_ptrs>(a[2]) : nullptr;
    const at::Tensor *out = p ? tensor_of(a[3]) : nullptr;
    void *ws;
    size_t ws_bytes;
    if (!out || !workspace_of(a[4], &ws, &ws_bytes)) return nullptr;
    return call_linear(d, *x, p, *out, a[3], ws, ws_bytes);
}

// layer_linear(desc, ptrs, workspaces, x, out or None) -> out, or None when `workspaces` (a dict by batch size) has no entry
// for the batch of x
PyObject *py_layer_linear(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 5) { PyErr_SetString(PyExc_TypeError, "layer_linear takes 5 arguments"); return nullptr; }
    const vptq_layer_desc *d = struct_of<vptq_layer_desc>(a[0]);
    const vptq_layer_ptrs *p = d ? struct_of<vptq_layer_ptrs>(a[1]) : nullptr;
    const at::Tensor *x = p ? tensor_of(a[3]) : nullptr;
    if (!x) return nullptr;
    if (x->dim() != 2) return assertion("x [B][N] and out [B][M]");
    PyObject *key = PyLong_FromLongLong(x->size(0));
    PyObject *w = key ? PyDict_GetItemWithError(a[2], key) : nullptr;
    Py_XDECREF(key);
    if (!w) {
        if (PyErr_Occurred()) return nullptr;
        Py_RETURN_NONE;
    }
    void *ws;
    size_t ws_bytes;
    if (!workspace_of(w, &ws, &ws_bytes)) return nullptr;
    if (a[4] != Py_None) {
        const at::Tensor *out = tensor_of(a[4]);
        return out ? call_linear(d, *x, p, *out, a[4], ws, ws_bytes) : nullptr;
    }
    PyObject *out_obj = nullptr;
    try {
        out_obj = THPVariable_Wrap(at::empty({x->size(0), d->M}, x->options().dtype(dtype_of(d->out_dtype))));
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    if (!out_obj) return nullptr;
    PyObject *r = call_linear(d, *x, p, THPVariable_Unpack(out_obj), out_obj, ws, ws_bytes);
    Py_DECREF(out_obj);
    return r;
}

// fused_linear(descs, ptrs, n, workspaces, x, outs) -> outs, or None when `workspaces` has no entry for the batch of x
PyObject *py_fused_linear(PyObject *, PyObject *const *a, Py_ssize_t n_args)
{
    if (n_args != 6) { PyErr_SetString(PyExc_TypeError, "fused_linear takes 6 arguments"); return nullptr; }
    const long n = PyLong_AsLong(a[2]);
    if (n < 1 || n > VPTQ_MAX_FUSED_LAYERS) return PyErr_Occurred() ? nullptr : fail(VPTQ_E_SHAPE);
    const vptq_layer_desc *d = struct_of<vptq_layer_desc>(a[0], n);
    const vptq_layer_ptrs *p = d ? struct_of<vptq_layer_ptrs>(a[1], n) : nullptr;
    const at::Tensor *x = p ? tensor_of(a[4]) : nullptr;
    if (!x) return nullptr;
    PyObject *key = PyLong_FromLongLong(x->size(0));
    PyObject *w = key ? PyDict_GetItemWithError(a[3], key) : nullptr;
    Py_XDECREF(key);
    if (!w) {
        if (PyErr_Occurred()) return nullptr;
        Py_RETURN_NONE;
    }
    void *ws;
    size_t ws_bytes;
    if (!workspace_of(w, &ws, &ws_bytes)) return nullptr;
    PyObject *outs = PySequence_Fast(a[5], "a sequence of output tensors was expected");
    if (!outs) return nullptr;
    void *op[VPTQ_MAX_FUSED_LAYERS];
    bool ok = PySequence_Fast_GET_SIZE(outs) == n;
    if (!ok) PyErr_SetString(PyExc_ValueError, "one output tensor per layer");
    for (long i = 0; ok && i < n; i++) {
        const at::Tensor *t = tensor_of(PySequence_Fast_GET_ITEM(outs, i));
        ok = t != nullptr;
        if (ok) op[i] = t->data_ptr();
    }
    Py_DECREF(outs);
    if (!ok) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = vptq_linear_fused(d, p, (int32_t)n, x->data_ptr(), (int32_t)x->size(0), op, ws, ws_bytes, current_stream());
    Py_END_ALLOW_THREADS
    if (rc != VPTQ_OK) return fail(rc);
    Py_INCREF(a[5]);
    return a[5];
}

// dequant(desc, ptrs, W_out) -> W_out (a restored 256 x 256 weight: 11.8 us a call through ctypes, all of it host time)
PyObject *py_dequant(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (n != 3) { PyErr_SetString(PyExc_TypeError, "dequant takes 3 arguments"); return nullptr; }
    const vptq_layer_desc *d = struct_of<vptq_layer_desc>(a[0]);
    const vptq_layer_ptrs *p = d ? struct_of<vptq_layer_ptrs>(a[1]) : nullptr;
    const at::Tensor *w = p ? tensor_of(a[2]) : nullptr;
    if (!w) return nullptr;
    if (!w->is_cuda() || !w->is_contiguous() || w->scalar_type() != at::kHalf) return assertion("a contiguous FP16 CUDA tensor");
    if (w->dim() != 2 || w->size(0) != d->M || w->size(1) != d->N) return assertion("W_out [M][N]");
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = vptq_dequant(d, p, w->data_ptr(), current_stream());
    Py_END_ALLOW_THREADS
    if (rc != VPTQ_OK) return fail(rc);
    Py_INCREF(a[2]);
    return a[2];
}

PyObject *py_set_error_class(PyObject *, PyObject *cls)
{
    Py_INCREF(cls);
    Py_XSETREF(g_error_class, cls);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_linear)), METH_FASTCALL, "vptq_linear on torch tensors"},
    {"dequant", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_dequant)), METH_FASTCALL, "vptq_dequant on torch tensors"},
    {"layer_linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_layer_linear)), METH_FASTCALL, "DeviceLayer.linear"},
    {"fused_linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_fused_linear)), METH_FASTCALL, "FusedLayers.linear"},
    {"set_error_class", py_set_error_class, METH_O, "exception raised for VPTQ_E_* codes"},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
