// The marshalling of hgf.linear_forward in native code: tensors to addresses, the current stream, the call.  The smallest layers take
// 4 us on the GPU, and a decode loop makes such calls one after the other: 512 -> 512, M = 4 took 10.5 us a call through ctypes, which
// the host spent on arguments, and takes 4.5 us now (one B200, calls back to back).
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/cuda/CUDAContext.h>

#include "../../include/hgf.h"

namespace {

decltype(&hgf_linear_forward) g_forward = nullptr;
decltype(&hgf_linear_forward_ln) g_forward_ln = nullptr;

// A tensor that is exactly one (or a Parameter); anything else answers through its own methods.
const at::Tensor *plain_tensor(PyObject *o) { return THPVariable_CheckExact(o) ? &THPVariable_Unpack(o) : nullptr; }

// A Python int, nothing that turns into one (TypeError: the caller goes through ctypes then, which takes ints alone, too).
bool integer(PyObject *o, unsigned long long *out) {
    if (!PyLong_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "int expected");
        return false;
    }
    *out = PyLong_AsUnsignedLongLongMask(o);
    return true;
}
bool method_value(PyObject *o, const char *name, unsigned long long *out) {
    PyObject *v = PyObject_CallMethod(o, name, nullptr);
    if (!v) return false;
    const bool ok = integer(v, out);
    Py_DECREF(v);
    return ok;
}
bool address(PyObject *o, void **out) {
    *out = nullptr;
    if (o == Py_None) return true;
    if (const at::Tensor *t = plain_tensor(o)) {
        *out = t->data_ptr();
        return true;
    }
    unsigned long long v = 0;
    if (!method_value(o, "data_ptr", &v)) return false;
    *out = reinterpret_cast<void *>(v);
    return true;
}
bool elements(PyObject *o, size_t *out) {
    if (const at::Tensor *t = plain_tensor(o)) {
        *out = (size_t)t->numel();
        return true;
    }
    unsigned long long v = 0;
    if (!method_value(o, "numel", &v)) return false;
    *out = (size_t)v;
    return true;
}
bool rows(PyObject *o, int64_t *out) {  // shape[0]
    const at::Tensor *t = plain_tensor(o);
    if (t && t->dim() > 0) {
        *out = t->size(0);
        return true;
    }
    PyObject *shape = PyObject_GetAttrString(o, "shape");
    PyObject *first = shape ? PySequence_GetItem(shape, 0) : nullptr;
    Py_XDECREF(shape);
    if (!first) return false;
    unsigned long long v = 0;
    const bool ok = integer(first, &v);
    *out = (int64_t)v;
    Py_DECREF(first);
    return ok;
}
bool integer(PyObject *o, int64_t *out) {
    unsigned long long v = 0;
    const bool ok = integer(o, &v);
    *out = (int64_t)v;
    return ok;
}

// linear_forward(x, packed, gamma, d_in, d_out, At, Bt, gate, y, workspace, flags, stream, ln_weight, ln_bias, eps, gate_group) -> status
PyObject *linear_forward(PyObject *, PyObject *const *a, Py_ssize_t n) try {
    if (n != 16) {
        PyErr_SetString(PyExc_TypeError, "linear_forward takes 16 arguments");
        return nullptr;
    }
    void *x, *packed, *At, *Bt, *gate, *y, *workspace, *ln_weight, *ln_bias, *stream;
    int64_t M, d_in, d_out, r = 0, flags, gate_group = 1;
    size_t workspace_bytes = 0;
    if (!rows(a[0], &M) || !address(a[0], &x) || !address(a[1], &packed) || !integer(a[3], &d_in) || !integer(a[4], &d_out) ||
        !address(a[5], &At) || !address(a[6], &Bt) || !address(a[7], &gate) || !address(a[8], &y) || !address(a[9], &workspace) ||
        !elements(a[9], &workspace_bytes) || !integer(a[10], &flags))
        return nullptr;
    if (a[5] != Py_None && !rows(a[5], &r)) return nullptr;
    const float gamma = (float)PyFloat_AsDouble(a[2]);
    if (PyErr_Occurred()) return nullptr;
    if (a[11] == Py_None) {
        stream = at::cuda::getCurrentCUDAStream().stream();
    } else {
        PyObject *s = PyObject_GetAttrString(a[11], "cuda_stream");
        if (!s) return nullptr;
        unsigned long long v = 0;
        const bool ok = integer(s, &v);
        Py_DECREF(s);
        if (!ok) return nullptr;
        stream = reinterpret_cast<void *>(v);
    }
    hgf_front_end fe = {};
    const bool front_end = a[12] != Py_None || a[15] != Py_None;
    if (front_end) {
        if (!address(a[12], &ln_weight) || !address(a[13], &ln_bias)) return nullptr;
        fe.ln_weight = (const float *)ln_weight;
        fe.ln_bias = (const float *)ln_bias;
        fe.eps = (float)PyFloat_AsDouble(a[14]);
        if (PyErr_Occurred() || (a[15] != Py_None && !integer(a[15], &gate_group))) return nullptr;
        fe.gate_group = gate_group ? gate_group : 1;
    }
    hgf_status st;
    Py_BEGIN_ALLOW_THREADS
    st = front_end ? g_forward_ln(x, M, packed, gamma, d_in, d_out, At, Bt, (int32_t)r, (const float *)gate, y, workspace, workspace_bytes, nullptr, &fe, (uint32_t)flags, stream)
                   : g_forward(x, M, packed, gamma, d_in, d_out, At, Bt, (int32_t)r, (const float *)gate, y, workspace, workspace_bytes, nullptr, (uint32_t)flags, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)st);
} catch (const std::exception &e) {  // (of torch: no device, a tensor without storage)
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
}

// bind(address of hgf_linear_forward, address of hgf_linear_forward_ln): in the library that hgf.lib() has loaded
PyObject *bind(PyObject *, PyObject *args) {
    unsigned long long forward, forward_ln;
    if (!PyArg_ParseTuple(args, "KK", &forward, &forward_ln)) return nullptr;
    g_forward = reinterpret_cast<decltype(g_forward)>(forward);
    g_forward_ln = reinterpret_cast<decltype(g_forward_ln)>(forward_ln);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"linear_forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(linear_forward)), METH_FASTCALL, nullptr},
                         {"bind", bind, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_hgf_python", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__hgf_python() { return PyModule_Create(&module); }
