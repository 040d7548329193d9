// CPython module `_native`: what a step call does on the host between Python and the C ABI, in one native call.
//
// A program that hands over nested lists of gradient tensors pays per tensor and step: dtype, size, layout and
// address read through Python attributes cost 0.37 us a tensor (95 us for 256 workers with one tensor each, where
// the GPU's part of the step is 5 us), here about 0.02 us.  Arguments, torch's current stream and the call itself add 1 us
// instead of 3.  No arithmetic, no checks beyond those of module.py, nothing kept from one call for the next but the
// buffer that the pointers are written to.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>
#include <exception>
#include <new>
#include <vector>

#include "../../include/desloc.h"

namespace {

// The library is loaded by the ctypes binding; its entry points arrive as addresses.
struct Entry {
    decltype(&desloc_step) step = nullptr;
    decltype(&desloc_step_masked) step_masked = nullptr;
    decltype(&desloc_step_normclip) step_normclip = nullptr;
    decltype(&desloc_step_diag) step_diag = nullptr;
    decltype(&desloc_rel_change) rel_change = nullptr;
    decltype(&desloc_get_diag_norms) diag_norms = nullptr;
    decltype(&desloc_step_host) step_host = nullptr;
} g_entry;

struct Table {
    PyObject_HEAD
    std::vector<int64_t> *numel;
    std::vector<void *> *ptrs;
    Py_ssize_t workers;
};

PyObject *table_new(PyTypeObject *type, PyObject *args, PyObject *) {
    PyObject *numel = nullptr;
    Py_ssize_t workers = 0;
    if (!PyArg_ParseTuple(args, "On", &numel, &workers)) return nullptr;
    PyObject *seq = PySequence_Fast(numel, "numel must be a sequence");
    if (!seq) return nullptr;
    Table *self = reinterpret_cast<Table *>(type->tp_alloc(type, 0));
    bool ok = self != nullptr;
    if (ok) {
        const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
        self->workers = workers;
        self->numel = new (std::nothrow) std::vector<int64_t>();
        self->ptrs = new (std::nothrow) std::vector<void *>();
        try {
            if (!self->numel || !self->ptrs || workers < 0) throw std::bad_alloc();
            self->ptrs->resize(static_cast<size_t>(n) * workers);
            for (Py_ssize_t i = 0; ok && i < n; ++i) {
                const long long v = PyLong_AsLongLong(PySequence_Fast_GET_ITEM(seq, i));
                ok = !(v == -1 && PyErr_Occurred());
                self->numel->push_back(v);
            }
        } catch (const std::bad_alloc &) {
            PyErr_NoMemory();
            ok = false;
        }
    }
    Py_DECREF(seq);
    if (!ok) {
        Py_XDECREF(reinterpret_cast<PyObject *>(self));
        return nullptr;
    }
    return reinterpret_cast<PyObject *>(self);
}

void table_dealloc(PyObject *o) {
    Table *self = reinterpret_cast<Table *>(o);
    delete self->numel;
    delete self->ptrs;
    Py_TYPE(o)->tp_free(o);
}

bool as_pointer(PyObject *o, void **out) {
    *out = o == Py_None ? nullptr : PyLong_AsVoidPtr(o);
    return !(*out == nullptr && PyErr_Occurred());
}

// fill(nested, kind, where, message) -> address of the pointer array [workers * tensors], row m = worker m.
// kind: 0 = fp32, 1 = bf16.  where: 0 = any device, 1 = host only.  A tensor that does not fit raises
// ValueError(message).  Returns None at the first element that is no torch.Tensor: the caller marshals the lists then.
PyObject *table_fill(PyObject *o, PyObject *const *args, Py_ssize_t nargs) {
    Table *self = reinterpret_cast<Table *>(o);
    if (nargs != 4) {
        PyErr_SetString(PyExc_TypeError, "fill(nested, kind, where, message)");
        return nullptr;
    }
    const long kind = PyLong_AsLong(args[1]), where = PyLong_AsLong(args[2]);
    if (PyErr_Occurred()) return nullptr;
    const at::ScalarType want = kind == 1 ? at::kBFloat16 : at::kFloat;
    const Py_ssize_t nt = static_cast<Py_ssize_t>(self->numel->size());
    const size_t room = self->ptrs->size();
    PyObject *rows = PySequence_Fast(args[0], "need one tensor list per worker");
    if (!rows) return nullptr;
    size_t count = 0;
    enum { OK, UNFIT, FOREIGN, FAILED } state = OK;
    try {
        for (Py_ssize_t m = 0; state == OK && m < PySequence_Fast_GET_SIZE(rows); ++m) {
            PyObject *row = PySequence_Fast(PySequence_Fast_GET_ITEM(rows, m), "need one tensor list per worker");
            if (!row) {
                state = FAILED;
                break;
            }
            for (Py_ssize_t k = 0; state == OK && k < nt && k < PySequence_Fast_GET_SIZE(row); ++k) {
                PyObject *item = PySequence_Fast_GET_ITEM(row, k);
                if (!THPVariable_Check(item)) {
                    state = FOREIGN;
                    break;
                }
                const at::Tensor &t = THPVariable_Unpack(item);
                if (t.scalar_type() != want || t.numel() != (*self->numel)[k] || !t.is_contiguous() ||
                    (where == 1 && t.is_cuda())) {
                    state = UNFIT;
                    break;
                }
                if (count < room) (*self->ptrs)[count] = t.data_ptr();
                ++count;
            }
            Py_DECREF(row);
        }
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        state = FAILED;
    }
    Py_DECREF(rows);
    if (state == FAILED) return nullptr;
    if (state == FOREIGN) Py_RETURN_NONE;
    if (state == UNFIT) {
        PyErr_SetObject(PyExc_ValueError, args[3]);
        return nullptr;
    }
    if (count != room) {
        PyErr_SetString(PyExc_ValueError, "need one gradient list per worker");
        return nullptr;
    }
    return PyLong_FromVoidPtr(self->ptrs->data());
}

// set(addresses) -> address of the pointer array, which holds them now: for what fill() leaves to the caller.
PyObject *table_set(PyObject *o, PyObject *list) {
    Table *self = reinterpret_cast<Table *>(o);
    PyObject *seq = PySequence_Fast(list, "addresses must be a sequence");
    if (!seq) return nullptr;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    bool ok = static_cast<size_t>(n) == self->ptrs->size();
    if (!ok) PyErr_SetString(PyExc_ValueError, "need one address per worker and tensor");
    for (Py_ssize_t i = 0; ok && i < n; ++i) ok = as_pointer(PySequence_Fast_GET_ITEM(seq, i), &(*self->ptrs)[i]);
    Py_DECREF(seq);
    return ok ? PyLong_FromVoidPtr(self->ptrs->data()) : nullptr;
}

PyMethodDef table_methods[] = {
    {"set", table_set, METH_O, nullptr},
    {"fill", reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(table_fill)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyTypeObject table_type = {PyVarObject_HEAD_INIT(nullptr, 0)};

// ---- step calls -----------------------------------------------------------------------------------
bool as_int64(PyObject *o, int64_t *out) {
    PyObject *n = PyNumber_Long(o);
    if (!n) return false;
    *out = PyLong_AsLongLong(n);
    Py_DECREF(n);
    return !(*out == -1 && PyErr_Occurred());
}
bool as_float(PyObject *o, float *out) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) return false;
    *out = static_cast<float>(v);
    return true;
}

// (context, t, lr, clip bound, max_norm, pointer array, device, which) -> sync mask, or a negative status.
// which: 0 = step, 1 = step_normclip, 2 = step_diag.  Runs on torch's current stream of the device.
PyObject *call_step(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
    void *ctx = nullptr, *ptrs = nullptr;
    int64_t t = 0, device = 0, which = 0;
    float lr = 0.f, bound = 0.f, max_norm = 0.f;
    if (nargs != 8) {
        PyErr_SetString(PyExc_TypeError, "step(ctx, t, lr, clip_bound, max_norm, grads, device, which)");
        return nullptr;
    }
    if (!as_pointer(args[0], &ctx) || !as_int64(args[1], &t) || !as_float(args[2], &lr) || !as_float(args[3], &bound) ||
        !as_float(args[4], &max_norm) || !as_pointer(args[5], &ptrs) || !as_int64(args[6], &device) ||
        !as_int64(args[7], &which))
        return nullptr;
    const void *const *g = static_cast<const void *const *>(ptrs);
    desloc_ctx *c = static_cast<desloc_ctx *>(ctx);
    uint32_t mask = 0;
    int rc = 0;
    try {
        void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device)).stream();
        Py_BEGIN_ALLOW_THREADS
        if (which == 0) rc = g_entry.step(c, t, lr, bound, g, stream, &mask);
        else if (which == 1) rc = g_entry.step_normclip(c, t, lr, bound, max_norm, g, stream, &mask);
        else rc = g_entry.step_diag(c, t, lr, bound, max_norm, g, stream, &mask);
        Py_END_ALLOW_THREADS
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
    return PyLong_FromLong(rc == DESLOC_OK ? static_cast<long>(mask) : rc);
}

// (context, mask, lr, clip bound, pointer array, device) -> status
PyObject *call_step_masked(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
    void *ctx = nullptr, *ptrs = nullptr;
    int64_t mask = 0, device = 0;
    float lr = 0.f, bound = 0.f;
    if (nargs != 6) {
        PyErr_SetString(PyExc_TypeError, "step_masked(ctx, mask, lr, clip_bound, grads, device)");
        return nullptr;
    }
    if (!as_pointer(args[0], &ctx) || !as_int64(args[1], &mask) || !as_float(args[2], &lr) || !as_float(args[3], &bound) ||
        !as_pointer(args[4], &ptrs) || !as_int64(args[5], &device))
        return nullptr;
    int rc = 0;
    try {
        void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device)).stream();
        Py_BEGIN_ALLOW_THREADS
        rc = g_entry.step_masked(static_cast<desloc_ctx *>(ctx), static_cast<uint32_t>(mask), lr, bound,
                                 static_cast<const void *const *>(ptrs), stream);
        Py_END_ALLOW_THREADS
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
    return PyLong_FromLong(rc);
}

// (context, t, lr, clip bound, host pointer array, device pointer array, device) -> sync mask, or a negative status
PyObject *call_step_host(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
    void *ctx = nullptr, *from = nullptr, *to = nullptr;
    int64_t t = 0, device = 0;
    float lr = 0.f, bound = 0.f;
    if (nargs != 7) {
        PyErr_SetString(PyExc_TypeError, "step_host(ctx, t, lr, clip_bound, host_grads, dev_grads, device)");
        return nullptr;
    }
    if (!as_pointer(args[0], &ctx) || !as_int64(args[1], &t) || !as_float(args[2], &lr) || !as_float(args[3], &bound) ||
        !as_pointer(args[4], &from) || !as_pointer(args[5], &to) || !as_int64(args[6], &device))
        return nullptr;
    uint32_t mask = 0;
    int rc = 0;
    try {
        void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device)).stream();
        Py_BEGIN_ALLOW_THREADS
        rc = g_entry.step_host(static_cast<desloc_ctx *>(ctx), t, lr, bound, static_cast<const void *const *>(from),
                               static_cast<void *const *>(to), stream, &mask);
        Py_END_ALLOW_THREADS
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
    return PyLong_FromLong(rc == DESLOC_OK ? static_cast<long>(mask) : rc);
}

// A list of n floats.
PyObject *float_list(const float *v, size_t n) {
    PyObject *list = PyList_New(static_cast<Py_ssize_t>(n));
    for (size_t i = 0; list && i < n; ++i) {
        PyObject *f = PyFloat_FromDouble(v[i]);
        if (!f) {
            Py_CLEAR(list);
            break;
        }
        PyList_SET_ITEM(list, static_cast<Py_ssize_t>(i), f);
    }
    return list;
}

// (context, array, pointer array, device, workers) -> list of floats, or a negative status
PyObject *call_rel_change(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
    void *ctx = nullptr, *ptrs = nullptr;
    int64_t array = 0, device = 0, workers = 0;
    if (nargs != 5) {
        PyErr_SetString(PyExc_TypeError, "rel_change(ctx, array, then, device, workers)");
        return nullptr;
    }
    if (!as_pointer(args[0], &ctx) || !as_int64(args[1], &array) || !as_pointer(args[2], &ptrs) ||
        !as_int64(args[3], &device) || !as_int64(args[4], &workers))
        return nullptr;
    int rc = 0;
    std::vector<float> out;
    try {
        out.resize(static_cast<size_t>(workers));
        void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device)).stream();
        Py_BEGIN_ALLOW_THREADS
        rc = g_entry.rel_change(static_cast<desloc_ctx *>(ctx), static_cast<int32_t>(array),
                                static_cast<const float *const *>(ptrs), out.data(), stream);
        Py_END_ALLOW_THREADS
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
    if (rc != DESLOC_OK) return PyLong_FromLong(rc);
    return float_list(out.data(), out.size());
}

// (context, workers, tensors, device) -> ([3][workers][tensors], [3][workers]) as nested lists, or a negative status
PyObject *call_diag_norms(PyObject *, PyObject *const *args, Py_ssize_t nargs) {
    void *ctx = nullptr;
    int64_t workers = 0, tensors = 0, device = 0;
    if (nargs != 4) {
        PyErr_SetString(PyExc_TypeError, "diag_norms(ctx, workers, tensors, device)");
        return nullptr;
    }
    if (!as_pointer(args[0], &ctx) || !as_int64(args[1], &workers) || !as_int64(args[2], &tensors) ||
        !as_int64(args[3], &device))
        return nullptr;
    int rc = 0;
    std::vector<float> per, tot;
    try {
        per.resize(static_cast<size_t>(3 * workers * tensors));
        tot.resize(static_cast<size_t>(3 * workers));
        void *stream = c10::cuda::getCurrentCUDAStream(static_cast<c10::DeviceIndex>(device)).stream();
        Py_BEGIN_ALLOW_THREADS
        rc = g_entry.diag_norms(static_cast<desloc_ctx *>(ctx), per.data(), tot.data(), stream);
        Py_END_ALLOW_THREADS
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
    if (rc != DESLOC_OK) return PyLong_FromLong(rc);
    PyObject *a = PyList_New(3), *b = PyList_New(3);
    bool ok = a && b;
    for (int k = 0; ok && k < 3; ++k) {
        PyObject *rows = PyList_New(static_cast<Py_ssize_t>(workers)), *t = float_list(tot.data() + k * workers, workers);
        ok = rows && t;
        for (int64_t m = 0; ok && m < workers; ++m) {
            PyObject *row = float_list(per.data() + (k * workers + m) * tensors, tensors);
            ok = row != nullptr;
            if (ok) PyList_SET_ITEM(rows, static_cast<Py_ssize_t>(m), row);
        }
        if (ok) {
            PyList_SET_ITEM(a, k, rows);
            PyList_SET_ITEM(b, k, t);
        } else {
            Py_XDECREF(rows);
            Py_XDECREF(t);
        }
    }
    PyObject *both = ok ? PyTuple_Pack(2, a, b) : nullptr;
    Py_XDECREF(a);
    Py_XDECREF(b);
    return both;
}

// bind(addresses of desloc_step, _step_masked, _step_normclip, _step_diag, _rel_change, _get_diag_norms, _step_host)
PyObject *bind_entries(PyObject *, PyObject *args) {
    unsigned long long a[7];
    if (!PyArg_ParseTuple(args, "KKKKKKK", &a[0], &a[1], &a[2], &a[3], &a[4], &a[5], &a[6])) return nullptr;
    g_entry.step = reinterpret_cast<decltype(g_entry.step)>(a[0]);
    g_entry.step_masked = reinterpret_cast<decltype(g_entry.step_masked)>(a[1]);
    g_entry.step_normclip = reinterpret_cast<decltype(g_entry.step_normclip)>(a[2]);
    g_entry.step_diag = reinterpret_cast<decltype(g_entry.step_diag)>(a[3]);
    g_entry.rel_change = reinterpret_cast<decltype(g_entry.rel_change)>(a[4]);
    g_entry.diag_norms = reinterpret_cast<decltype(g_entry.diag_norms)>(a[5]);
    g_entry.step_host = reinterpret_cast<decltype(g_entry.step_host)>(a[6]);
    Py_RETURN_NONE;
}

template <typename F>
PyCFunction fast(F f) {
    return reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(f));
}

PyMethodDef methods[] = {{"bind", bind_entries, METH_VARARGS, nullptr},
                         {"step", fast(call_step), METH_FASTCALL, nullptr},
                         {"step_masked", fast(call_step_masked), METH_FASTCALL, nullptr},
                         {"step_host", fast(call_step_host), METH_FASTCALL, nullptr},
                         {"diag_norms", fast(call_diag_norms), METH_FASTCALL, nullptr},
                         {"rel_change", fast(call_rel_change), METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};

PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    table_type.tp_name = "_native.Table";
    table_type.tp_basicsize = sizeof(Table);
    table_type.tp_flags = Py_TPFLAGS_DEFAULT;
    table_type.tp_new = table_new;
    table_type.tp_dealloc = table_dealloc;
    table_type.tp_methods = table_methods;
    if (PyType_Ready(&table_type) < 0) return nullptr;
    PyObject *m = PyModule_Create(&module_def);
    if (!m) return nullptr;
    if (PyModule_AddObjectRef(m, "Table", reinterpret_cast<PyObject *>(&table_type)) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    // This module reads torch's own objects, whose layout is that of one build: module.py compares.
    if (PyModule_AddStringConstant(m, "torch_version", DESLOC_TORCH_VERSION) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
