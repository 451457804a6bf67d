// Argument marshalling of the Python binding's per-call entry points in one native call: tensors to device
// pointers (with the checks of _binding._dptr), the current CUDA stream, then the library function, whose
// address the caller passes, with the interpreter lock released.  The pure Python path costs 7 us a call and
// 0.5 us a tensor on the host of a GB300, which is more than the kernels of short signals and small chunks
// take; this one 1 us and 0.02 us.
#include <Python.h>

#include <cstdint>
#include <exception>
#include <vector>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

// Device pointer of a contiguous float32 CUDA tensor; nullptr with a Python error set otherwise.
bool tensor_pointer(PyObject *o, const char *name, void **ptr, int64_t *numel) {
    if (THPVariable_Check(o)) {
        const at::Tensor &t = THPVariable_Unpack(o);
        if (t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous()) {
            *ptr = t.data_ptr();
            if (numel) *numel = t.numel();
            return true;
        }
    }
    PyErr_Format(PyExc_TypeError, "%s must be a contiguous float32 CUDA tensor", name);
    return false;
}

bool optional_pointer(PyObject *o, const char *name, void **ptr) {
    *ptr = nullptr;
    return o == Py_None || tensor_pointer(o, name, ptr, nullptr);
}

// A raw stream handle (int), or None: the current stream of the current device.
bool stream_pointer(PyObject *o, void **s) {
    if (o == Py_None) {
        *s = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    *s = PyLong_AsVoidPtr(o);
    return !PyErr_Occurred();
}

template <class F>
PyObject *guarded(F &&f) {
    try {
        return f();
    } catch (const std::exception &e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// run(function, filter, x, y, zi, zf, stream): sos_filter_run or sos_filter_run_noalloc
PyObject *run(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        if (n != 7) return PyErr_Format(PyExc_TypeError, "run takes 7 arguments");
        using Fn = int (*)(void *, const float *, float *, int64_t, const float *, float *, void *);
        void *fn = PyLong_AsVoidPtr(a[0]), *f = PyLong_AsVoidPtr(a[1]), *x, *y, *zi, *zf, *s;
        int64_t len = 0;
        if (PyErr_Occurred() || !tensor_pointer(a[2], "x", &x, &len) || !tensor_pointer(a[3], "y", &y, nullptr) ||
            !optional_pointer(a[4], "zi", &zi) || !optional_pointer(a[5], "zf", &zf) || !stream_pointer(a[6], &s))
            return nullptr;
        int rc;
        Py_BEGIN_ALLOW_THREADS;
        rc = reinterpret_cast<Fn>(fn)(f, static_cast<const float *>(x), static_cast<float *>(y), len,
                                      static_cast<const float *>(zi), static_cast<float *>(zf), s);
        Py_END_ALLOW_THREADS;
        return PyLong_FromLong(rc);
    });
}

// Pointers of a sequence of n tensors (entries may be None where `none` allows it).
bool sequence_pointers(PyObject *seq, Py_ssize_t n, const char *name, bool none, std::vector<void *> &ptrs,
                       std::vector<int64_t> *numel) {
    PyObject *fast = PySequence_Fast(seq, "a sequence of tensors");
    if (!fast) return false;
    bool ok = PySequence_Fast_GET_SIZE(fast) == n;
    if (!ok) PyErr_Format(PyExc_ValueError, "%s: %zd entries for %zd signals", name, PySequence_Fast_GET_SIZE(fast), n);
    ptrs.resize(static_cast<size_t>(n));
    if (numel) numel->resize(static_cast<size_t>(n));
    for (Py_ssize_t i = 0; ok && i < n; ++i) {
        PyObject *o = PySequence_Fast_GET_ITEM(fast, i);
        if (none && o == Py_None)
            ptrs[i] = nullptr;
        else
            ok = tensor_pointer(o, name, &ptrs[i], numel ? &(*numel)[i] : nullptr);
    }
    Py_DECREF(fast);
    return ok;
}

// run_batch(function, filters, xs, ys, zis, zfs, stream): sos_filter_run_batch_ex; filters are objects whose
// attribute _hv, or handle, is the library's handle as an int
PyObject *run_batch(PyObject *, PyObject *const *a, Py_ssize_t nargs) {
    return guarded([&]() -> PyObject * {
        if (nargs != 7) return PyErr_Format(PyExc_TypeError, "run_batch takes 7 arguments");
        static PyObject *attr = PyUnicode_InternFromString("_hv"), *slow = PyUnicode_InternFromString("handle");
        using Fn = int (*)(int, void *const *, void *const *, void *const *, const int64_t *, void *const *,
                           void *const *, void *);
        void *fn = PyLong_AsVoidPtr(a[0]), *s;
        const Py_ssize_t n = PyObject_Length(a[2]);
        if (PyErr_Occurred()) return nullptr;
        std::vector<void *> f(static_cast<size_t>(n)), x, y, zi, zf;
        std::vector<int64_t> len;
        PyObject *fast = PySequence_Fast(a[1], "a sequence of filters");
        if (!fast) return nullptr;
        bool ok = PySequence_Fast_GET_SIZE(fast) == n;
        if (!ok) PyErr_Format(PyExc_ValueError, "filters: %zd entries for %zd signals", PySequence_Fast_GET_SIZE(fast), n);
        for (Py_ssize_t i = 0; ok && i < n; ++i) {
            PyObject *h = PyObject_GetAttr(PySequence_Fast_GET_ITEM(fast, i), attr);
            if (!h && PyErr_ExceptionMatches(PyExc_AttributeError)) {
                PyErr_Clear();
                h = PyObject_GetAttr(PySequence_Fast_GET_ITEM(fast, i), slow);
            }
            f[i] = h ? PyLong_AsVoidPtr(h) : nullptr;
            Py_XDECREF(h);
            ok = !PyErr_Occurred();
        }
        Py_DECREF(fast);
        if (!ok || !sequence_pointers(a[2], n, "x", false, x, &len) || !sequence_pointers(a[3], n, "y", false, y, nullptr) ||
            (a[4] != Py_None && !sequence_pointers(a[4], n, "zi", true, zi, nullptr)) ||
            (a[5] != Py_None && !sequence_pointers(a[5], n, "zf", true, zf, nullptr)) || !stream_pointer(a[6], &s))
            return nullptr;
        int rc;
        Py_BEGIN_ALLOW_THREADS;
        rc = reinterpret_cast<Fn>(fn)(static_cast<int>(n), f.data(), x.data(), y.data(), len.data(),
                                      a[4] == Py_None ? nullptr : zi.data(), a[5] == Py_None ? nullptr : zf.data(), s);
        Py_END_ALLOW_THREADS;
        return PyLong_FromLong(rc);
    });
}

PyMethodDef methods[] = {
    {"run", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(run)), METH_FASTCALL, nullptr},
    {"run_batch", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(run_batch)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
