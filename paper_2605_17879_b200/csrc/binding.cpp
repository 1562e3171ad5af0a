// Python marshalling of the calls a monitor makes every step: checks the tensors, takes their device pointers and the
// current stream, and calls the C ABI with the GIL released.  The same checks written in Python cost more than the
// kernels of a small fleet: ten output tensors, five attributes each, a stream object and a foreign call are some 15 us
// per evaluation, against under 2 us here.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/guard_b200.h"

namespace {

// The device pointer of an optional tensor, or false with a Python error set.  `type`: the wanted scalar type.
bool device_ptr(PyObject *obj, c10::ScalarType type, int64_t numel, void **out) {
    *out = nullptr;
    if (!obj || obj == Py_None) return true;
    if (!THPVariable_Check(obj)) {
        PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor");
        return false;
    }
    const at::Tensor &t = THPVariable_Unpack(obj);
    if (!t.is_cuda() || !t.is_contiguous()) {
        PyErr_SetString(PyExc_ValueError, "expected a contiguous CUDA tensor");
        return false;
    }
    if (t.scalar_type() != type) {
        PyErr_Format(PyExc_ValueError, "expected dtype %s, got %s", c10::toString(type), c10::toString(t.scalar_type()));
        return false;
    }
    if (t.numel() < numel) {
        PyErr_Format(PyExc_ValueError, "tensor too small: %lld < %lld elements", (long long)t.numel(), (long long)numel);
        return false;
    }
    *out = t.data_ptr();
    return true;
}

// out[name], or None (borrowed for a plain dict, else kept alive by the caller through `hold`).
PyObject *lookup(PyObject *out, PyObject *name, PyObject **hold) {
    if (PyDict_CheckExact(out)) {
        PyObject *v = PyDict_GetItemWithError(out, name);
        return v ? v : (PyErr_Occurred() ? nullptr : Py_None);
    }
    return *hold = PyObject_CallMethod(out, "get", "O", name);
}

struct Output {
    const char *name;
    c10::ScalarType type;
    PyObject *key;
};

// The device pointers of a mapping's outputs; numel[i] elements at least, a negative number skips the output.  keep: a new
// tuple of N, which receives references to them, or NULL.
template <int N>
bool output_ptrs(PyObject *out, Output (&spec)[N], const int64_t (&numel)[N], void *(&ptr)[N], PyObject *keep = nullptr) {
    for (int i = 0; i < N; ++i) {
        ptr[i] = nullptr;
        if (keep) {                // (no slot is ever empty)
            Py_INCREF(Py_None);
            PyTuple_SET_ITEM(keep, i, Py_None);
        }
        if (numel[i] < 0) continue;
        if (!spec[i].key) spec[i].key = PyUnicode_InternFromString(spec[i].name);
        PyObject *hold = nullptr, *v = lookup(out, spec[i].key, &hold);
        const bool ok = v && device_ptr(v, spec[i].type, numel[i], &ptr[i]);
        if (ok && keep) {
            Py_INCREF(v);
            PyTuple_SET_ITEM(keep, i, v);
            Py_DECREF(Py_None);
        }
        Py_XDECREF(hold);
        if (!ok) return false;
    }
    return true;
}

// Makes the device current where it is not, and hands out its current stream.
struct Here {
    c10::cuda::OptionalCUDAGuard guard;
    void *stream;
    explicit Here(int device) {
        if (c10::cuda::current_device() != device) guard.set_index((c10::DeviceIndex)device);
        stream = (void *)c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream();
    }
};

// A reference that is dropped unless it is given away.
struct Ref {
    PyObject *o;
    ~Ref() { Py_XDECREF(o); }
    PyObject *give() {
        PyObject *r = o;
        o = nullptr;
        return r;
    }
};

bool to_ll(PyObject *o, long long *v) {
    *v = PyLong_AsLongLong(o);
    return !(*v == -1 && PyErr_Occurred());
}

bool want_args(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return false;
}

// current_stream(device) -> int
PyObject *py_current_stream(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long dev;
    if (!want_args(n, 1) || !to_ll(args[0], &dev)) return nullptr;
    try {
        return PyLong_FromVoidPtr((void *)c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)dev).stream());
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// ingest(handle, device, R, M, block, step_med, step_mad) -> status
PyObject *py_ingest(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long h, dev, R, M;
    if (!want_args(n, 7) || !to_ll(args[0], &h) || !to_ll(args[1], &dev) || !to_ll(args[2], &R) || !to_ll(args[3], &M)) return nullptr;
    if (!THPVariable_Check(args[4])) {
        PyErr_SetString(PyExc_ValueError, "block must be a tensor");
        return nullptr;
    }
    try {
        const at::Tensor &b = THPVariable_Unpack(args[4]);
        if (b.dim() != 3 || b.size(1) != R || b.size(2) != M) {
            PyErr_Format(PyExc_ValueError, "block must be [B, %lld, %lld]", R, M);
            return nullptr;
        }
        const int64_t B = b.size(0);
        void *pb, *pm, *pd;
        if (!device_ptr(args[4], c10::kFloat, 0, &pb) || !device_ptr(args[5], c10::kFloat, B * M, &pm) ||
            !device_ptr(args[6], c10::kFloat, B * M, &pd))
            return nullptr;
        Here here((int)dev);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = guard_ingest((guard_ctx *)h, (const float *)pb, B > 0x7FFFFFFF ? -1 : (int)B, (float *)pm, (float *)pd, here.stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

Output g_score_out[10] = {{"wmed", c10::kFloat, nullptr},      {"fleet_med", c10::kFloat, nullptr}, {"fleet_mad", c10::kFloat, nullptr},
                          {"scores", c10::kFloat, nullptr},    {"counts", c10::kUInt16, nullptr},   {"mask", c10::kUInt32, nullptr},
                          {"flags", c10::kByte, nullptr},      {"tier", c10::kByte, nullptr},       {"topk_idx", c10::kInt, nullptr},
                          {"topk_score", c10::kFloat, nullptr}};

// score(handle, device, R, M, K, out, hold) -> status; with hold, references to the outputs in the place of a zero
PyObject *py_score(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long h, dev, R, M, K;
    if (!want_args(n, 7) || !to_ll(args[0], &h) || !to_ll(args[1], &dev) || !to_ll(args[2], &R) || !to_ll(args[3], &M) || !to_ll(args[4], &K))
        return nullptr;
    try {
        const int64_t numel[10] = {R * M, M, M, R * M, R * M, R, R, R, K > 0 ? K : -1, K > 0 ? K : -1};
        void *p[10];
        Ref keep{args[6] == Py_True ? PyTuple_New(10) : nullptr};
        if (args[6] == Py_True && !keep.o) return nullptr;
        if (!output_ptrs(args[5], g_score_out, numel, p, keep.o)) return nullptr;
        Here here((int)dev);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = guard_score((guard_ctx *)h, (float *)p[0], (float *)p[1], (float *)p[2], (float *)p[3], (uint16_t *)p[4], (uint32_t *)p[5],
                         (uint8_t *)p[6], (uint8_t *)p[7], (int32_t *)p[8], (float *)p[9], here.stream);
        Py_END_ALLOW_THREADS
        return rc == GUARD_OK && keep.o ? keep.give() : PyLong_FromLong(rc);
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

Output g_node_out[3] = {{"node_flag", c10::kByte, nullptr}, {"node_tier", c10::kByte, nullptr}, {"node_stall", c10::kUInt16, nullptr}};

// node_verdict(handle, device, nodes, out) -> status
PyObject *py_node_verdict(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long h, dev, N;
    if (!want_args(n, 4) || !to_ll(args[0], &h) || !to_ll(args[1], &dev) || !to_ll(args[2], &N)) return nullptr;
    try {
        const int64_t numel[3] = {N, N, N};
        void *p[3];
        if (!output_ptrs(args[3], g_node_out, numel, p)) return nullptr;
        Here here((int)dev);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = guard_node_verdict((guard_ctx *)h, (uint8_t *)p[0], (uint8_t *)p[1], (uint16_t *)p[2], here.stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// join(handle, device) -> status
PyObject *py_join(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long h, dev;
    if (!want_args(n, 2) || !to_ll(args[0], &h) || !to_ll(args[1], &dev)) return nullptr;
    try {
        Here here((int)dev);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = guard_join((guard_ctx *)h, here.stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// A per-metric parameter.  dir (whole): any iterable of M values that int() takes.  The others: anything with a length, of M
// numbers, or one number for all metrics.
template <typename T>
bool per_metric(PyObject *obj, int M, bool whole, T *out) {
    auto one = [&](PyObject *v, T *dst) {
        if (whole) {
            PyObject *i = PyNumber_Long(v);
            if (!i) return false;
            *dst = (T)PyLong_AsUnsignedLongLongMask(i);
            Py_DECREF(i);
            return !PyErr_Occurred();
        }
        const double x = PyFloat_AsDouble(v);
        if (x == -1.0 && PyErr_Occurred()) return false;
        *dst = (T)x;
        return true;
    };
    if (!whole && (PyFloat_Check(obj) || PyLong_Check(obj) || !PyObject_HasAttrString(obj, "__len__"))) {
        if (!one(obj, &out[0])) return false;
        for (int m = 1; m < M; ++m) out[m] = out[0];
        return true;
    }
    PyObject *seq = PySequence_Fast(obj, "expected an iterable of per-metric values");
    if (!seq) return false;
    const Py_ssize_t len = PySequence_Fast_GET_SIZE(seq);
    bool ok = len == M;
    if (!ok) PyErr_Format(PyExc_ValueError, "expected %d per-metric values, got %zd", M, len);
    for (int m = 0; ok && m < M; ++m) ok = one(PySequence_Fast_GET_ITEM(seq, m), &out[m]);
    Py_DECREF(seq);
    return ok;
}

Output g_sweep_out[8] = {{"gpu_med", c10::kFloat, nullptr},   {"fleet_med", c10::kFloat, nullptr}, {"fleet_mad", c10::kFloat, nullptr},
                         {"fleet_cut", c10::kFloat, nullptr}, {"fail_mask", c10::kUInt32, nullptr}, {"gpu_pass", c10::kByte, nullptr},
                         {"node_pass", c10::kByte, nullptr},  {"status", c10::kUInt32, nullptr}};

// sweep_qualify(device, S, nodes, gpus_per_node, dir, thr, floor_rel, floor_abs, pct_ppm, workspace, out) -> status
PyObject *py_sweep_qualify(PyObject *, PyObject *const *args, Py_ssize_t n) {
    long long dev, nodes, gpn, pct;
    if (!want_args(n, 11) || !to_ll(args[0], &dev) || !to_ll(args[2], &nodes) || !to_ll(args[3], &gpn) || !to_ll(args[8], &pct)) return nullptr;
    try {
        if (!THPVariable_Check(args[1]) || !THPVariable_Check(args[9])) {
            PyErr_SetString(PyExc_ValueError, "S and workspace must be tensors");
            return nullptr;
        }
        const at::Tensor &S = THPVariable_Unpack(args[1]);
        const int64_t G = S.size(0), reps = S.size(1), M = S.size(2);
        int8_t dir[GUARD_MAX_METRICS];
        float thr[GUARD_MAX_METRICS], frel[GUARD_MAX_METRICS], fabs_[GUARD_MAX_METRICS];
        if (M < 1 || M > GUARD_MAX_METRICS) {
            PyErr_SetString(PyExc_ValueError, "number of metrics out of range");
            return nullptr;
        }
        void *ps, *pw;
        const int64_t numel[8] = {G * M, M, M, M, G, G, nodes, 1};
        void *p[8];
        if (!per_metric(args[4], (int)M, true, dir) || !per_metric(args[5], (int)M, false, thr) || !per_metric(args[6], (int)M, false, frel) ||
            !per_metric(args[7], (int)M, false, fabs_) || !device_ptr(args[1], c10::kFloat, 0, &ps) || !device_ptr(args[9], c10::kByte, 0, &pw) ||
            !output_ptrs(args[10], g_sweep_out, numel, p))
            return nullptr;
        guard_thresholds th{0, 2, 1, 8, 0.10f, 0.20f, dir, thr, frel, fabs_};
        const size_t wbytes = (size_t)THPVariable_Unpack(args[9]).numel();
        Here here((int)dev);
        int rc;
        Py_BEGIN_ALLOW_THREADS
        rc = guard_sweep_qualify((const float *)ps, (int)nodes, (int)gpn, (int)reps, (int)M, &th, (int32_t)pct, pw, wbytes, (float *)p[0],
                                 (float *)p[1], (float *)p[2], (float *)p[3], (uint32_t *)p[4], (uint8_t *)p[5], (uint8_t *)p[6],
                                 (uint32_t *)p[7], here.stream);
        Py_END_ALLOW_THREADS
        return PyLong_FromLong(rc);
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

PyMethodDef g_methods[] = {{"current_stream", (PyCFunction)(void (*)(void))py_current_stream, METH_FASTCALL, nullptr},
                           {"ingest", (PyCFunction)(void (*)(void))py_ingest, METH_FASTCALL, nullptr},
                           {"score", (PyCFunction)(void (*)(void))py_score, METH_FASTCALL, nullptr},
                           {"node_verdict", (PyCFunction)(void (*)(void))py_node_verdict, METH_FASTCALL, nullptr},
                           {"join", (PyCFunction)(void (*)(void))py_join, METH_FASTCALL, nullptr},
                           {"sweep_qualify", (PyCFunction)(void (*)(void))py_sweep_qualify, METH_FASTCALL, nullptr},
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_guard_native", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__guard_native(void) { return PyModule_Create(&g_module); }
