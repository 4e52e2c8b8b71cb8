// Native side of the Python binding for calls so short that Python's own work would be most of them: scoring a schedule is
// 4 us of host time in the library, and took 25 with output tensors, stream and arguments handled in Python (2.4 us for
// each of five torch.empty, 3.2 for the current stream). Argument handling only; the work is libkvp.so's.
// Every function turns what torch throws into the Python exception torch itself raises for it (out of memory, no device, a
// tensor without storage): nothing may be thrown through the interpreter, which would end the process.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/kvp.h"

namespace {

PyObject* value_error(const char* what)
{
    PyErr_SetString(PyExc_ValueError, what);
    return nullptr;
}

// the checks of kvp._ptr; null is allowed for None
bool device_ptr(PyObject* o, at::ScalarType dtype, bool check, void** out)
{
    if (o == Py_None) { *out = nullptr; return true; }
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a tensor"); return false; }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || !t.is_contiguous()) { value_error("expected a contiguous CUDA tensor"); return false; }
    if (check && t.scalar_type() != dtype) { value_error("expected dtype torch.int32"); return false; }
    *out = t.data_ptr();
    return true;
}

bool problem_of(PyObject* const* args, kvp_problem** p, unsigned long long* steps, unsigned long long* w32)
{
    *p = static_cast<kvp_problem*>(PyLong_AsVoidPtr(args[0]));
    *steps = PyLong_AsUnsignedLongLong(args[1]);
    *w32 = PyLong_AsUnsignedLongLong(args[2]);
    return !PyErr_Occurred();
}

// how many schedules a tensor holds
bool batch_of(PyObject* o, unsigned long long per, uint32_t* n)
{
    if (!THPVariable_Check(o)) { PyErr_SetString(PyExc_TypeError, "expected a tensor"); return false; }
    const uint64_t total = (uint64_t)THPVariable_Unpack(o).numel();
    if (total % per) { value_error("schedules must be [n][steps][W32]"); return false; }
    *n = (uint32_t)(total / per);
    return true;
}

bool stream_of(PyObject* o, int device, void** st)
{
    if (o == Py_None) { *st = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream(); return true; }
    *st = PyLong_AsVoidPtr(o);
    return !PyErr_Occurred();
}

// Other Python threads run meanwhile: a call into the library launches, may allocate, and waits when the stream's launch
// queue is full. (Arguments stay alive: the caller's frame holds them.)
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};

at::Tensor make(at::IntArrayRef size, at::ScalarType dtype, c10::Device dev) { return at::detail::empty_cuda(size, dtype, dev, std::nullopt); }

PyObject* k_step_ticks; PyObject* k_total_ticks; PyObject* k_step_seconds; PyObject* k_total_seconds; PyObject* k_bad_step;

bool put(PyObject* dict, PyObject* key, const at::Tensor& t)
{
    if (!t.defined()) return PyDict_SetItem(dict, key, Py_None) == 0;
    PyObject* v = THPVariable_Wrap(t);
    if (!v) return false;
    const int rc = PyDict_SetItem(dict, key, v);
    Py_DECREF(v);
    return rc == 0;
}

// eval(problem, steps, w32, schedules, want_steps, want_seconds, stream or None) -> dict of tensors, or an error code
PyObject* eval(PyObject*, PyObject* const* args, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    if (nargs != 7) return value_error("eval takes 7 arguments");
    kvp_problem* p;
    unsigned long long S, w32;
    uint32_t n;
    void *sched, *st;
    if (!problem_of(args, &p, &S, &w32) || !batch_of(args[3], S * w32, &n) || !device_ptr(args[3], at::kInt, true, &sched)) return nullptr;
    const bool steps = PyObject_IsTrue(args[4]), seconds = PyObject_IsTrue(args[5]);
    const c10::Device dev = THPVariable_Unpack(args[3]).device();
    if (!stream_of(args[6], dev.index(), &st)) return nullptr;
    at::Tensor a, b, c, d, e;
    const int64_t rows[2] = {(int64_t)n, (int64_t)S}, one[1] = {(int64_t)n};
    int rc;
    {
        Unlocked unlocked;
        if (steps) a = make(rows, at::kLong, dev);
        b = make(one, at::kLong, dev);
        if (steps && seconds) c = make(rows, at::kDouble, dev);
        if (seconds) d = make(one, at::kDouble, dev);
        e = make(one, at::kInt, dev);
        rc = kvp_eval(p, static_cast<uint32_t*>(sched), n, steps ? static_cast<uint64_t*>(a.data_ptr()) : nullptr,
                      static_cast<uint64_t*>(b.data_ptr()), c.defined() ? static_cast<double*>(c.data_ptr()) : nullptr,
                      seconds ? static_cast<double*>(d.data_ptr()) : nullptr, static_cast<int32_t*>(e.data_ptr()), st);
    }
    if (rc) return PyLong_FromLong(rc);
    PyObject* out = PyDict_New();
    if (!out || !put(out, k_step_ticks, a) || !put(out, k_total_ticks, b) || !put(out, k_step_seconds, c) ||
        !put(out, k_total_seconds, d) || !put(out, k_bad_step, e)) {
        Py_XDECREF(out);
        return nullptr;
    }
    return out;
    END_HANDLE_TH_ERRORS
}

// eval_noalloc(problem, steps, w32, schedules, step_ticks, total_ticks, step_seconds, total_seconds, bad_step, stream or
// None) -> error code
PyObject* eval_noalloc(PyObject*, PyObject* const* args, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    if (nargs != 10) return value_error("eval_noalloc takes 10 arguments");
    kvp_problem* p;
    unsigned long long S, w32;
    uint32_t n;
    void *sched, *o[5], *st;
    if (!problem_of(args, &p, &S, &w32) || !batch_of(args[3], S * w32, &n) || !device_ptr(args[3], at::kInt, true, &sched)) return nullptr;
    for (int i = 0; i < 5; ++i)
        if (!device_ptr(args[4 + i], at::kInt, false, &o[i])) return nullptr;
    if (!stream_of(args[9], THPVariable_Unpack(args[3]).device().index(), &st)) return nullptr;
    int rc;
    {
        Unlocked unlocked;
        rc = kvp_eval_noalloc(p, static_cast<uint32_t*>(sched), n, static_cast<uint64_t*>(o[0]), static_cast<uint64_t*>(o[1]),
                              static_cast<double*>(o[2]), static_cast<double*>(o[3]), static_cast<int32_t*>(o[4]), st);
    }
    return PyLong_FromLong(rc);
    END_HANDLE_TH_ERRORS
}

// eval_counts(problem, steps, w32, schedules, stream or None) -> tensor, or an error code
PyObject* eval_counts(PyObject*, PyObject* const* args, Py_ssize_t nargs)
{
    HANDLE_TH_ERRORS
    if (nargs != 5) return value_error("eval_counts takes 5 arguments");
    kvp_problem* p;
    unsigned long long S, w32;
    uint32_t n;
    void *sched, *st;
    if (!problem_of(args, &p, &S, &w32) || !batch_of(args[3], S * w32, &n) || !device_ptr(args[3], at::kInt, true, &sched)) return nullptr;
    const c10::Device dev = THPVariable_Unpack(args[3]).device();
    if (!stream_of(args[4], dev.index(), &st)) return nullptr;
    const int64_t shape[3] = {(int64_t)n, (int64_t)S, 4};
    at::Tensor t;
    int rc;
    {
        Unlocked unlocked;
        t = make(shape, at::kInt, dev);
        rc = kvp_eval_counts(p, static_cast<uint32_t*>(sched), n, static_cast<uint32_t*>(t.data_ptr()), st);
    }
    return rc ? PyLong_FromLong(rc) : THPVariable_Wrap(t);
    END_HANDLE_TH_ERRORS
}

// current_stream() -> the cudaStream_t of the current device's current stream
PyObject* current_stream(PyObject*, PyObject*)
{
    HANDLE_TH_ERRORS
    return PyLong_FromVoidPtr(c10::cuda::getCurrentCUDAStream().stream());
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"current_stream", current_stream, METH_NOARGS, nullptr},
    {"eval", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(eval)), METH_FASTCALL, nullptr},
    {"eval_noalloc", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(eval_noalloc)), METH_FASTCALL, nullptr},
    {"eval_counts", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(eval_counts)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_kvp_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__kvp_torch()
{
    k_step_ticks = PyUnicode_InternFromString("step_ticks");
    k_total_ticks = PyUnicode_InternFromString("total_ticks");
    k_step_seconds = PyUnicode_InternFromString("step_seconds");
    k_total_seconds = PyUnicode_InternFromString("total_seconds");
    k_bad_step = PyUnicode_InternFromString("bad_step");
    return PyModule_Create(&module);
}
