// Native argument marshalling of the calls that follow a generation stage: rewards, group statistics, allocation, advantages.
// Each launches one kernel of a few microseconds, and a Python wrapper over ctypes spent longer on its arguments than the GPU on
// the kernel (47 us of host time for the five calls of a sampling batch).  Same checks and the same C entry points; the status
// is returned to the Python wrapper, which raises.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/pc.h"

namespace {

decltype(&pc_reward_last_token) f_reward = nullptr;
decltype(&pc_group_stats) f_stats = nullptr;
decltype(&pc_allocate) f_allocate = nullptr;
decltype(&pc_allocate_variance) f_allocate_variance = nullptr;
decltype(&pc_grpo_advantage) f_advantage = nullptr;

// Device address of a contiguous CUDA tensor of the wanted type (ScalarType::Undefined: any); None is NULL, an int is an address.
bool pointer(PyObject* o, c10::ScalarType want, void** out) {
    if (o == Py_None) {
        *out = nullptr;
        return true;
    }
    if (PyLong_Check(o)) {
        *out = PyLong_AsVoidPtr(o);
        return *out != nullptr || !PyErr_Occurred();
    }
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "expected a CUDA tensor");
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda()) PyErr_SetString(PyExc_TypeError, "expected a CUDA tensor");
    else if (!t.is_contiguous()) PyErr_SetString(PyExc_TypeError, "expected a contiguous tensor");
    else if (want != c10::ScalarType::Undefined && t.scalar_type() != want)
        PyErr_Format(PyExc_TypeError, "expected dtype %s, got %s", c10::toString(want), c10::toString(t.scalar_type()));
    else {
        *out = t.data_ptr();
        return true;
    }
    return false;
}

// The positional arguments of one call, read in order; `ok` turns false, with a Python error set, at the first bad one.
struct Args {
    PyObject* const* a;
    Py_ssize_t n, at = 0;
    bool ok = true;
    PyObject* next() {
        if (ok && at >= n) {
            PyErr_SetString(PyExc_TypeError, "too few arguments");
            ok = false;
        }
        return ok ? a[at++] : nullptr;
    }
    template <typename T> T* ptr(c10::ScalarType want) {
        void* p = nullptr;
        PyObject* o = next();
        if (ok) ok = pointer(o, want, &p);
        return static_cast<T*>(p);
    }
    int32_t* i32() { return ptr<int32_t>(c10::kInt); }
    int64_t* i64() { return ptr<int64_t>(c10::kLong); }
    float* f32() { return ptr<float>(c10::kFloat); }
    int integer() {
        PyObject* o = next();
        if (!ok) return 0;
        const long v = PyLong_AsLong(o);
        if (v == -1 && PyErr_Occurred()) ok = false;
        if (ok && (v > INT32_MAX || v < INT32_MIN)) {
            PyErr_SetString(PyExc_OverflowError, "argument does not fit a C int");
            ok = false;
        }
        return (int)v;
    }
    double number() {
        PyObject* o = next();
        if (!ok) return 0.;
        const double v = PyFloat_AsDouble(o);
        if (v == -1. && PyErr_Occurred()) ok = false;
        return v;
    }
};

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

PyObject* reward_last_token(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    Args a{args, nargs};
    const int n = a.integer();
    int32_t* tokens = a.i32();
    int64_t* last = a.i64();
    int32_t* threshold = a.i32();
    float* reward = a.f32();
    return a.ok ? PyLong_FromLong(f_reward(stream(), n, tokens, last, threshold, reward)) : nullptr;
}

PyObject* group_stats(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    Args a{args, nargs};
    const int n_groups = a.integer();
    float* rewards = a.f32();
    int32_t *start = a.i32(), *count = a.i32(), *n = a.i32(), *success = a.i32();
    float *mean = a.f32(), *var = a.f32();
    return a.ok ? PyLong_FromLong(f_stats(stream(), n_groups, rewards, start, count, n, success, mean, var)) : nullptr;
}

// params: a ctypes structure laid out like pc_alloc_params
PyObject* allocate(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    Args a{args, nargs};
    const int n_prompts = a.integer();
    int32_t *success = a.i32(), *pilot_n = a.i32();
    PyObject* params = a.next();
    int32_t *status = a.i32(), *extra = a.i32(), *evict = a.i32(), *selected = a.i32();
    int64_t* total = a.i64();
    if (!a.ok) return nullptr;
    Py_buffer view;
    if (PyObject_GetBuffer(params, &view, PyBUF_SIMPLE) != 0) return nullptr;
    pc_alloc_params p{};
    const bool fits = view.len == (Py_ssize_t)sizeof(p);
    if (fits) p = *static_cast<const pc_alloc_params*>(view.buf);
    PyBuffer_Release(&view);
    if (!fits) {
        PyErr_SetString(PyExc_TypeError, "params must be an AllocParams structure");
        return nullptr;
    }
    return PyLong_FromLong(f_allocate(stream(), n_prompts, success, pilot_n, &p, status, extra, evict, selected, total));
}

PyObject* allocate_variance(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    Args a{args, nargs};
    const int n_prompts = a.integer();
    float* var = a.f32();
    int32_t* pilot_n = a.i32();
    const double var_min = a.number();
    const int n_commit = a.integer(), b_t = a.integer();
    int32_t *status = a.i32(), *extra = a.i32(), *selected = a.i32();
    int64_t* total = a.i64();
    return a.ok ? PyLong_FromLong(f_allocate_variance(stream(), n_prompts, var, pilot_n, var_min, n_commit, b_t, status, extra, selected, total)) : nullptr;
}

PyObject* grpo_advantage(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    Args a{args, nargs};
    const int n_groups = a.integer();
    float* rewards = a.f32();
    int32_t *start = a.i32(), *count = a.i32(), *status = a.ptr<int32_t>(c10::ScalarType::Undefined);
    float* adv = a.f32();
    return a.ok ? PyLong_FromLong(f_advantage(stream(), n_groups, rewards, start, count, status, adv)) : nullptr;
}

// Addresses of the entry points in the loaded library, in the order of the functions above.
PyObject* bind(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    if (nargs != 5) {
        PyErr_SetString(PyExc_TypeError, "bind takes five addresses");
        return nullptr;
    }
    void* p[5];
    for (int i = 0; i < 5; ++i) {
        p[i] = PyLong_AsVoidPtr(args[i]);
        if (p[i] == nullptr) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_ValueError, "null address");
    }
    f_reward = reinterpret_cast<decltype(f_reward)>(p[0]);
    f_stats = reinterpret_cast<decltype(f_stats)>(p[1]);
    f_allocate = reinterpret_cast<decltype(f_allocate)>(p[2]);
    f_allocate_variance = reinterpret_cast<decltype(f_allocate_variance)>(p[3]);
    f_advantage = reinterpret_cast<decltype(f_advantage)>(p[4]);
    Py_RETURN_NONE;
}

// torch reports errors (no driver, a tensor without storage) as C++ exceptions; they become Python's.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
    try {
        return F(self, args, nargs);
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

#define PC_METHOD(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<f>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {PC_METHOD(bind), PC_METHOD(reward_last_token), PC_METHOD(group_stats), PC_METHOD(allocate),
                         PC_METHOD(allocate_variance), PC_METHOD(grpo_advantage), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pc_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pc_calls() {
    PyObject* m = PyModule_Create(&module);
    if (m != nullptr && PyModule_AddStringConstant(m, "built_for", PC_CALLS_KEY) != 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
