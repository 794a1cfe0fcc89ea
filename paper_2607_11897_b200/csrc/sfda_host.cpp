// Native marshalling of the decode calls: checks the tensors, takes their addresses and the current stream, calls the
// C ABI.  One token of one sequence keeps the GPU busy for 2.4 us; the same checks in Python with ctypes took 15 us.
// Errors as in the Python wrappers of the other calls: ValueError for layout and place, TypeError for the element type;
// what torch itself throws (a tensor without storage, no driver) comes back as the Python exception torch makes of it.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

typedef int (*StepFn)(const void *, const void *, const void *, const float *, const float *, const float *, float *, void *, void *,
                      int, int, int, int, int, void *);
typedef int (*StepFusedFn)(const void *, const void *, const void *, const float *, const float *, const float *, float, float, float,
                           float, float *, void *, void *, int, int, int, int, int, void *);
StepFn g_step = nullptr;
StepFusedFn g_step_fused = nullptr;

// Address of a CUDA tensor of the wanted type; NULL for None where that is allowed.  false: a Python error is set.
bool address(PyObject *obj, const char *name, at::ScalarType type, void **out)
{
    *out = nullptr;
    if (obj == Py_None) return true;
    if (!THPVariable_Check(obj)) {
        PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
        return false;
    }
    const at::Tensor &t = THPVariable_Unpack(obj);
    if (!t.is_contiguous()) {
        PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
        return false;
    }
    if (!t.is_cuda()) {
        PyErr_Format(PyExc_ValueError, "%s must live on cuda", name);
        return false;
    }
    if (t.scalar_type() != type) {
        PyErr_Format(PyExc_TypeError, "%s must be %s", name, type == at::kFloat ? "torch.float32" : "torch.bfloat16");
        return false;
    }
    *out = t.data_ptr();
    return true;
}

bool stream_of(PyObject *obj, void **out)
{
    if (obj == Py_None) {
        *out = c10::cuda::getCurrentCUDAStream().stream();
        return true;
    }
    PyObject *h = PyObject_GetAttrString(obj, "cuda_stream");
    if (!h) return false;
    *out = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
}

// step(q, k, v, alpha, theta, beta, S, o, o_im, stream); step_fused the same with four floats after beta
PyObject *call(PyObject *const *args, Py_ssize_t n, bool fused)
{
    HANDLE_TH_ERRORS
    static const char *const plain[] = {"q", "k", "v", "alpha", "theta", "beta", "S", "o", "o_im"};
    static const char *const raw[] = {"q", "k_raw", "v", "a_raw", "b_raw", "c_raw", "S", "o", "o_im"};
    const char *const *name = fused ? raw : plain;
    const int skip = fused ? 4 : 0;
    if (n != 10 + skip) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    if (!g_step || !g_step_fused) {
        PyErr_SetString(PyExc_RuntimeError, "bind has not been called");
        return nullptr;
    }
    if (!THPVariable_Check(args[0]) || !THPVariable_Check(args[2])) {
        PyErr_SetString(PyExc_TypeError, "q and v must be tensors");
        return nullptr;
    }
    const at::Tensor &q = THPVariable_Unpack(args[0]), &v = THPVariable_Unpack(args[2]);
    if (q.dim() != 3 || v.dim() < 1) {
        PyErr_SetString(PyExc_ValueError, "q must be [B, H, d_k] and v [B, H, d_v]");
        return nullptr;
    }
    const at::ScalarType type = q.scalar_type();
    if (type != at::kFloat && type != at::kBFloat16) {
        PyErr_SetString(PyExc_TypeError, "q, k, v must be float32 or bfloat16");
        return nullptr;
    }
    void *p[9], *stream;
    for (int i = 0; i < 9; ++i) {
        const bool wide = i >= 3 && i <= 6;                       // alpha, theta, beta, S
        if (!address(args[i < 6 ? i : i + skip], name[i], wide ? at::kFloat : type, &p[i])) return nullptr;
    }
    if (!stream_of(args[9 + skip], &stream)) return nullptr;
    const int B = (int)q.size(0), H = (int)q.size(1), dk = (int)q.size(2), dv = (int)v.size(-1), dt = type == at::kBFloat16;
    float f[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i = 0; i < skip; ++i) {
        const double x = PyFloat_AsDouble(args[6 + i]);
        if (x == -1.0 && PyErr_Occurred()) return nullptr;
        f[i] = (float)x;
    }
    // The launch runs without the interpreter's lock, as a call through ctypes does: it blocks while the launch queue is
    // full, and what empties the queue may be a host callback that needs the lock.
    int rc;
    Py_BEGIN_ALLOW_THREADS
    const float *alpha = static_cast<const float *>(p[3]), *theta = static_cast<const float *>(p[4]), *beta = static_cast<const float *>(p[5]);
    float *S = static_cast<float *>(p[6]);
    rc = fused ? g_step_fused(p[0], p[1], p[2], alpha, theta, beta, f[0], f[1], f[2], f[3], S, p[7], p[8], B, H, dk, dv, dt, stream)
               : g_step(p[0], p[1], p[2], alpha, theta, beta, S, p[7], p[8], B, H, dk, dv, dt, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
    END_HANDLE_TH_ERRORS
}

PyObject *step(PyObject *, PyObject *const *args, Py_ssize_t n) { return call(args, n, false); }
PyObject *step_fused(PyObject *, PyObject *const *args, Py_ssize_t n) { return call(args, n, true); }

// bind(address of sfda_step, address of sfda_step_fused)
PyObject *bind(PyObject *, PyObject *const *args, Py_ssize_t n)
{
    if (n != 2) {
        PyErr_SetString(PyExc_TypeError, "bind takes two addresses");
        return nullptr;
    }
    void *a = PyLong_AsVoidPtr(args[0]), *b = PyLong_AsVoidPtr(args[1]);
    if (PyErr_Occurred()) return nullptr;
    g_step = reinterpret_cast<StepFn>(a);
    g_step_fused = reinterpret_cast<StepFusedFn>(b);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, nullptr},
                         {"step", (PyCFunction)(void (*)(void))step, METH_FASTCALL, nullptr},
                         {"step_fused", (PyCFunction)(void (*)(void))step_fused, METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_host", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject *PyInit__host(void) { return PyModule_Create(&module); }
