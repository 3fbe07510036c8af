// The calls of the decode loop without the interpreter in between: argument checks and the library call of
// segkv_decode_step, segkv_append, segkv_decode_sdpa, segkv_truncate_last and segkv_steps for one handle.
//
// Six tensors checked from Python cost about 3 us of a call and marshalling them through ctypes another one, which is
// as much as a small layer's step takes on the GPU.  Here each check reads the tensor object directly.  A call
// whose arguments are not plainly what the step expects (a tensor of another shape, type or place, a tensor subclass, a
// step that is no int) is not made: the method answers None, and the caller takes its general path, which
// raises what it has always raised.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

struct Fns {
    int (*decode_step)(void*, int, const int32_t*, const void*, const void*, const void*, void*, const float*, void*);
    int (*append)(void*, int, const int32_t*, const void*, const void*, void*);
    int (*decode_sdpa)(void*, const void*, void*, const float*, void*);
    int (*truncate_last)(void*);
    int (*steps)(void*);
};

struct Hot {
    PyObject_HEAD
    void* handle;
    Fns fn;
    long long rows, heads, kv_heads, head_dim;
    at::ScalarType dtype;
};

// Device address of a plain contiguous CUDA tensor of this type and shape; None stands for a null pointer.
bool tensor(PyObject* o, at::ScalarType type, const long long* shape, int dims, void** p) {
    *p = nullptr;
    if (o == Py_None) return true;
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.is_cuda() || t.scalar_type() != type || t.layout() != at::kStrided || t.dim() != dims) return false;
    const auto sizes = t.sizes();
    for (int i = 0; i < dims; ++i)
        if (sizes[i] != shape[i]) return false;
    if (!t.is_contiguous()) return false;
    *p = t.data_ptr();
    return true;
}

bool step_of(PyObject* o, int* step) {
    if (!PyLong_CheckExact(o)) return false;
    int over = 0;
    const long v = PyLong_AsLongAndOverflow(o, &over);
    if (over || v != (long)(int)v) return false;
    *step = (int)v;
    return true;
}

// The checks, then the call.  An exception of the tensor library (a tensor without storage, say) leaves the call to the
// general path.
template <typename Check, typename Run>
PyObject* checked(Check check, Run run) {
    void* st = nullptr;
    try {
        if (!check()) Py_RETURN_NONE;
        st = c10::cuda::getCurrentCUDAStream().stream();
    } catch (...) {
        Py_RETURN_NONE;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = run(st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// decode_step(step, beam_parent, k_new, v_new, q, out, slopes)
PyObject* hot_decode_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    const Hot* h = reinterpret_cast<Hot*>(self);
    int step = 0;
    void *par, *k, *v, *q, *out, *sl;
    const long long kv[3] = {h->rows, h->kv_heads, h->head_dim}, qs[3] = {h->rows, h->heads, h->head_dim};
    return checked(
        [&] {
            return n == 7 && step_of(a[0], &step) && tensor(a[1], at::kInt, kv, 1, &par) && tensor(a[2], h->dtype, kv, 3, &k) &&
                   tensor(a[3], h->dtype, kv, 3, &v) && tensor(a[4], h->dtype, qs, 3, &q) && tensor(a[5], h->dtype, qs, 3, &out) &&
                   tensor(a[6], at::kFloat, &h->heads, 1, &sl);
        },
        [&](void* st) { return h->fn.decode_step(h->handle, step, (const int32_t*)par, k, v, q, out, (const float*)sl, st); });
}

// append(step, beam_parent, k_new, v_new)
PyObject* hot_append(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    const Hot* h = reinterpret_cast<Hot*>(self);
    int step = 0;
    void *par, *k, *v;
    const long long kv[3] = {h->rows, h->kv_heads, h->head_dim};
    return checked(
        [&] {
            return n == 4 && step_of(a[0], &step) && tensor(a[1], at::kInt, kv, 1, &par) && tensor(a[2], h->dtype, kv, 3, &k) &&
                   tensor(a[3], h->dtype, kv, 3, &v);
        },
        [&](void* st) { return h->fn.append(h->handle, step, (const int32_t*)par, k, v, st); });
}

// decode_sdpa(q, out, slopes)
PyObject* hot_decode_sdpa(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    const Hot* h = reinterpret_cast<Hot*>(self);
    void *q, *out, *sl;
    const long long qs[3] = {h->rows, h->heads, h->head_dim};
    return checked(
        [&] {
            return n == 3 && tensor(a[0], h->dtype, qs, 3, &q) && tensor(a[1], h->dtype, qs, 3, &out) &&
                   tensor(a[2], at::kFloat, &h->heads, 1, &sl);
        },
        [&](void* st) { return h->fn.decode_sdpa(h->handle, q, out, (const float*)sl, st); });
}

PyObject* hot_truncate_last(PyObject* self, PyObject*) {
    const Hot* h = reinterpret_cast<Hot*>(self);
    return PyLong_FromLong(h->fn.truncate_last(h->handle));
}

PyObject* hot_steps(PyObject* self, PyObject*) {
    const Hot* h = reinterpret_cast<Hot*>(self);
    return PyLong_FromLong(h->fn.steps(h->handle));
}

// Hot(handle, rows, heads, kv_heads, head_dim, bf16, (addresses of decode_step, append, decode_sdpa, truncate_last, steps))
PyObject* hot_new(PyTypeObject* type, PyObject* args, PyObject*) {
    unsigned long long handle, f[5];
    long long rows, heads, kv_heads, head_dim;
    int bf16;
    if (!PyArg_ParseTuple(args, "KLLLLp(KKKKK)", &handle, &rows, &heads, &kv_heads, &head_dim, &bf16, &f[0], &f[1], &f[2], &f[3], &f[4]))
        return nullptr;
    Hot* h = reinterpret_cast<Hot*>(type->tp_alloc(type, 0));
    if (!h) return nullptr;
    h->handle = reinterpret_cast<void*>(handle);
    h->rows = rows;
    h->heads = heads;
    h->kv_heads = kv_heads;
    h->head_dim = head_dim;
    h->dtype = bf16 ? at::kBFloat16 : at::kHalf;
    h->fn.decode_step = reinterpret_cast<decltype(Fns::decode_step)>(f[0]);
    h->fn.append = reinterpret_cast<decltype(Fns::append)>(f[1]);
    h->fn.decode_sdpa = reinterpret_cast<decltype(Fns::decode_sdpa)>(f[2]);
    h->fn.truncate_last = reinterpret_cast<decltype(Fns::truncate_last)>(f[3]);
    h->fn.steps = reinterpret_cast<decltype(Fns::steps)>(f[4]);
    return reinterpret_cast<PyObject*>(h);
}

PyMethodDef methods[] = {
    {"decode_step", (PyCFunction)(void (*)(void))hot_decode_step, METH_FASTCALL, nullptr},
    {"append", (PyCFunction)(void (*)(void))hot_append, METH_FASTCALL, nullptr},
    {"decode_sdpa", (PyCFunction)(void (*)(void))hot_decode_sdpa, METH_FASTCALL, nullptr},
    {"truncate_last", hot_truncate_last, METH_NOARGS, nullptr},
    {"steps", hot_steps, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyTypeObject hot_type = {PyVarObject_HEAD_INIT(nullptr, 0)};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "segkv_hot", nullptr, -1, nullptr, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_segkv_hot(void) {
    hot_type.tp_name = "segkv_hot.Hot";
    hot_type.tp_basicsize = sizeof(Hot);
    hot_type.tp_flags = Py_TPFLAGS_DEFAULT;
    hot_type.tp_new = hot_new;
    hot_type.tp_methods = methods;
    if (PyType_Ready(&hot_type) < 0) return nullptr;
    PyObject* m = PyModule_Create(&module);
    if (!m) return nullptr;
    Py_INCREF(&hot_type);
    if (PyModule_AddObject(m, "Hot", reinterpret_cast<PyObject*>(&hot_type)) < 0) return nullptr;
    return m;
}
