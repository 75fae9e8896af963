// The Python side of the calls a step is made of: argument marshalling in native code.
//
// One function per C entry point, same argument order as in binding.py; tensors become pointers, the return code
// comes back as an int.  Through ctypes the same marshalling took 12 us for an attention call and 7-9 us for the
// others, more than enqueueing the kernels takes (5-6 us), and eager calls on small batches were bound by it: the
// 8-node fp32 step 47 -> 32 us, one contemplate-token embedding 11.1 -> 7.6 us.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "confu.h"

namespace {

// Arguments in order; a conversion that fails leaves a Python exception set and makes `ok` false.
struct Reader {
    PyObject* const* args;
    Py_ssize_t n, at = 0;
    bool ok = true;

    PyObject* next()
    {
        if (at >= n) {
            if (ok) PyErr_SetString(PyExc_TypeError, "too few arguments");
            ok = false;
            return Py_None;
        }
        return args[at++];
    }
    const at::Tensor* tensor(PyObject* o)
    {
        if (!ok) return nullptr;
        if (!THPVariable_Check(o)) {
            PyErr_SetString(PyExc_TypeError, "expected a tensor, an address or None");
            ok = false;
            return nullptr;
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "device, contiguous tensors only");
            ok = false;
            return nullptr;
        }
        return &t;
    }
    void* ptr(size_t* bytes = nullptr)
    {
        PyObject* o = next();
        if (!ok || o == Py_None) return nullptr;
        if (PyLong_Check(o)) return PyLong_AsVoidPtr(o);
        const at::Tensor* t = tensor(o);
        if (!t) return nullptr;
        if (bytes) *bytes = t->nbytes();
        return t->data_ptr();
    }
    template <typename T> T* as() { return static_cast<T*>(ptr()); }
    long long integer()
    {
        PyObject* o = next();
        if (!ok) return 0;
        const long long v = PyLong_AsLongLong(o);
        if (v == -1 && PyErr_Occurred()) ok = false;
        return v;
    }
    float real()
    {
        PyObject* o = next();
        if (!ok) return 0.f;
        const double v = PyFloat_AsDouble(o);
        if (v == -1.0 && PyErr_Occurred()) ok = false;
        return (float)v;
    }
    // memory of a ctypes object (at least `bytes` of it)
    void* memory(size_t bytes)
    {
        PyObject* o = next();
        if (!ok) return nullptr;
        Py_buffer view;
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
            ok = false;
            return nullptr;
        }
        void* p = view.buf;                          // the object outlives the call: the caller holds it
        if ((size_t)view.len < bytes) {
            PyErr_SetString(PyExc_TypeError, "object too small");
            ok = false;
        }
        PyBuffer_Release(&view);
        return ok ? p : nullptr;
    }
    confu_ctx* ctx()                                 // None: a null context, which the call refuses
    {
        if (ok && at < n && args[at] == Py_None) {
            ++at;
            return nullptr;
        }
        void* p = memory(sizeof(void*));
        return p ? *static_cast<confu_ctx**>(p) : nullptr;
    }
    const confu_dims* dims() { return static_cast<const confu_dims*>(memory(sizeof(confu_dims))); }
    // a torch stream, or None for the current one
    void* stream()
    {
        PyObject* o = next();
        if (!ok) return nullptr;
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        PyObject* s = PyObject_GetAttrString(o, "cuda_stream");
        if (!s) {
            ok = false;
            return nullptr;
        }
        void* p = PyLong_AsVoidPtr(s);
        Py_DECREF(s);
        return p;
    }
};

#define BEGIN                                                   \
    Reader r{args, n_args};                                     \
    try {
#define END(call)                                               \
        if (!r.ok) return nullptr;                              \
        int rc;                                                 \
        Py_BEGIN_ALLOW_THREADS                                  \
        rc = call;                                              \
        Py_END_ALLOW_THREADS                                    \
        return PyLong_FromLong(rc);                             \
    } catch (const std::exception& e) {                         \
        PyErr_SetString(PyExc_RuntimeError, e.what());          \
        return nullptr;                                         \
    }

PyObject* tree_plan(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const confu_dims* dims = r.dims();
    auto seq_start = r.as<int64_t>();
    auto prefix_len = r.as<int32_t>(), parent = r.as<int32_t>(), con_owner = r.as<int32_t>();
    void* plan = r.ptr();
    auto status = r.as<int32_t>();
    void* st = r.stream();
    END(confu_tree_plan(ctx, dims, seq_start, prefix_len, parent, con_owner, plan, status, st))
}

PyObject* tree_attention(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const confu_dims* dims = r.dims();
    void *q = r.ptr(), *k = r.ptr(), *v = r.ptr();
    const int64_t n_slots = r.integer();
    auto seq_start = r.as<int64_t>();
    auto prefix_len = r.as<int32_t>();
    void *ks = r.ptr(), *vs = r.ptr();
    auto parent = r.as<int32_t>(), con_owner = r.as<int32_t>();
    void *plan = r.ptr(), *out = r.ptr();
    auto lse = r.as<float>();
    auto status = r.as<int32_t>();
    void* st = r.stream();
    END(confu_tree_attention(ctx, dims, q, k, v, n_slots, seq_start, prefix_len, ks, vs, parent, con_owner, plan, out, lse, status, st))
}

PyObject* tree_accept(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const int B = (int)r.integer(), T = (int)r.integer(), C = (int)r.integer(), V = (int)r.integer(), dtype = (int)r.integer();
    void *tl = r.ptr(), *dl = r.ptr();
    auto tokens = r.as<int32_t>(), parent = r.as<int32_t>(), con_owner = r.as<int32_t>();
    auto uniforms = r.as<float>();
    const float temperature = r.real();
    const int mode = (int)r.integer();
    auto accept_len = r.as<int32_t>(), path = r.as<int32_t>(), next_token = r.as<int32_t>(), future_row = r.as<int32_t>(),
         counters = r.as<int32_t>();
    size_t ws_bytes = 0;
    void* ws = r.ptr(&ws_bytes);
    auto status = r.as<int32_t>();
    void* st = r.stream();
    END(confu_tree_accept(ctx, B, T, C, V, dtype, tl, dl, tokens, parent, con_owner, uniforms, temperature, mode, accept_len, path,
                          next_token, future_row, counters, ws, ws_bytes, status, st))
}

PyObject* tree_accept_match(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const int B = (int)r.integer(), T = (int)r.integer(), C = (int)r.integer(), V = (int)r.integer(), dtype = (int)r.integer();
    void* tl = r.ptr();
    auto tokens = r.as<int32_t>(), parent = r.as<int32_t>(), con_owner = r.as<int32_t>();
    auto uniforms = r.as<float>();
    const float temperature = r.real();
    auto accept_len = r.as<int32_t>(), path = r.as<int32_t>(), next_token = r.as<int32_t>(), future_row = r.as<int32_t>(),
         counters = r.as<int32_t>(), status = r.as<int32_t>();
    void* st = r.stream();
    END(confu_tree_accept_match(ctx, B, T, C, V, dtype, tl, tokens, parent, con_owner, uniforms, temperature, accept_len, path,
                                next_token, future_row, counters, status, st))
}

PyObject* kv_compact(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const confu_dims* dims = r.dims();
    const int n_layers = (int)r.integer();
    auto k = r.as<void*>(), v = r.as<void*>();
    auto seq_start = r.as<int64_t>();
    auto prefix_len = r.as<int32_t>(), accept_len = r.as<int32_t>(), path = r.as<int32_t>(), new_len = r.as<int32_t>(),
         status = r.as<int32_t>();
    void* st = r.stream();
    END(confu_kv_compact(ctx, dims, n_layers, k, v, seq_start, prefix_len, accept_len, path, new_len, status, st))
}

PyObject* kv_append(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const confu_dims* dims = r.dims();
    void *k_rows = r.ptr(), *v_rows = r.ptr(), *k = r.ptr(), *v = r.ptr();
    auto seq_start = r.as<int64_t>();
    auto prefix_len = r.as<int32_t>();
    void* st = r.stream();
    END(confu_kv_append(ctx, dims, k_rows, v_rows, k, v, seq_start, prefix_len, st))
}

// hidden, experts give the sizes; the type code is the caller's
PyObject* con_embedding(PyObject*, PyObject* const* args, Py_ssize_t n_args)
{
    BEGIN
    confu_ctx* ctx = r.ctx();
    const int dtype = (int)r.integer();
    const at::Tensor* hidden = r.tensor(r.next());
    void *router_w = r.ptr(), *router_b = r.ptr();
    const at::Tensor* experts = r.tensor(r.next());
    const int k_expert = (int)r.integer(), renormalize = (int)r.integer();
    void* out = r.ptr();
    auto sel = r.as<int32_t>();
    auto gate = r.as<float>();
    auto status = r.as<int32_t>();
    void* st = r.stream();
    if (r.ok && (hidden->dim() != 2 || experts->dim() != 2)) {
        PyErr_SetString(PyExc_ValueError, "hidden and experts are matrices");
        return nullptr;
    }
    END(confu_con_embedding(ctx, (int)hidden->size(0), (int)hidden->size(1), (int)experts->size(1), (int)experts->size(0), k_expert,
                            dtype, hidden->data_ptr(), router_w, router_b, experts->data_ptr(), renormalize, out, sel, gate, status, st))
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(tree_plan), FAST(tree_attention), FAST(tree_accept), FAST(tree_accept_match), FAST(kv_compact),
                         FAST(kv_append), FAST(con_embedding), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() { return PyModule_Create(&module); }
