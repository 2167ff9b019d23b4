// The checks of a call's tensors, and the call, in native code: what the wrappers of binding.py do in Python for a call
// whose tensors are all as they should be.  A wrapper's Python took 4 to 6 us around a C call of 2 to 6, more than the kernels of a
// short call take (kv_cache_append + mha_decode_step, 3 x 1 head x 229 rows: 17.0 -> 5.6 us).  A function here returns None, before
// anything is enqueued, where a tensor is not plainly what the C entry point takes -- a subclass, another type, shape or place -- and
// the wrapper then goes through its own checks, which say what is wrong.
#include <Python.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/mqa_decode.h"

namespace {

struct Shape {
    int64_t d[4];
    int n;
};

// `o` is a contiguous CUDA tensor of this type and shape: its address (an empty tensor's may be null), else false.
bool plain(PyObject* o, at::ScalarType type, const Shape& shape, void** p) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.scalar_type() != type || !t.is_cuda() || t.layout() != at::kStrided || t.dim() != shape.n) return false;
    for (int i = 0; i < shape.n; ++i)
        if (t.size(i) != shape.d[i]) return false;
    if (!t.is_contiguous()) return false;
    *p = t.data_ptr();
    return true;
}
// The same for an optional tensor: None is a null address.
bool plain_or_none(PyObject* o, at::ScalarType type, const Shape& shape, void** p) {
    if (o == Py_None) { *p = nullptr; return true; }
    return plain(o, type, shape, p);
}
// Sizes of an exact tensor, all of them small enough for an int
bool sizes(PyObject* o, Shape* s) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.layout() != at::kStrided || !t.is_cuda() || t.dim() < 1 || t.dim() > 4) return false;
    s->n = (int)t.dim();
    for (int i = 0; i < s->n; ++i) {
        s->d[i] = t.size(i);
        if (s->d[i] > 0x7fffffff) return false;
    }
    return true;
}
// The workspace, a tensor whose bytes are all that counts
bool bytes_of(PyObject* o, void** p, size_t* bytes) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& t = THPVariable_Unpack(o);
    *p = t.data_ptr();
    *bytes = (size_t)t.numel() * t.element_size();
    return true;
}
// The stream to call on: the handle given, or the one that is current on the tensor's device, if that device is current.
bool stream_for(PyObject* tensor, PyObject* given, mqa_stream_t* stream) {
    const c10::DeviceIndex at = THPVariable_Unpack(tensor).device().index();
    if (at != c10::cuda::current_device()) return false;
    if (given == Py_None) {
        *stream = c10::cuda::getCurrentCUDAStream(at).stream();
        return true;
    }
    *stream = PyLong_AsVoidPtr(given);
    return !PyErr_Occurred();        // (no handle: guarded() passes the error on)
}
template <typename Call>
PyObject* without_gil(Call call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

constexpr auto kBf16 = at::kBFloat16;

// (K, V, k_new, v_new, lens, advance, status, stream)
PyObject* append(PyObject*, PyObject* const* a, Py_ssize_t n) {
    Shape K, V;
    void *Kp, *Vp, *kp, *vp, *lens, *status;
    mqa_stream_t stream;
    if (n != 8 || !sizes(a[0], &K) || !sizes(a[1], &V) || K.n < 3 || V.n != K.n) Py_RETURN_NONE;
    const int64_t b = K.d[0], heads = K.n == 4 ? K.d[1] : 1, m = K.d[K.n - 2], k = K.d[K.n - 1], v = V.d[V.n - 1];
    const Shape Vs = K.n == 4 ? Shape{{b, heads, m, v}, 4} : Shape{{b, m, v}, 3};
    const Shape kn = K.n == 4 ? Shape{{b, heads, k}, 3} : Shape{{b, k}, 2}, vn = K.n == 4 ? Shape{{b, heads, v}, 3} : Shape{{b, v}, 2};
    if (!plain(a[0], kBf16, K, &Kp) || !plain(a[1], kBf16, Vs, &Vp) || !plain(a[2], kBf16, kn, &kp) || !plain(a[3], kBf16, vn, &vp) ||
        !plain(a[4], at::kInt, Shape{{b}, 1}, &lens) || !plain_or_none(a[6], at::kInt, Shape{{1}, 1}, &status) || !stream_for(a[0], a[7], &stream))
        Py_RETURN_NONE;
    const int advance = PyObject_IsTrue(a[5]);
    if (advance < 0) return nullptr;
    return without_gil([&] {
        return kv_cache_append(Kp, Vp, kp, vp, static_cast<int32_t*>(lens), advance, static_cast<int32_t*>(status), (int)b, (int)heads, (int)m, (int)k,
                               (int)v, stream);
    });
}

// A step over the cache: (q, K, V, lens, o, workspace, status, stream)
template <decltype(&mqa_decode_step) CALL, bool MULTI_QUERY>
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    Shape q, K, V;
    void *qp, *Kp, *Vp, *lens, *o, *status, *ws = nullptr;
    size_t ws_bytes = 0;
    mqa_stream_t stream;
    if (n != 8 || !sizes(a[0], &q) || q.n != 3 || !sizes(a[1], &K) || !sizes(a[2], &V) || K.n != (MULTI_QUERY ? 3 : 4) || V.n != K.n) Py_RETURN_NONE;
    const int64_t b = q.d[0], h = q.d[1], k = q.d[2], m = K.d[K.n - 2], v = V.d[V.n - 1];
    const Shape Ks = MULTI_QUERY ? Shape{{b, m, k}, 3} : Shape{{b, h, m, k}, 4}, Vs = MULTI_QUERY ? Shape{{b, m, v}, 3} : Shape{{b, h, m, v}, 4};
    if (!plain(a[0], kBf16, q, &qp) || !plain(a[1], kBf16, Ks, &Kp) || !plain(a[2], kBf16, Vs, &Vp) || !plain(a[3], at::kInt, Shape{{b}, 1}, &lens) ||
        !plain(a[4], at::kFloat, Shape{{b, h, v}, 3}, &o) || !plain_or_none(a[6], at::kInt, Shape{{1}, 1}, &status) ||
        (a[5] != Py_None && !bytes_of(a[5], &ws, &ws_bytes)) || !stream_for(a[0], a[7], &stream))
        Py_RETURN_NONE;
    return without_gil([&] {
        return CALL(qp, Kp, Vp, static_cast<const int32_t*>(lens), static_cast<float*>(o), ws, ws_bytes, static_cast<int32_t*>(status), (int)b, (int)h,
                    (int)m, (int)k, (int)v, stream);
    });
}

// (Q, K, V, start, O, workspace, status, stream)
PyObject* prefill(PyObject*, PyObject* const* a, Py_ssize_t n) {
    Shape Q, K, V;
    void *Qp, *Kp, *Vp, *start, *O, *status, *ws;
    size_t ws_bytes;
    mqa_stream_t stream;
    if (n != 8 || !sizes(a[0], &Q) || Q.n != 4 || !sizes(a[1], &K) || !sizes(a[2], &V) || K.n != 3 || V.n != 3) Py_RETURN_NONE;
    const int64_t b = Q.d[0], h = Q.d[1], t = Q.d[2], k = Q.d[3], m = K.d[1], v = V.d[2];
    if (!plain(a[0], kBf16, Q, &Qp) || !plain(a[1], kBf16, Shape{{b, m, k}, 3}, &Kp) || !plain(a[2], kBf16, Shape{{b, m, v}, 3}, &Vp) ||
        !plain_or_none(a[3], at::kInt, Shape{{b}, 1}, &start) || !plain(a[4], at::kFloat, Shape{{b, h, t, v}, 4}, &O) ||
        !bytes_of(a[5], &ws, &ws_bytes) || !plain_or_none(a[6], at::kInt, Shape{{1}, 1}, &status) || !stream_for(a[0], a[7], &stream))
        Py_RETURN_NONE;
    return without_gil([&] {
        return mqa_prefill_attention(Qp, Kp, Vp, static_cast<const int32_t*>(start), static_cast<float*>(O), ws, ws_bytes, static_cast<int32_t*>(status),
                                     (int)b, (int)h, (int)t, (int)m, (int)k, (int)v, stream);
    });
}

// What torch throws about a tensor that has no plain memory (a vmap's, say) is no more than "not plainly what the call takes".
using Fast = PyObject* (*)(PyObject*, PyObject* const*, Py_ssize_t);
template <Fast F>
PyObject* guarded(PyObject* self, PyObject* const* a, Py_ssize_t n) {
    try {
        PyObject* r = F(self, a, n);
        if (r == Py_None && PyErr_Occurred()) { Py_DECREF(r); r = nullptr; }
        return r;
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

PyMethodDef kMethods[] = {
    {"kv_cache_append", (PyCFunction)(void*)guarded<append>, METH_FASTCALL, nullptr},
    {"mqa_decode_step", (PyCFunction)(void*)guarded<step<mqa_decode_step, true>>, METH_FASTCALL, nullptr},
    {"mha_decode_step", (PyCFunction)(void*)guarded<step<mha_decode_step, false>>, METH_FASTCALL, nullptr},
    {"mqa_prefill_attention", (PyCFunction)(void*)guarded<prefill>, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "checked_call", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_checked_call() { return PyModule_Create(&kModule); }
