// Native side of the Python binding: the checks and the marshalling of the calls that a serving loop makes.
//
// A decode step of a small model runs in less time than the same checks took in Python (about 12 us a call: shapes,
// dtypes, ctypes conversions).  Every function here takes exactly the positional arguments its Python wrapper names,
// and either calls the C ABI and returns its cq_status, or returns None without having called anything: an argument is
// missing or is not what the call needs, and the wrapper's own checks then say what is wrong (or fill in a default).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/cq.h"

namespace {

struct Args {
    PyObject* const* a;
    bool ok = true;

    const at::Tensor* tensor(int i, c10::ScalarType type, bool cuda)
    {
        if (!THPVariable_Check(a[i])) { ok = false; return nullptr; }
        const at::Tensor& t = THPVariable_Unpack(a[i]);
        if (t.is_cuda() != cuda || t.scalar_type() != type || !t.is_contiguous()) { ok = false; return nullptr; }
        return &t;
    }
    const at::Tensor* device(int i, c10::ScalarType type) { return tensor(i, type, true); }
    const at::Tensor* host(int i, c10::ScalarType type) { return tensor(i, type, false); }
    const at::Tensor* optional(int i, c10::ScalarType type) { return a[i] == Py_None ? nullptr : device(i, type); }
    int64_t integer(int i)
    {
        const long long v = PyLong_Check(a[i]) ? PyLong_AsLongLong(a[i]) : -1;
        if (!PyLong_Check(a[i]) || (v == -1 && PyErr_Occurred())) { PyErr_Clear(); ok = false; return 0; }
        return v;
    }
    int small(int i)
    {
        const int64_t v = integer(i);
        if (v < INT_MIN || v > INT_MAX) ok = false;
        return ok ? (int)v : 0;
    }
    float real(int i)
    {
        if (PyFloat_Check(a[i])) return (float)PyFloat_AS_DOUBLE(a[i]);
        ok = false;
        return 0.f;
    }
};

void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

bool is_shape(const at::Tensor& t, std::initializer_list<int64_t> want)
{
    return t.sizes() == c10::IntArrayRef(want.begin(), want.size());
}

// codebook (n_heads, head_dim / c, 2^b, c)
bool is_book(const at::Tensor& t, int64_t n_heads, int64_t head_dim, int c, int b)
{
    return c > 0 && b >= 1 && b <= 16 && is_shape(t, {n_heads, head_dim / c, (int64_t)1 << b, c});
}

// both code buffers hold what the shape needs (a shape the library refuses needs nothing: its own status says so)
bool hold_codes(const at::Tensor& k, const at::Tensor& v, int64_t n_seq, int64_t cap, int64_t n_heads, int64_t head_dim, int c, int b)
{
    const int64_t need = (int64_t)cq_codes_bytes(n_seq, cap, (int)n_heads, (int)head_dim, c, b);
    return k.numel() >= need && v.numel() >= need;
}

// The status of a library call, which runs without the interpreter's lock: a launch waits where the launch queue is full
// (and the host step for the GPU), and other Python threads go on meanwhile.  (The arguments are taken under the lock; the
// tensors live on in the caller's frame.)
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <typename... Params, typename... A>
PyObject* call(int (*function)(Params...), A... a)
{
    int st;
    {
        Unlocked unlocked;
        st = function(a...);
    }
    return PyLong_FromLong(st);
}

constexpr auto kHalf = c10::ScalarType::Half;
constexpr auto kFloat = c10::ScalarType::Float;
constexpr auto kInt = c10::ScalarType::Int;
constexpr auto kByte = c10::ScalarType::Byte;

// q, k_new, v_new, seq_lens, k_codes, v_codes, k_cb, v_cb, scale, c, b, max_tokens, out, workspace
PyObject* decode_step(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 14) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *q = a.device(0, kHalf), *kn = a.device(1, kHalf), *vn = a.device(2, kHalf), *sl = a.device(3, kInt);
    const at::Tensor *kc = a.device(4, kByte), *vc = a.device(5, kByte), *kb = a.device(6, kFloat), *vb = a.device(7, kFloat);
    const float scale = a.real(8);
    const int c = a.small(9), b = a.small(10);
    const int64_t cap = a.integer(11);
    const at::Tensor *out = a.device(12, kFloat), *ws = a.device(13, kByte);
    if (!a.ok || q->dim() != 3 || kb->dim() != 4) Py_RETURN_NONE;
    const int64_t ns = q->size(0), hq = q->size(1), D = q->size(2), hkv = kb->size(0);
    if (!is_shape(*kn, {ns, hkv, D}) || !is_shape(*vn, {ns, hkv, D}) || sl->numel() != ns || !hold_codes(*kc, *vc, ns, cap, hkv, D, c, b))
        Py_RETURN_NONE;
    return call(cq_decode_step, q->data_ptr(), kn->data_ptr(), vn->data_ptr(), (const int32_t*)sl->data_ptr(), kc->data_ptr(), vc->data_ptr(),
                (const float*)kb->data_ptr(), (const float*)vb->data_ptr(), scale, (int)ns, (int)hq, (int)hkv, (int)D, c, b,
                cap, (float*)out->data_ptr(), ws->data_ptr(), (size_t)ws->numel(), current_stream());
}

// q, k_new, v_new, seq_lens (host), k_codes, v_codes, k_cb, v_cb, scale, c, b, max_tokens, out (host), workspace
PyObject* decode_step_host(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 14) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *q = a.host(0, kHalf), *kn = a.host(1, kHalf), *vn = a.host(2, kHalf), *sl = a.host(3, kInt);
    const at::Tensor *kc = a.device(4, kByte), *vc = a.device(5, kByte), *kb = a.device(6, kFloat), *vb = a.device(7, kFloat);
    const float scale = a.real(8);
    const int c = a.small(9), b = a.small(10);
    const int64_t cap = a.integer(11);
    const at::Tensor *out = a.host(12, kFloat), *ws = a.device(13, kByte);
    if (!a.ok || q->dim() != 3 || kb->dim() < 1) Py_RETURN_NONE;
    const int64_t ns = q->size(0), hq = q->size(1), D = q->size(2), hkv = kb->size(0);
    return call(cq_decode_step_host, q->data_ptr(), kn->data_ptr(), vn->data_ptr(), (const int32_t*)sl->data_ptr(), kc->data_ptr(), vc->data_ptr(),
                (const float*)kb->data_ptr(), (const float*)vb->data_ptr(), scale, (int)ns, (int)hq, (int)hkv, (int)D, c, b, cap,
                (float*)out->data_ptr(), ws->data_ptr(), (size_t)ws->numel(), current_stream());
}

// q, k_codes, v_codes, k_cb, v_cb, seq_lens, scale, c, b, max_tokens, out, workspace, variant
PyObject* decode_attn(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 13) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *q = a.device(0, kHalf), *kc = a.device(1, kByte), *vc = a.device(2, kByte), *kb = a.device(3, kFloat), *vb = a.device(4, kFloat);
    const at::Tensor* sl = a.device(5, kInt);
    const float scale = a.real(6);
    const int c = a.small(7), b = a.small(8);
    const int64_t cap = a.integer(9);
    const at::Tensor *out = a.device(10, kFloat), *ws = a.device(11, kByte);
    const int variant = a.small(12);
    if (!a.ok || q->dim() != 3 || kb->dim() != 4) Py_RETURN_NONE;
    const int64_t ns = q->size(0), hq = q->size(1), D = q->size(2), hkv = kb->size(0);
    if (!is_book(*kb, hkv, D, c, b) || !is_book(*vb, hkv, D, c, b) || sl->numel() != ns || !hold_codes(*kc, *vc, ns, cap, hkv, D, c, b)) Py_RETURN_NONE;
    return call(cq_decode_attn_variant, q->data_ptr(), kc->data_ptr(), vc->data_ptr(), (const float*)kb->data_ptr(), (const float*)vb->data_ptr(),
                (const int32_t*)sl->data_ptr(), scale, (int)ns, (int)hq, (int)hkv, (int)D, c, b, cap,
                (float*)out->data_ptr(), ws->data_ptr(), (size_t)ws->numel(), variant, current_stream());
}

// q, k_codes, v_codes, k_cb, v_cb, seq_lens, rope_cos, rope_sin, scale, c, b, max_tokens, pairing, out, workspace, variant
PyObject* decode_attn_rope(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 16) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *q = a.device(0, kHalf), *kc = a.device(1, kByte), *vc = a.device(2, kByte), *kb = a.device(3, kFloat), *vb = a.device(4, kFloat);
    const at::Tensor *sl = a.device(5, kInt), *cs = a.device(6, kFloat), *sn = a.device(7, kFloat);
    const float scale = a.real(8);
    const int c = a.small(9), b = a.small(10);
    const int64_t cap = a.integer(11);
    const int pairing = a.small(12);
    const at::Tensor *out = a.device(13, kFloat), *ws = a.device(14, kByte);
    const int variant = a.small(15);
    if (!a.ok || q->dim() != 3 || kb->dim() < 1) Py_RETURN_NONE;
    const int64_t ns = q->size(0), hq = q->size(1), D = q->size(2), hkv = kb->size(0);
    if (!is_shape(*cs, {cap, D / 2}) || !is_shape(*sn, {cap, D / 2}) || !hold_codes(*kc, *vc, ns, cap, hkv, D, c, b)) Py_RETURN_NONE;
    return call(cq_decode_attn_rope_variant, q->data_ptr(), kc->data_ptr(), vc->data_ptr(), (const float*)kb->data_ptr(), (const float*)vb->data_ptr(),
                (const int32_t*)sl->data_ptr(), (const float*)cs->data_ptr(), (const float*)sn->data_ptr(), pairing,
                scale, (int)ns, (int)hq, (int)hkv, (int)D, c, b, cap, (float*)out->data_ptr(), ws->data_ptr(),
                (size_t)ws->numel(), variant, current_stream());
}

// q, k_codes, v_codes, k_cb, v_cb, seq_lens, scale, c, b, max_tokens, out, variant
PyObject* prefill_attn(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 12) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *q = a.device(0, kHalf), *kc = a.device(1, kByte), *vc = a.device(2, kByte), *kb = a.device(3, kFloat), *vb = a.device(4, kFloat);
    const at::Tensor* sl = a.device(5, kInt);
    const float scale = a.real(6);
    const int c = a.small(7), b = a.small(8);
    const int64_t cap = a.integer(9);
    const at::Tensor* out = a.device(10, kFloat);
    const int variant = a.small(11);
    if (!a.ok || q->dim() != 4 || kb->dim() != 4) Py_RETURN_NONE;
    const int64_t ns = q->size(0), nq = q->size(1), hq = q->size(2), D = q->size(3), hkv = kb->size(0);
    if (nq > INT_MAX || !is_book(*kb, hkv, D, c, b) || !is_book(*vb, hkv, D, c, b) || sl->numel() != ns || !hold_codes(*kc, *vc, ns, cap, hkv, D, c, b))
        Py_RETURN_NONE;
    return call(cq_prefill_attn_variant, q->data_ptr(), kc->data_ptr(), vc->data_ptr(), (const float*)kb->data_ptr(), (const float*)vb->data_ptr(),
                (const int32_t*)sl->data_ptr(), scale, (int)ns, (int)nq, (int)hq, (int)hkv, (int)D, c, b, cap,
                (float*)out->data_ptr(), variant, current_stream());
}

// x, codebooks, seq_offsets | None, c, b, codes_out, max_tokens, token_offset, variant
PyObject* encode(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 9) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *x = a.device(0, kHalf), *cb = a.device(1, kFloat), *so = a.optional(2, kInt);
    const int c = a.small(3), b = a.small(4);
    const at::Tensor* codes = a.device(5, kByte);
    const int64_t cap = a.integer(6), offset = a.integer(7);
    const int variant = a.small(8);
    if (!a.ok || x->dim() != 4) Py_RETURN_NONE;
    const int64_t ns = x->size(0), nt = x->size(1), h = x->size(2), D = x->size(3);
    if (!is_book(*cb, h, D, c, b) || (so && so->numel() != ns) || !hold_codes(*codes, *codes, ns, cap, h, D, c, b)) Py_RETURN_NONE;
    return call(cq_encode_variant, x->data_ptr(), (const float*)cb->data_ptr(), so ? (const int32_t*)so->data_ptr() : nullptr, ns, nt, offset, cap,
                (int)h, (int)D, c, b, codes->data_ptr(), variant, current_stream());
}

// k, v, k_cb, v_cb, seq_offsets | None, c, b, k_codes, v_codes, max_tokens, token_offset
PyObject* encode_kv(PyObject*, PyObject* const* argv, Py_ssize_t n)
{
    if (n != 11) Py_RETURN_NONE;
    Args a{argv};
    const at::Tensor *k = a.device(0, kHalf), *v = a.device(1, kHalf), *kb = a.device(2, kFloat), *vb = a.device(3, kFloat), *so = a.optional(4, kInt);
    const int c = a.small(5), b = a.small(6);
    const at::Tensor *kc = a.device(7, kByte), *vc = a.device(8, kByte);
    const int64_t cap = a.integer(9), offset = a.integer(10);
    if (!a.ok || k->dim() != 4 || k->sizes() != v->sizes()) Py_RETURN_NONE;
    const int64_t ns = k->size(0), nt = k->size(1), h = k->size(2), D = k->size(3);
    return call(cq_encode_kv, k->data_ptr(), v->data_ptr(), (const float*)kb->data_ptr(), (const float*)vb->data_ptr(),
                so ? (const int32_t*)so->data_ptr() : nullptr, ns, nt, offset, cap, (int)h, (int)D, c, b, kc->data_ptr(),
                vc->data_ptr(), current_stream());
}

// torch throws where a tensor has no memory (under tracing or vmap) or no current stream: no exception may leave for the
// interpreter.  Nothing has been called then, and the wrapper's own checks meet the same error as a Python exception.
template <PyObject* (*function)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* argv, Py_ssize_t n)
{
    try {
        return function(self, argv, n);
    } catch (...) {
        Py_RETURN_NONE;
    }
}

#define CQ_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&guarded<&name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {CQ_METHOD(decode_step), CQ_METHOD(decode_step_host), CQ_METHOD(decode_attn), CQ_METHOD(decode_attn_rope),
                         CQ_METHOD(prefill_attn), CQ_METHOD(encode), CQ_METHOD(encode_kv), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cq_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cq_native() { return PyModule_Create(&module); }
