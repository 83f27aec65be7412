// The calls of a rollout's inner loop without Python between the tensors and the library: checks every tensor (device,
// contiguity, type), takes addresses and sizes and calls the C entry point.  A step of a small block is bound by the host:
// the call cost it 17.3 us, of which the library's own 3 launches 10.  8 steps of one block of 32 rows at D = 256, V = 4096:
// 155 us with ctypes, 104 us with this.
//
// Each function returns the entry point's status, or None when an argument is not what it should be: the caller then
// goes through the checks of binding.py, which say what is wrong.  A tensor without memory of its own (a FakeTensor of a
// trace, the batched tensor of vmap) throws where it is asked for its address: that is caught, and None as well.
#include <Python.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/dare.h"

namespace {

decltype(&dare_denoise_block) f_denoise = nullptr;
decltype(&dare_denoise_block_sampled) f_denoise_sampled = nullptr;
decltype(&dare_attn_varlen) f_varlen = nullptr;

// Walks the argument list; `ok` turns false at the first argument that does not fit.
struct Args {
    PyObject* const* v;
    Py_ssize_t n, at = 0;
    bool ok = true;
    long device = -1;

    PyObject* next() {
        if (at >= n) { ok = false; return Py_None; }
        return v[at++];
    }
    const at::Tensor* tensor(at::ScalarType type) {      // NULL for None
        PyObject* o = next();
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) { ok = false; return nullptr; }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || t.get_device() != device || !t.is_contiguous() || t.scalar_type() != type) ok = false;
        return &t;
    }
    void* ptr(at::ScalarType type) {
        const at::Tensor* t = tensor(type);
        return t && ok ? t->data_ptr() : nullptr;
    }
    void* bf16() { return ptr(at::kBFloat16); }
    int32_t* i32() { return static_cast<int32_t*>(ptr(at::kInt)); }
    float* f32() { return static_cast<float*>(ptr(at::kFloat)); }
    int32_t* counts() {                                   // a device tensor or a page-locked host tensor
        PyObject* o = v[at < n ? at : n - 1];
        if (o != Py_None && THPVariable_Check(o)) {
            const at::Tensor& t = THPVariable_Unpack(o);
            if (!t.is_cuda()) {
                ++at;
                if (!t.is_pinned() || !t.is_contiguous() || t.scalar_type() != at::kInt) { ok = false; return nullptr; }
                return static_cast<int32_t*>(t.data_ptr());
            }
        }
        return i32();
    }
    long long integer() {
        const long long x = PyLong_AsLongLong(next());
        if (x == -1 && PyErr_Occurred()) { PyErr_Clear(); ok = false; }
        return x;
    }
    unsigned long long bits() {                           // an integer modulo 2^64
        const unsigned long long x = PyLong_AsUnsignedLongLongMask(next());
        if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
        return x;
    }
    int flag() {
        const int x = PyObject_IsTrue(next());
        if (x < 0) { PyErr_Clear(); ok = false; }
        return x > 0;
    }
    double real() {
        const double x = PyFloat_AsDouble(next());
        if (x == -1.0 && PyErr_Occurred()) { PyErr_Clear(); ok = false; }
        return x;
    }
    void* address() { return reinterpret_cast<void*>(static_cast<uintptr_t>(integer())); }
};

// (handle, device, stream, scale, q, k_pre, v_pre, prefix_len, k_blk, v_blk, k_suf, v_suf, suffix_len, attn_out, lse, hidden, w,
//  mask_id, exclude, [temperature, seed, step,] tokens, block_start, mode, threshold, k, pred, conf, n_committed, n_remaining)
template <bool SAMPLED>
PyObject* denoise_checked(PyObject* const* argv, Py_ssize_t n) {
    Args a{argv, n};
    dare_ctx* ctx = static_cast<dare_ctx*>(a.address());
    a.device = static_cast<long>(a.integer());
    void* stream = a.address();
    const float scale = static_cast<float>(a.real());
    const at::Tensor* q = a.tensor(at::kBFloat16);
    const at::Tensor* k_pre = a.tensor(at::kBFloat16);
    if (!a.ok || !q || !k_pre || q->dim() != 4 || k_pre->dim() != 4) Py_RETURN_NONE;
    void* v_pre = a.bf16();
    const int32_t* prefix_len = a.i32();
    void *k_blk = a.bf16(), *v_blk = a.bf16();
    const at::Tensor* k_suf = a.tensor(at::kBFloat16);
    void* v_suf = a.bf16();
    const int32_t* suffix_len = a.i32();
    void* out = a.bf16();
    float* lse = a.f32();
    const at::Tensor* hidden = a.tensor(at::kBFloat16);
    const at::Tensor* w = a.tensor(at::kBFloat16);
    const int32_t mask_id = static_cast<int32_t>(a.integer());
    const int exclude = a.flag();
    const float temperature = SAMPLED ? static_cast<float>(a.real()) : 0.f;
    const uint64_t seed = SAMPLED ? a.bits() : 0;
    const uint32_t step = SAMPLED ? static_cast<uint32_t>(a.bits()) : 0;
    const at::Tensor* tokens = a.tensor(at::kInt);
    const int block_start = static_cast<int>(a.integer()), mode = static_cast<int>(a.integer());
    const float threshold = static_cast<float>(a.real());
    const int k = static_cast<int>(a.integer());
    int32_t* pred = a.i32();
    float* conf = a.f32();
    int32_t *n_committed = a.counts(), *n_remaining = a.counts();
    if (!a.ok || a.at != n || !hidden || !w || !tokens || hidden->dim() != 2 || w->dim() < 1 || tokens->dim() < 2 ||
        (k_suf && k_suf->dim() != 4))
        Py_RETURN_NONE;
    const int B = static_cast<int>(q->size(0)), L = static_cast<int>(q->size(1)), Hq = static_cast<int>(q->size(2));
    const int d = static_cast<int>(q->size(3)), Hkv = static_cast<int>(k_pre->size(1));
    const int prefix_cap = static_cast<int>(k_pre->size(2)), suffix_cap = k_suf ? static_cast<int>(k_suf->size(2)) : 0;
    // (everything that may throw stands in front of the part without the interpreter's lock)
    const void *q_ptr = q->data_ptr(), *k_ptr = k_pre->data_ptr(), *suf = k_suf ? k_suf->data_ptr() : nullptr;
    const void *x_ptr = hidden->data_ptr(), *w_ptr = w->data_ptr();
    const int D = static_cast<int>(hidden->size(1)), V = static_cast<int>(w->size(0));
    int32_t* tok = static_cast<int32_t*>(tokens->data_ptr());
    const int64_t row_stride = tokens->size(1);
    int rc;
    Py_BEGIN_ALLOW_THREADS;
    if (SAMPLED)
        rc = f_denoise_sampled(ctx, B, L, Hq, Hkv, d, prefix_cap, suffix_cap, scale, q_ptr, k_ptr, v_pre, prefix_len, k_blk, v_blk,
                               suf, v_suf, suffix_len, out, lse, x_ptr, D, w_ptr, V, mask_id, exclude, temperature, seed, step, tok,
                               row_stride, block_start, mode, threshold, k, pred, conf, n_committed, n_remaining, stream);
    else
        rc = f_denoise(ctx, B, L, Hq, Hkv, d, prefix_cap, suffix_cap, scale, q_ptr, k_ptr, v_pre, prefix_len, k_blk, v_blk, suf,
                       v_suf, suffix_len, out, lse, x_ptr, D, w_ptr, V, mask_id, exclude, tok, row_stride, block_start, mode,
                       threshold, k, pred, conf, n_committed, n_remaining, stream);
    Py_END_ALLOW_THREADS;
    return PyLong_FromLong(rc);
}

// (handle, device, stream, scale, q, k, v, cu_seqlens, max_seqlen, out, lse)
PyObject* varlen_checked(PyObject* const* argv, Py_ssize_t n) {
    Args a{argv, n};
    dare_ctx* ctx = static_cast<dare_ctx*>(a.address());
    a.device = static_cast<long>(a.integer());
    void* stream = a.address();
    const float scale = static_cast<float>(a.real());
    const at::Tensor *q = a.tensor(at::kBFloat16), *k = a.tensor(at::kBFloat16);
    void* v = a.bf16();
    const at::Tensor* cu = a.tensor(at::kInt);
    const int max_seqlen = static_cast<int>(a.integer());
    void* out = a.bf16();
    float* lse = a.f32();
    if (!a.ok || a.at != n || !q || !k || !cu || q->dim() != 3 || k->dim() < 2) Py_RETURN_NONE;
    const int total = static_cast<int>(q->size(0)), Hq = static_cast<int>(q->size(1)), d = static_cast<int>(q->size(2));
    const int Hkv = static_cast<int>(k->size(1)), n_seqs = static_cast<int>(cu->numel()) - 1;
    const void *q_ptr = q->data_ptr(), *k_ptr = k->data_ptr();
    const int32_t* cu_ptr = static_cast<const int32_t*>(cu->data_ptr());
    int rc;
    Py_BEGIN_ALLOW_THREADS;
    rc = f_varlen(ctx, total, n_seqs, max_seqlen, Hq, Hkv, d, scale, q_ptr, k_ptr, v, cu_ptr, out, lse, stream);
    Py_END_ALLOW_THREADS;
    return PyLong_FromLong(rc);
}

template <PyObject* (*CALL)(PyObject* const*, Py_ssize_t)>
PyObject* entry(PyObject*, PyObject* const* argv, Py_ssize_t n) {
    try {
        return CALL(argv, n);
    } catch (...) {      // (none comes from the library: its entry points do not throw)
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}

// bind(path of libdare.so): resolves the entry points in the library that binding.py has loaded
PyObject* bind(PyObject*, PyObject* arg) {
    const char* path = PyUnicode_AsUTF8(arg);
    if (!path) return nullptr;
    void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
    if (lib) {
        f_denoise = reinterpret_cast<decltype(f_denoise)>(dlsym(lib, "dare_denoise_block"));
        f_denoise_sampled = reinterpret_cast<decltype(f_denoise_sampled)>(dlsym(lib, "dare_denoise_block_sampled"));
        f_varlen = reinterpret_cast<decltype(f_varlen)>(dlsym(lib, "dare_attn_varlen"));
    }
    if (!f_denoise || !f_denoise_sampled || !f_varlen) {
        PyErr_Format(PyExc_RuntimeError, "%s does not export the library's entry points", path);
        return nullptr;
    }
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    {"denoise_block", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<denoise_checked<false>>)), METH_FASTCALL, nullptr},
    {"denoise_block_sampled", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<denoise_checked<true>>)), METH_FASTCALL, nullptr},
    {"attn_varlen", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(&entry<varlen_checked>)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
