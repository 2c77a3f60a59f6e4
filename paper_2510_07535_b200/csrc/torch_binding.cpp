// Native half of the Python binding: takes the tensors of one call, checks them (dtype, device, contiguity) and hands
// their pointers, with torch's current stream, to the C entry point.  Marshalling only.
//
// A step's seventeen arguments cost 13 us through ctypes and Python-level checks - as much as the GPU takes for a short
// context - and about a microsecond here.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <utility>

#include "../../include/owlverify.h"

namespace {

enum Type { kI32, kF32, kBf16, kF16 };
struct Spec { const char* name; Type type; };

const char* type_name(Type t) {
    switch (t) {
        case kI32: return "torch.int32";
        case kF32: return "torch.float32";
        case kBf16: return "torch.bfloat16";
        default: return "torch.float16";
    }
}
at::ScalarType scalar_type(Type t) {
    switch (t) {
        case kI32: return at::kInt;
        case kF32: return at::kFloat;
        case kBf16: return at::kBFloat16;
        default: return at::kHalf;
    }
}

// data pointer of a contiguous tensor of the expected type on CUDA device `device`; None is a null pointer
bool tensor_ptr(PyObject* o, const Spec& s, int device, void** out) {
    if (o == Py_None) { *out = nullptr; return true; }
    if (!THPVariable_Check(o)) {
        PyErr_Format(PyExc_TypeError, "%s: expected a tensor or None", s.name);
        return false;
    }
    const at::Tensor& t = THPVariable_Unpack(o);
    if (t.scalar_type() != scalar_type(s.type) || !t.is_cuda() || t.get_device() != device || !t.is_contiguous()) {
        PyErr_Format(PyExc_TypeError, "%s: expected contiguous %s tensor on cuda:%d, got %s on %s", s.name, type_name(s.type), device,
                     c10::toString(t.scalar_type()), t.device().str().c_str());
        return false;
    }
    *out = t.data_ptr();
    return true;
}

// `count` tensors from `args` on into pointers
bool tensors(PyObject* const* args, const Spec* spec, size_t count, int device, void** ptr) {
    for (size_t i = 0; i < count; ++i)
        if (!tensor_ptr(args[i], spec[i], device, &ptr[i])) return false;
    return true;
}

// owl_dims out of the ctypes structure, known by the layout that its buffer states (raw bytes of that size are refused)
bool dims_of(PyObject* o, owl_dims* out) {
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_FORMAT) != 0) return false;
    static const char kLayout[] = "T{<i:batch:<i:total_nodes:";
    const bool ok = view.len == (Py_ssize_t)sizeof(owl_dims) && view.format && strncmp(view.format, kLayout, sizeof kLayout - 1) == 0;
    if (ok) memcpy(out, view.buf, sizeof *out);
    else PyErr_SetString(PyExc_TypeError, "dims: not an OwlDims");
    PyBuffer_Release(&view);
    return ok;
}

// (the low 32 bits of any integer, as ctypes' c_int32 takes it)
bool int_of(PyObject* o, int* out) {
    const unsigned long v = PyLong_AsUnsignedLongMask(o);
    *out = (int)(unsigned)v;
    return !(v == (unsigned long)-1 && PyErr_Occurred());
}

// What the calls on a context begin with: (handle, device, ...)
struct Head {
    owl_ctx* ctx = nullptr;
    int device = 0;
    bool parse(PyObject* const* args, Py_ssize_t nargs, Py_ssize_t want) {
        if (nargs != want) {
            PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, nargs);
            return false;
        }
        ctx = static_cast<owl_ctx*>(PyLong_AsVoidPtr(args[0]));
        return !PyErr_Occurred() && int_of(args[1], &device);
    }
    void* stream() const { return c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream(); }
};

// runs the C call without the interpreter lock: a launch may block while the device's queue is full
template <typename F>
PyObject* unlocked(F&& f) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

template <typename... A, size_t... I>
int invoke(int (*f)(owl_ctx*, const owl_dims*, A...), owl_ctx* ctx, const owl_dims* d, void* const* p, std::index_sequence<I...>) {
    return f(ctx, d, static_cast<A>(p[I])...);
}
// f(ctx, dims, pointers..., stream) called as (handle, device, dims, tensors...)
template <typename... A>
PyObject* pointer_call(int (*f)(owl_ctx*, const owl_dims*, A...), const Spec (&spec)[sizeof...(A) - 1], PyObject* const* args,
                       Py_ssize_t nargs) {
    constexpr size_t n = sizeof...(A) - 1;
    Head h;
    owl_dims d;
    void* p[n + 1];
    if (!h.parse(args, nargs, 3 + n) || !dims_of(args[2], &d) || !tensors(args + 3, spec, n, h.device, p)) return nullptr;
    p[n] = h.stream();
    return unlocked([&] { return invoke(f, h.ctx, &d, p, std::make_index_sequence<n + 1>()); });
}

#define OWL_CALL(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs)

OWL_CALL(verify_attn) {
    static const Spec s[] = {{"q", kBf16}, {"k_cache", kBf16}, {"v_cache", kBf16}, {"block_table", kI32}, {"ctx_lens", kI32},
                             {"node_offsets", kI32}, {"tree_parent", kI32}, {"out", kBf16}, {"lse", kF32}};
    return pointer_call(owl_verify_attn, s, args, nargs);
}
OWL_CALL(verify_attn_f16) {
    static const Spec s[] = {{"q", kF16}, {"k_cache", kF16}, {"v_cache", kF16}, {"block_table", kI32}, {"ctx_lens", kI32},
                             {"node_offsets", kI32}, {"tree_parent", kI32}, {"out", kF16}, {"lse", kF32}};
    return pointer_call(owl_verify_attn_f16, s, args, nargs);
}
OWL_CALL(tree_accept) {
    static const Spec s[] = {{"logits", kF32}, {"draft_tokens", kI32}, {"node_offsets", kI32}, {"tree_parent", kI32},
                             {"accept_len", kI32}, {"accept_path", kI32}, {"bonus_token", kI32}, {"node_argmax", kI32}};
    return pointer_call(owl_tree_accept, s, args, nargs);
}
OWL_CALL(tree_accept_spec) {
    static const Spec s[] = {{"logits", kF32}, {"draft_tokens", kI32}, {"node_offsets", kI32}, {"tree_parent", kI32}, {"accept_len", kI32},
                             {"accept_path", kI32}, {"bonus_token", kI32}, {"spec_node", kI32}, {"node_argmax", kI32}};
    return pointer_call(owl_tree_accept_spec, s, args, nargs);
}
OWL_CALL(verify_step) {
    static const Spec s[] = {{"q", kBf16}, {"k_cache", kBf16}, {"v_cache", kBf16}, {"block_table", kI32}, {"ctx_lens", kI32},
                             {"node_offsets", kI32}, {"tree_parent", kI32}, {"out", kBf16}, {"lse", kF32}, {"logits", kF32},
                             {"draft_tokens", kI32}, {"accept_len", kI32}, {"accept_path", kI32}, {"bonus_token", kI32}, {"node_argmax", kI32}};
    return pointer_call(owl_verify_step, s, args, nargs);
}
OWL_CALL(kv_commit) {
    static const Spec s[] = {{"k_cache", kBf16}, {"v_cache", kBf16}, {"block_table", kI32}, {"ctx_lens", kI32}, {"node_offsets", kI32},
                             {"accept_len", kI32}, {"accept_path", kI32}};
    return pointer_call(owl_kv_commit, s, args, nargs);
}

// (handle, device, dims, spec_token, inputs, outputs)
OWL_CALL(prepare_spec_tree) {
    static const Spec s[] = {{"node_offsets", kI32}, {"tree_parent", kI32}, {"draft_tokens", kI32}, {"ctx_lens", kI32},
                             {"out_node_offsets", kI32}, {"out_tree_parent", kI32}, {"out_draft_tokens", kI32}, {"out_input_ids", kI32},
                             {"out_position_ids", kI32}};
    Head h;
    owl_dims d;
    int token;
    void* p[9];
    if (!h.parse(args, nargs, 13) || !dims_of(args[2], &d) || !int_of(args[3], &token) || !tensors(args + 4, s, 9, h.device, p)) return nullptr;
    auto i = [&](int k) { return static_cast<int32_t*>(p[k]); };
    void* stream = h.stream();
    return unlocked([&] { return owl_prepare_spec_tree(h.ctx, &d, i(0), i(1), i(2), i(3), token, i(4), i(5), i(6), i(7), i(8), stream); });
}
// (handle, device, dims, spec_token, inputs, outputs)
OWL_CALL(prepare_hybrid) {
    static const Spec s[] = {{"node_offsets", kI32}, {"tree_parent", kI32}, {"draft_tokens", kI32}, {"ctx_lens", kI32}, {"route", kI32},
                             {"out_node_offsets", kI32}, {"out_tree_parent", kI32}, {"out_draft_tokens", kI32}, {"out_input_ids", kI32},
                             {"out_position_ids", kI32}};
    Head h;
    owl_dims d;
    int token;
    void* p[10];
    if (!h.parse(args, nargs, 14) || !dims_of(args[2], &d) || !int_of(args[3], &token) || !tensors(args + 4, s, 10, h.device, p)) return nullptr;
    auto i = [&](int k) { return static_cast<int32_t*>(p[k]); };
    void* stream = h.stream();
    return unlocked([&] { return owl_prepare_hybrid(h.ctx, &d, i(0), i(1), i(2), i(3), i(4), token, i(5), i(6), i(7), i(8), i(9), stream); });
}
// (handle, device, dims, hidden_dim, tensors)
OWL_CALL(lm_head_accept) {
    static const Spec s[] = {{"hidden", kBf16}, {"weight", kBf16}, {"draft_tokens", kI32}, {"node_offsets", kI32}, {"tree_parent", kI32},
                             {"accept_len", kI32}, {"accept_path", kI32}, {"bonus_token", kI32}, {"node_argmax", kI32}};
    Head h;
    owl_dims d;
    int hidden_dim;
    void* p[9];
    if (!h.parse(args, nargs, 13) || !dims_of(args[2], &d) || !int_of(args[3], &hidden_dim) || !tensors(args + 4, s, 9, h.device, p)) return nullptr;
    auto i = [&](int k) { return static_cast<int32_t*>(p[k]); };
    void* stream = h.stream();
    return unlocked([&] { return owl_lm_head_accept(h.ctx, &d, hidden_dim, p[0], p[1], i(2), i(3), i(4), i(5), i(6), i(7), i(8), stream); });
}
// (handle, device, rows, d_in, d, alpha, eps, tensors)
OWL_CALL(lstm_cell) {
    static const Spec s[] = {{"h", kBf16}, {"emb", kBf16}, {"w", kBf16}, {"ln_c_gamma", kF32}, {"ln_c_beta", kF32}, {"ln_z_gamma", kF32},
                             {"ln_z_beta", kF32}, {"z", kF32}, {"h_out_f32", kF32}, {"h_out_bf16", kBf16}, {"workspace", kF32}};
    Head h;
    int rows, d_in, d;
    void* p[11];
    if (!h.parse(args, nargs, 18) || !int_of(args[2], &rows) || !int_of(args[3], &d_in) || !int_of(args[4], &d)) return nullptr;
    const float alpha = (float)PyFloat_AsDouble(args[5]), eps = (float)PyFloat_AsDouble(args[6]);
    if (PyErr_Occurred() || !tensors(args + 7, s, 11, h.device, p)) return nullptr;
    auto f = [&](int k) { return static_cast<float*>(p[k]); };
    void* stream = h.stream();
    return unlocked([&] {
        return owl_lstm_cell(h.ctx, rows, d_in, d, p[0], p[1], p[2], alpha, f(3), f(4), f(5), f(6), eps, f(7), f(8), p[9], f(10), stream);
    });
}
// (0, device, dims, tensors): no context
OWL_CALL(tree_accept_static) {
    static const Spec s[] = {{"logits", kF32}, {"draft_tokens", kI32}, {"node_offsets", kI32}, {"tree_parent", kI32}, {"accept_len", kI32},
                             {"accept_path", kI32}, {"bonus_token", kI32}, {"node_argmax", kI32}, {"device_status", kI32}};
    Head h;
    owl_dims d;
    void* p[9];
    if (!h.parse(args, nargs, 12) || !dims_of(args[2], &d) || !tensors(args + 3, s, 9, h.device, p)) return nullptr;
    auto i = [&](int k) { return static_cast<int32_t*>(p[k]); };
    void* stream = h.stream();
    return unlocked([&] { return owl_tree_accept_static(&d, static_cast<float*>(p[0]), i(1), i(2), i(3), i(4), i(5), i(6), i(7), i(8), stream); });
}

// torch throws: from a tensor that has no storage or no strides, or where there is no device.  In Python that is an
// ordinary exception.
template <PyObject* (*kCall)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    return kCall(self, args, nargs);
    END_HANDLE_TH_ERRORS
}

#define OWL_METHOD(name) {#name, (PyCFunction)(void (*)(void))guarded<name>, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {OWL_METHOD(verify_attn), OWL_METHOD(verify_attn_f16), OWL_METHOD(tree_accept), OWL_METHOD(tree_accept_spec),
                         OWL_METHOD(verify_step), OWL_METHOD(kv_commit), OWL_METHOD(prepare_spec_tree), OWL_METHOD(prepare_hybrid),
                         OWL_METHOD(lm_head_accept), OWL_METHOD(lstm_cell), OWL_METHOD(tree_accept_static), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_owl_native", "Tensor marshalling for libowlverify", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__owl_native(void) { return PyModule_Create(&module); }
