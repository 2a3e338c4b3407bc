// The short way from Python to the C ABI: a CPython extension module that reads what a call needs straight from the
// torch tensors (pointers, sizes, types, the current stream) and calls the library function of the same name.
//
// What it is for: a call that runs 5 to 10 us on the GPU must not take longer than that on the host.  Marshalling the
// same arguments in Python through ctypes takes 7 to 10 us a call (a few dozen attribute reads, a structure, a stream
// object).
//
// Every function answers with the library's return code, or with -1 where an argument is not of the plain form it
// handles (not exactly a torch.Tensor, wrong type, shape or device, not contiguous, an object that is no number; a tensor
// that has no memory to point at, which torch reports by a C++ exception: those of vmap, grad and tracing): nothing was
// launched then, and api.py goes its long way, whose checks say what is wrong.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/flat_attn.h"

namespace {

// A call's arguments, taken in order; `bad` once one of them is not plain.
struct Args {
    PyObject* const* a;
    Py_ssize_t n, i = 0;
    bool bad = false;

    PyObject* next() {
        if (i >= n) { bad = true; return Py_None; }
        return a[i++];
    }
    // A contiguous CUDA tensor of this type; nullptr for None where that is allowed, and where the argument is bad.
    const at::Tensor* tensor(at::ScalarType type, bool none_ok = false) {
        PyObject* o = next();
        if (o == Py_None && none_ok) return nullptr;
        if (bad || !THPVariable_CheckExact(o)) { bad = true; return nullptr; }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || t.scalar_type() != type || !t.is_contiguous()) { bad = true; return nullptr; }
        return &t;
    }
    const at::Tensor* bf16() { return tensor(at::kBFloat16); }
    double number() {
        PyObject* o = next();
        if (PyFloat_CheckExact(o)) return PyFloat_AS_DOUBLE(o);
        if (PyLong_CheckExact(o)) {
            const double v = PyLong_AsDouble(o);
            if (v == -1.0 && PyErr_Occurred()) { PyErr_Clear(); bad = true; }
            return v;
        }
        bad = true;
        return 0;
    }
    int whole() {
        PyObject* o = next();
        if (!PyLong_CheckExact(o)) { bad = true; return 0; }
        int over = 0;
        const long long v = PyLong_AsLongLongAndOverflow(o, &over);
        if (over || v < INT32_MIN || v > INT32_MAX) { bad = true; return 0; }
        return static_cast<int>(v);
    }
    int truth() {
        PyObject* o = next();
        if (o == Py_True) return 1;
        if (o == Py_False) return 0;
        bad = true;
        return 0;
    }
    // The status word: an address on the GPU is all the library asks of it.
    int32_t* status() {
        PyObject* o = next();
        if (o == Py_None) return nullptr;
        if (bad || !THPVariable_CheckExact(o) || !THPVariable_Unpack(o).is_cuda()) { bad = true; return nullptr; }
        return static_cast<int32_t*>(THPVariable_Unpack(o).data_ptr());
    }
    // None (the current stream of the current device), an address, or an object with a cuda_stream.
    void* stream() {
        PyObject* o = next();
        if (bad) return nullptr;
        if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
        if (PyLong_CheckExact(o)) return address(o);
        PyObject* s = PyObject_GetAttrString(o, "cuda_stream");
        if (!s) { PyErr_Clear(); bad = true; return nullptr; }
        void* p = address(s);
        Py_DECREF(s);
        return p;
    }
    void* address(PyObject* o) {
        void* p = PyLong_Check(o) ? PyLong_AsVoidPtr(o) : nullptr;
        if (!PyLong_Check(o) || PyErr_Occurred()) { PyErr_Clear(); bad = true; }
        return p;
    }
    void end() { if (i != n) bad = true; }
};

inline bool is(const at::Tensor& t, std::initializer_list<int64_t> want) { return t.sizes().equals(at::IntArrayRef(want)); }
inline bool small(int64_t v) { return v >= 0 && v <= INT32_MAX; }
inline PyObject* no() { return PyLong_FromLong(-1); }
template <typename T> inline T* at_(const at::Tensor* t) { return t ? static_cast<T*>(t->data_ptr()) : nullptr; }
inline void* ptr(const at::Tensor* t) { return at_<void>(t); }

// Runs `call`, which throws nothing (pointers are taken from the tensors before it), without the interpreter lock (the
// driver may block in a launch) and answers with its code.
template <typename F> PyObject* run(F&& call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// Q, O [B,H,Nq,d] and K, V [B,H,Nk,d] of one type.
bool qkvo(Args& a, at::ScalarType type, flat_attn_params_t& p) {
    const at::Tensor *q = a.tensor(type), *k = a.tensor(type), *v = a.tensor(type), *o = a.tensor(type);
    if (a.bad || q->dim() != 4 || k->dim() != 4) return false;
    const int64_t B = q->size(0), H = q->size(1), Nq = q->size(2), d = q->size(3), Nk = k->size(2);
    if (!is(*k, {B, H, Nk, d}) || !is(*v, {B, H, Nk, d}) || !is(*o, {B, H, Nq, d})) return false;
    if (!small(B) || !small(H) || !small(Nq) || !small(Nk) || !small(d)) return false;
    p.Q = ptr(q); p.K = ptr(k); p.V = ptr(v); p.O = ptr(o);
    p.B = static_cast<int>(B); p.H = static_cast<int>(H); p.Nq = static_cast<int>(Nq); p.Nk = static_cast<int>(Nk);
    p.d = static_cast<int>(d);
    p.dtype = type == at::kFloat ? FLAT_DTYPE_F32 : FLAT_DTYPE_BF16;
    return true;
}

at::ScalarType type_of(PyObject* o) {
    return THPVariable_CheckExact(o) ? THPVariable_Unpack(o).scalar_type() : at::ScalarType::Undefined;
}

PyObject* fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {       // Q, K, V, O, scale, stream
    Args a{args, n};
    flat_attn_params_t p{};
    if (!qkvo(a, at::kBFloat16, p)) return no();
    p.scale = static_cast<float>(a.number());
    void* st = a.stream();
    a.end();
    if (a.bad) return no();
    return run([&] { return flat_attn_fwd(p.Q, p.K, p.V, p.O, p.B, p.H, p.Nq, p.Nk, p.d, p.scale, st); });
}

PyObject* fwd_ex(PyObject*, PyObject* const* args, Py_ssize_t n) {
    // Q, K, V, O, scale, k_valid_len, status, variant, stream, causal, lse, bias, block_mask
    if (n < 1) return no();
    Args a{args, n};
    flat_attn_params_t p{};
    const at::ScalarType type = type_of(args[0]);
    if ((type != at::kBFloat16 && type != at::kFloat) || !qkvo(a, type, p)) return no();
    p.scale = static_cast<float>(a.number());
    const at::Tensor* valid = a.tensor(at::kInt, true);
    p.status = a.status();
    p.variant = a.whole();
    void* st = a.stream();
    p.causal = a.truth();
    const at::Tensor* lse = a.tensor(at::kFloat, true);
    const at::ScalarType bias_type = a.i < n ? type_of(args[a.i]) : at::ScalarType::Undefined;
    const at::Tensor* bias = a.tensor(bias_type == at::kFloat ? at::kFloat : at::kBFloat16, true);
    const at::Tensor* map = a.tensor(at::kByte, true);
    a.end();
    if (a.bad || (valid && !is(*valid, {p.B})) || (lse && !is(*lse, {p.B, p.H, p.Nq}))) return no();
    p.k_valid_len = at_<const int32_t>(valid);
    p.lse = at_<float>(lse);
    const int64_t Nq = p.Nq, Nk = p.Nk, tq = (Nq + 127) / 128, tk = (Nk + 127) / 128;
    // [B or 1, H or 1, rows, cols]: the strides of the batch and the head, 0 where the values repeat
    auto strides = [&](const at::Tensor& t, int64_t rows, int64_t cols, long long& sb, long long& sh) {
        if (t.dim() != 4 || t.size(2) != rows || t.size(3) != cols || (t.size(0) != 1 && t.size(0) != p.B) ||
            (t.size(1) != 1 && t.size(1) != p.H))
            return false;
        sh = t.size(1) == 1 ? 0 : rows * cols;
        sb = t.size(0) == 1 ? 0 : t.size(1) * rows * cols;
        return true;
    };
    if (bias) {
        if (!strides(*bias, Nq, Nk, p.bias_stride_b, p.bias_stride_h)) return no();
        p.bias = ptr(bias);
        p.bias_dtype = bias_type == at::kFloat ? FLAT_DTYPE_F32 : FLAT_DTYPE_BF16;
    }
    if (map) {
        if (!strides(*map, tq, tk, p.block_mask_stride_b, p.block_mask_stride_h)) return no();
        p.block_mask = at_<const uint8_t>(map);
    }
    return run([&] { return flat_attn_fwd_ex(&p, st); });
}

// Q, K, V, O, dO, lse, dQ, dK, dV, delta, scale, [k_valid_len, status, causal,] stream
bool bwd_args(Args& a, bool ex, flat_attn_bwd_params_t& p, void*& st) {
    flat_attn_params_t f{};
    if (!qkvo(a, at::kBFloat16, f)) return false;
    const at::Tensor *dO = a.bf16(), *lse = a.tensor(at::kFloat), *dQ = a.bf16(), *dK = a.bf16(), *dV = a.bf16(),
                     *delta = a.tensor(at::kFloat);
    p.scale = static_cast<float>(a.number());
    const at::Tensor* valid = ex ? a.tensor(at::kInt, true) : nullptr;
    p.status = ex ? a.status() : nullptr;
    p.causal = ex ? a.truth() : 0;
    st = a.stream();
    a.end();
    if (a.bad || !is(*dO, {f.B, f.H, f.Nq, f.d}) || !is(*dQ, {f.B, f.H, f.Nq, f.d}) || !is(*dK, {f.B, f.H, f.Nk, f.d}) ||
        !is(*dV, {f.B, f.H, f.Nk, f.d}) || !is(*lse, {f.B, f.H, f.Nq}) || !is(*delta, {f.B, f.H, f.Nq}) ||
        (valid && !is(*valid, {f.B})))
        return false;
    p.Q = f.Q; p.K = f.K; p.V = f.V; p.O = f.O;
    p.dO = ptr(dO); p.dQ = ptr(dQ); p.dK = ptr(dK); p.dV = ptr(dV);
    p.lse = at_<const float>(lse); p.delta = at_<float>(delta);
    p.B = f.B; p.H = f.H; p.Nq = f.Nq; p.Nk = f.Nk; p.d = f.d;
    p.k_valid_len = at_<const int32_t>(valid);
    return true;
}

PyObject* bwd(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a{args, n};
    flat_attn_bwd_params_t p{};
    void* st = nullptr;
    if (!bwd_args(a, false, p, st)) return no();
    return run([&] {
        return flat_attn_bwd(p.Q, p.K, p.V, p.O, p.dO, p.lse, p.dQ, p.dK, p.dV, p.delta, p.B, p.H, p.Nq, p.Nk, p.d, p.scale, st);
    });
}

PyObject* bwd_ex(PyObject*, PyObject* const* args, Py_ssize_t n) {
    Args a{args, n};
    flat_attn_bwd_params_t p{};
    void* st = nullptr;
    if (!bwd_args(a, true, p, st)) return no();
    return run([&] { return flat_attn_bwd_ex(&p, st); });
}

PyObject* varlen_fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {
    // Q, K, V, O, cu_seqlens_q, cu_seqlens_k, max_seqlen_q, scale, causal, status, stream
    Args a{args, n};
    const at::Tensor *Q = a.bf16(), *K = a.bf16(), *V = a.bf16(), *O = a.bf16(), *cq = a.tensor(at::kInt), *ck = a.tensor(at::kInt);
    const int longest = a.whole();
    const float scale = static_cast<float>(a.number());
    const int causal = a.truth();
    int32_t* status = a.status();
    void* st = a.stream();
    a.end();
    if (a.bad || Q->dim() != 3 || K->dim() != 3 || cq->dim() != 1 || ck->dim() != 1) return no();
    const int64_t tq = Q->size(0), H = Q->size(1), d = Q->size(2), tk = K->size(0), seqs = cq->size(0) - 1;
    if (!is(*K, {tk, H, d}) || !is(*V, {tk, H, d}) || !is(*O, {tq, H, d}) || ck->size(0) != seqs + 1 || seqs < 1 ||
        !small(seqs) || !small(H) || !small(d))
        return no();
    void *q = ptr(Q), *k = ptr(K), *v = ptr(V), *o = ptr(O);
    const int32_t *cuq = at_<const int32_t>(cq), *cuk = at_<const int32_t>(ck);
    return run([&] {
        return flat_attn_varlen_fwd(q, k, v, o, cuq, cuk, static_cast<int>(seqs), static_cast<int>(H), static_cast<int>(d), tq, tk,
                                    longest, scale, causal, status, st);
    });
}

PyObject* layer_fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {
    // X, Wqkv, Wo, Y, Q, K, V, O, scale, causal, status, stream
    Args a{args, n};
    const at::Tensor *X = a.bf16(), *Wqkv = a.bf16(), *Wo = a.bf16(), *Y = a.bf16(), *Q = a.bf16(), *K = a.bf16(), *V = a.bf16(),
                     *O = a.bf16();
    const float scale = static_cast<float>(a.number());
    const int causal = a.truth();
    int32_t* status = a.status();
    void* st = a.stream();
    a.end();
    if (a.bad || Q->dim() != 4 || X->dim() != 3) return no();
    const int64_t B = Q->size(0), H = Q->size(1), N = Q->size(2), d = Q->size(3), Dm = X->size(2);
    if (!small(B) || !small(H) || !small(N) || !small(d) || !small(Dm) || !is(*X, {B, N, Dm}) || !is(*Wqkv, {3 * H * d, Dm}) ||
        !is(*Wo, {Dm, H * d}) || !is(*Y, {B, N, Dm}) || !is(*K, {B, H, N, d}) || !is(*V, {B, H, N, d}) || !is(*O, {B, H, N, d}))
        return no();
    void *x = ptr(X), *wqkv = ptr(Wqkv), *wo = ptr(Wo), *y = ptr(Y), *q = ptr(Q), *k = ptr(K), *v = ptr(V), *o = ptr(O);
    return run([&] {
        return flat_attn_layer_fwd(x, wqkv, wo, y, q, k, v, o, static_cast<int>(B), static_cast<int>(N), static_cast<int>(H),
                                   static_cast<int>(d), static_cast<int>(Dm), scale, causal, status, st);
    });
}

PyObject* fc_fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {    // X, W, Y, status, stream
    Args a{args, n};
    const at::Tensor *X = a.bf16(), *W = a.bf16(), *Y = a.bf16();
    int32_t* status = a.status();
    void* st = a.stream();
    a.end();
    if (a.bad || X->dim() < 1 || W->dim() != 2 || Y->dim() != X->dim()) return no();
    const int64_t K = X->size(-1), Nout = W->size(0), M = K > 0 ? X->numel() / K : 0;
    if (W->size(1) != K || Y->size(-1) != Nout || !X->sizes().slice(0, X->dim() - 1).equals(Y->sizes().slice(0, Y->dim() - 1)) ||
        M < 1 || !small(M) || !small(K) || !small(Nout))
        return no();
    void *x = ptr(X), *w = ptr(W), *y = ptr(Y);
    return run([&] { return flat_fc_fwd(x, w, y, static_cast<int>(M), static_cast<int>(K), static_cast<int>(Nout), status, st); });
}

PyObject* layernorm_fwd(PyObject*, PyObject* const* args, Py_ssize_t n) {   // X, gamma, beta, Y, eps, residual, stream
    Args a{args, n};
    const at::Tensor *X = a.bf16(), *g = a.bf16(), *b = a.bf16(), *Y = a.bf16();
    const float eps = static_cast<float>(a.number());
    const at::Tensor* R = a.tensor(at::kBFloat16, true);
    void* st = a.stream();
    a.end();
    if (a.bad || X->dim() < 1) return no();
    const int64_t D = X->size(-1), M = D > 0 ? X->numel() / D : 0;
    if (!small(D) || M < 1 || !is(*g, {D}) || !is(*b, {D}) || !Y->sizes().equals(X->sizes()) || (R && !R->sizes().equals(X->sizes())))
        return no();
    void *x = ptr(X), *r = ptr(R), *gamma = ptr(g), *beta = ptr(b), *y = ptr(Y);
    return run([&] { return flat_layernorm_fwd(x, r, gamma, beta, y, M, static_cast<int>(D), eps, st); });
}

// The functions as Python sees them: no C++ exception leaves them.
typedef PyObject* Fast(PyObject*, PyObject* const*, Py_ssize_t);
template <Fast* F> PyObject* guarded(PyObject* self, PyObject* const* args, Py_ssize_t n) {
    try {
        return F(self, args, n);
    } catch (...) {
        PyErr_Clear();
        return no();
    }
}

#define FAST(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(guarded<f>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(fwd), FAST(fwd_ex), FAST(bwd), FAST(bwd_ex), FAST(varlen_fwd), FAST(layer_fwd), FAST(fc_fwd),
                         FAST(layernorm_fwd), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// `built_for`: what the module was compiled against (build.py rebuilds it when that is no longer what is there)
PyMODINIT_FUNC PyInit__binding() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", BINDING_KEY) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
