// The argument marshalling of binding.py's most frequent calls in native code (a CPython module): shapes, types and layouts of the
// tensors are checked and their addresses, the sizes and the current stream are passed to the C ABI.  The Python code
// around ctypes takes 4 us a call, as long as the kernel of a small problem; this takes a few tenths.
//
// A call is made here only when everything about it is plain: torch.Tensor or Parameter itself, dense CUDA tensors without the
// dispatch key of a wrapper, transform or mode, contiguous, of the expected type and shape, the output given, int and
// float options.  For anything else a function returns -1 without having done anything, and binding.py goes its general way, which
// has the checks and raises the errors.  Otherwise the return value is the forge_status of the call.
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAStream.h>

#include <pthread.h>

#include <cmath>

#include "../../include/forge.h"

namespace {

struct Entries {
    decltype(&forge_attn_fused) attn[3];  // bf16, fp16, fp32
    decltype(&forge_attn_decode_splitkv) decode[2];
    decltype(&forge_linear_act) linear[2];
    decltype(&forge_linear_act_w8a16) linear_w8;
    decltype(&forge_linear_swiglu) swiglu;
} lib;
bool bound = false;

const at::ScalarType kTypes[3] = {at::kBFloat16, at::kHalf, at::kFloat};

// The tensor behind an argument if it is plain, else nullptr.
const at::Tensor* plain(PyObject* o, at::ScalarType type, int dims) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    static const uint64_t dense = c10::DispatchKeySet({c10::DispatchKey::CUDA, c10::DispatchKey::AutogradCUDA,
                                                       c10::DispatchKey::ADInplaceOrView, c10::DispatchKey::AutocastCUDA}).raw_repr();
    if (!t.defined() || (t.key_set().raw_repr() & ~dense) != 0 || !t.is_cuda() || t.scalar_type() != type || t.dim() != dims ||
        !t.is_contiguous())
        return nullptr;
    return &t;
}
// The same for one that may be None (*absent).
const at::Tensor* plain_or_none(PyObject* o, at::ScalarType type, int dims, bool* absent) {
    *absent = o == Py_None;
    return *absent ? nullptr : plain(o, type, dims);
}
void* address(const at::Tensor* t) { return t ? t->mutable_data_ptr() : nullptr; }

bool as_int(PyObject* o, int* v) {
    if (!PyLong_CheckExact(o)) return false;
    int overflow = 0;
    const long x = PyLong_AsLongAndOverflow(o, &overflow);
    if (overflow || x < INT32_MIN || x > INT32_MAX) return false;
    *v = (int)x;
    return true;
}
// A size as an int; the C ABI's sizes are ints, larger ones go the general way.
bool small(int64_t n, int* v) {
    *v = (int)n;
    return n >= 0 && n <= INT32_MAX;
}
bool as_scale(PyObject* o, int64_t D, float* v) {
    if (o == Py_None) *v = (float)std::pow((double)D, -0.5);
    else if (PyFloat_CheckExact(o)) *v = (float)PyFloat_AS_DOUBLE(o);
    else return false;
    return D > 0;
}
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

PyObject* not_plain() { return PyLong_FromLong(-1); }
bool ready(Py_ssize_t n, Py_ssize_t want) { return bound && n == want && !at::impl::torch_function_mode_enabled(); }

// Runs the call without the interpreter lock (a launch waits when the queue of launches is full).
template <typename F>
PyObject* run(F call) {
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = call();
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(st);
}

// C++ exceptions of torch end here: the general way meets the same condition and reports it.
template <typename F>
PyObject* guarded(F f) {
    try {
        return f();
    } catch (...) {
        return not_plain();
    }
}

// attn(type, q, k, v, mask_kind, lens, scale, out)
PyObject* py_attn(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        int ty, mask, B, Hq, Hkv, Sq, Skv, D;
        float scale;
        bool no_lens;
        if (!ready(n, 8) || !as_int(a[0], &ty) || ty < 0 || ty > 2 || !as_int(a[4], &mask)) return not_plain();
        const at::Tensor *q = plain(a[1], kTypes[ty], 4), *k = plain(a[2], kTypes[ty], 4), *v = plain(a[3], kTypes[ty], 4);
        const at::Tensor *out = plain(a[7], kTypes[ty], 4), *lens = plain_or_none(a[5], at::kInt, 1, &no_lens);
        if (!q || !k || !v || !out || (!lens && !no_lens)) return not_plain();
        const auto qs = q->sizes(), ks = k->sizes();
        if (ks[0] != qs[0] || ks[3] != qs[3] || v->sizes() != ks || out->sizes() != qs || (lens && lens->size(0) != qs[0]) ||
            !small(qs[0], &B) || !small(qs[1], &Hq) || !small(ks[1], &Hkv) || !small(qs[2], &Sq) || !small(ks[2], &Skv) ||
            !small(qs[3], &D) || !as_scale(a[6], D, &scale))
            return not_plain();
        void *pq = address(q), *pk = address(k), *pv = address(v), *po = address(out), *s = stream();
        const int32_t* pl = static_cast<const int32_t*>(address(lens));
        return run([&] { return lib.attn[ty](pq, pk, pv, po, B, Hq, Hkv, Sq, Skv, D, mask, pl, scale, s); });
    });
}

// decode(type, q, k_cache, v_cache, lens, num_splits, scale, out, workspace)
PyObject* py_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        int ty, splits, B, Hq, Hkv, Smax, D;
        float scale;
        if (!ready(n, 9) || !as_int(a[0], &ty) || ty < 0 || ty > 1 || !as_int(a[5], &splits)) return not_plain();
        const at::Tensor *q = plain(a[1], kTypes[ty], 3), *k = plain(a[2], kTypes[ty], 4), *v = plain(a[3], kTypes[ty], 4);
        const at::Tensor *lens = plain(a[4], at::kInt, 1), *out = plain(a[7], kTypes[ty], 3), *ws = plain(a[8], at::kByte, 1);
        if (!q || !k || !v || !lens || !out || !ws) return not_plain();
        const auto qs = q->sizes(), ks = k->sizes();
        if (ks[0] != qs[0] || ks[3] != qs[2] || v->sizes() != ks || out->sizes() != qs || lens->size(0) != qs[0] ||
            !small(qs[0], &B) || !small(qs[1], &Hq) || !small(ks[1], &Hkv) || !small(ks[2], &Smax) || !small(qs[2], &D) ||
            !as_scale(a[6], D, &scale))
            return not_plain();
        void *pq = address(q), *pk = address(k), *pv = address(v), *po = address(out), *pw = address(ws), *s = stream();
        const int32_t* pl = static_cast<const int32_t*>(address(lens));
        const size_t bytes = (size_t)ws->numel();
        return run([&] { return lib.decode[ty](pq, pk, pv, po, B, Hq, Hkv, Smax, D, pl, splits, scale, pw, bytes, s); });
    });
}

// The sizes of x [M,K], w ([K,N] for layout 0, else [N,K]) and out [M,N].
bool linear_sizes(const at::Tensor* x, const at::Tensor* w, const at::Tensor* out, int layout, int* M, int* N, int* K) {
    const auto xs = x->sizes(), ws = w->sizes(), os = out->sizes();
    return ws[layout == 0 ? 0 : 1] == xs[1] && os[0] == xs[0] && os[1] == ws[layout == 0 ? 1 : 0] && small(xs[0], M) &&
           small(os[1], N) && small(xs[1], K);
}

// linear(type, x, w, b, residual, act, w_layout, out)
PyObject* py_linear(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        int ty, act, layout, M, N, K;
        bool no_b, no_r;
        if (!ready(n, 8) || !as_int(a[0], &ty) || ty < 0 || ty > 1 || !as_int(a[5], &act) || !as_int(a[6], &layout)) return not_plain();
        const at::Tensor *x = plain(a[1], kTypes[ty], 2), *w = plain(a[2], kTypes[ty], 2), *out = plain(a[7], kTypes[ty], 2);
        const at::Tensor *b = plain_or_none(a[3], kTypes[ty], 1, &no_b), *r = plain_or_none(a[4], kTypes[ty], 2, &no_r);
        if (!x || !w || !out || (!b && !no_b) || (!r && !no_r) || !linear_sizes(x, w, out, layout, &M, &N, &K) ||
            (b && b->size(0) != N) || (r && r->sizes() != out->sizes()))
            return not_plain();
        void *px = address(x), *pw = address(w), *pb = address(b), *pr = address(r), *po = address(out), *s = stream();
        return run([&] { return lib.linear[ty](px, pw, pb, pr, po, M, N, K, act, layout, s); });
    });
}

// linear_w8(x, w_int8, scale, b, residual, act, out)
PyObject* py_linear_w8(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        int act, M, N, K;
        bool no_b, no_r;
        if (!ready(n, 7) || !as_int(a[5], &act)) return not_plain();
        const at::Tensor *x = plain(a[0], at::kHalf, 2), *w = plain(a[1], at::kChar, 2), *sc = plain(a[2], at::kFloat, 1);
        const at::Tensor* out = plain(a[6], at::kHalf, 2);
        const at::Tensor *b = plain_or_none(a[3], at::kHalf, 1, &no_b), *r = plain_or_none(a[4], at::kHalf, 2, &no_r);
        if (!x || !w || !sc || !out || (!b && !no_b) || (!r && !no_r) || !linear_sizes(x, w, out, 1, &M, &N, &K) ||
            sc->size(0) != N || (b && b->size(0) != N) || (r && r->sizes() != out->sizes()))
            return not_plain();
        void *px = address(x), *pw = address(w), *pb = address(b), *pr = address(r), *po = address(out), *s = stream();
        const float* ps = static_cast<const float*>(address(sc));
        return run([&] { return lib.linear_w8(px, pw, ps, pb, pr, po, M, N, K, act, s); });
    });
}

// swiglu(x, w_gate, w_up, w_layout, out)
PyObject* py_swiglu(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        int layout, M, N, K;
        if (!ready(n, 5) || !as_int(a[3], &layout)) return not_plain();
        const at::Tensor *x = plain(a[0], at::kBFloat16, 2), *wg = plain(a[1], at::kBFloat16, 2), *wu = plain(a[2], at::kBFloat16, 2);
        const at::Tensor* out = plain(a[4], at::kBFloat16, 2);
        if (!x || !wg || !wu || !out || !linear_sizes(x, wg, out, layout, &M, &N, &K) || wu->sizes() != wg->sizes()) return not_plain();
        void *px = address(x), *pg = address(wg), *pu = address(wu), *po = address(out), *s = stream();
        return run([&] { return lib.swiglu(px, pg, pu, po, M, N, K, layout, s); });
    });
}

// bind(addresses of the nine entry points, in the order of Entries)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void* p[9];
    if (n != 9) { PyErr_SetString(PyExc_TypeError, "nine addresses expected"); return nullptr; }
    for (int i = 0; i < 9; ++i) {
        p[i] = PyLong_AsVoidPtr(a[i]);
        if (!p[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "address expected");
            return nullptr;
        }
    }
    for (int i = 0; i < 3; ++i) lib.attn[i] = reinterpret_cast<decltype(lib.attn[0])>(p[i]);
    for (int i = 0; i < 2; ++i) lib.decode[i] = reinterpret_cast<decltype(lib.decode[0])>(p[3 + i]);
    for (int i = 0; i < 2; ++i) lib.linear[i] = reinterpret_cast<decltype(lib.linear[0])>(p[5 + i]);
    lib.linear_w8 = reinterpret_cast<decltype(lib.linear_w8)>(p[7]);
    lib.swiglu = reinterpret_cast<decltype(lib.swiglu)>(p[8]);
    // a forked child cannot use its parent's CUDA context: the general way says so
    static const int at_fork = pthread_atfork(nullptr, nullptr, [] { bound = false; });
    bound = at_fork == 0;
    Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr
PyMethodDef methods[] = {{"attn", FAST(py_attn)},           {"decode", FAST(py_decode)}, {"linear", FAST(py_linear)},
                         {"linear_w8", FAST(py_linear_w8)}, {"swiglu", FAST(py_swiglu)}, {"bind", FAST(py_bind)},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "host_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// built_for: the torch and Python this was compiled against (build.py, host_calls_stamp()); binding.py uses the module with no other.
PyMODINIT_FUNC PyInit_host_calls() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", FORGE_HOST_CALLS_STAMP) < 0) {
        Py_DECREF(m);
        return nullptr;
    }
    return m;
}
