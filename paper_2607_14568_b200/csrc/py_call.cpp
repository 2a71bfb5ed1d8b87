// Native side of the Python binding: takes the tensors of a call, checks them and calls the C entry point.
//
// A call on a small problem (one decode token, a short prompt) is shorter on the GPU than ctypes marshalling and
// attribute look-ups on seven to ten tensors take on the host (17 us a decode call, 5 us through this
// module), so the checks and the marshalling are done here.  Every function returns the library's status code, or -1 when an
// argument is not what the entry point takes; the caller (binding.py) then words the error.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <exception>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "gdn.h"
#include "gdn_attn.h"

namespace {

constexpr long kNotTaken = -1;

// A tensor argument: present() is false for None, ok is false for anything that does not fit.
struct Arg {
    const at::Tensor* t = nullptr;
    bool ok = true;
    Arg(PyObject* o, at::ScalarType dtype, bool optional = false) {
        if (o == Py_None) { ok = optional; return; }
        if (!THPVariable_Check(o)) { ok = false; return; }
        t = &THPVariable_Unpack(o);
        ok = t->is_cuda() && t->scalar_type() == dtype && t->is_contiguous();
    }
    template <typename P> P* ptr() const { return t ? static_cast<P*>(t->data_ptr()) : nullptr; }
    int64_t dim() const { return t->dim(); }
    at::IntArrayRef sizes() const { return t->sizes(); }
    bool is(std::initializer_list<int64_t> s) const { return !t || t->sizes() == at::IntArrayRef(s); }
};

bool stream_of(PyObject* o, gdn_stream_t* s) {
    if (o == Py_None) { *s = reinterpret_cast<gdn_stream_t>(c10::cuda::getCurrentCUDAStream().stream()); return true; }
    PyObject* h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) { PyErr_Clear(); h = o; Py_INCREF(h); }
    void* p = PyLong_Check(h) ? PyLong_AsVoidPtr(h) : nullptr;
    const bool ok = PyLong_Check(h) && !PyErr_Occurred();
    Py_DECREF(h);
    if (!ok) { PyErr_Clear(); return false; }
    *s = reinterpret_cast<gdn_stream_t>(p);
    return true;
}

bool int_of(PyObject* o, int* v) {
    const long x = PyLong_Check(o) ? PyLong_AsLong(o) : -1;
    if (!PyLong_Check(o) || PyErr_Occurred() || x != (int)x) { PyErr_Clear(); return false; }
    *v = (int)x;
    return true;
}

bool float_of(PyObject* o, float* v) {
    if (!PyFloat_Check(o) && !PyLong_Check(o)) return false;
    const double x = PyFloat_AsDouble(o);
    if (PyErr_Occurred()) { PyErr_Clear(); return false; }
    *v = (float)x;
    return true;
}

// The tensors every prefill entry point has, and the sizes they imply.
struct Prefill {
    Arg q, k, v, a, b, s0, out, fin, cu;
    int B = 0, T = 0, H = 0, dk = 0, dv = 0;
    bool ok = false;
    Prefill(PyObject* q_, PyObject* k_, PyObject* v_, PyObject* a_, PyObject* b_, PyObject* s0_, PyObject* out_, PyObject* fin_, PyObject* cu_,
            at::ScalarType io)
        : q(q_, io), k(k_, io), v(v_, io), a(a_, at::kFloat), b(b_, at::kFloat), s0(s0_, at::kFloat, true), out(out_, io),
          fin(fin_, at::kFloat, true), cu(cu_, at::kInt, true) {
        if (!(q.ok && k.ok && v.ok && a.ok && b.ok && s0.ok && out.ok && fin.ok && cu.ok)) return;
        const int64_t nd = cu.t ? 3 : 4;
        if (q.dim() != nd || v.dim() != nd || a.dim() != nd - 1) return;
        const auto qs = q.sizes(), vs = v.sizes();
        if (k.sizes() != qs || out.sizes() != vs || vs.slice(0, nd - 1) != qs.slice(0, nd - 1)) return;
        if (a.sizes() != qs.slice(0, nd - 1) || b.sizes() != a.sizes()) return;
        const int64_t nB = cu.t ? cu.t->numel() - 1 : qs[0];
        if (qs[nd - 3] > INT32_MAX || nB > INT32_MAX || qs[nd - 2] > INT32_MAX) return;
        B = (int)nB;
        T = (int)qs[nd - 3];
        H = (int)qs[nd - 2];
        dk = (int)qs[nd - 1];
        dv = (int)vs[nd - 1];
        ok = s0.is({B, H, dk, dv}) && fin.is({B, H, dk, dv});
    }
};

PyObject* result(long rc) { return PyLong_FromLong(rc); }

// Calls the entry point without the interpreter lock, as ctypes does: a launch blocks when the queue is full, and what it waits
// for may be a host callback or another stream's work that a Python thread has yet to run.  (The arguments are plain values by
// then; the caller's frame holds the tensors.)
template <typename... P, typename... A>
PyObject* call(int (*entry)(P...), A... args) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = entry(args...);
    Py_END_ALLOW_THREADS
    return result(rc);
}
#define NEED(n) if (nargs != (n)) return result(kNotTaken)
#define REFUSE_UNLESS(c) if (!(c)) return result(kNotTaken)

using PrefillFn = int (*)(const void*, const void*, const void*, const float*, const float*, const float*, void*, float*, const int32_t*, int,
                          int, int, int, int, int, gdn_stream_t);

int f32_entry(const void* q, const void* k, const void* v, const float* a, const float* b, const float* s0, void* out, float* fin,
              const int32_t* cu, int B, int T, int H, int dk, int dv, int chunk, gdn_stream_t s) {
    return gdn_chunk_prefill_f32(static_cast<const float*>(q), static_cast<const float*>(k), static_cast<const float*>(v), a, b, s0,
                                 static_cast<float*>(out), fin, cu, B, T, H, dk, dv, chunk, s);
}

// q, k, v, log_alpha, beta, initial_state, out, final_state, cu_seqlens, chunk, stream
template <PrefillFn F, at::ScalarType IO>
PyObject* prefill(PyObject*, PyObject* const* x, Py_ssize_t nargs) {
    NEED(11);
    const Prefill p(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], x[8], IO);
    int chunk;
    gdn_stream_t s;
    REFUSE_UNLESS(p.ok && int_of(x[9], &chunk) && stream_of(x[10], &s));
    return call(F, p.q.ptr<void>(), p.k.ptr<void>(), p.v.ptr<void>(), p.a.ptr<float>(), p.b.ptr<float>(), p.s0.ptr<float>(),
                p.out.ptr<void>(), p.fin.ptr<float>(), p.cu.ptr<int32_t>(), p.B, p.T, p.H, p.dk, p.dv, chunk, s);
}

// q_raw, k_raw, v, a_raw, b_raw, gate_scale, norm_eps, initial_state, out, final_state, cu_seqlens, chunk, stream
PyObject* prefill_raw(PyObject*, PyObject* const* x, Py_ssize_t nargs) {
    NEED(13);
    const Prefill p(x[0], x[1], x[2], x[3], x[4], x[7], x[8], x[9], x[10], at::kBFloat16);
    int chunk;
    float scale, eps;
    gdn_stream_t s;
    REFUSE_UNLESS(p.ok && float_of(x[5], &scale) && float_of(x[6], &eps) && int_of(x[11], &chunk) && stream_of(x[12], &s));
    return call(gdn_chunk_prefill_raw, p.q.ptr<void>(), p.k.ptr<void>(), p.v.ptr<void>(), p.a.ptr<float>(), p.b.ptr<float>(), scale, eps,
                p.s0.ptr<float>(), p.out.ptr<void>(), p.fin.ptr<float>(), p.cu.ptr<int32_t>(), p.B, p.T, p.H, p.dk, p.dv, chunk, s);
}

// q, k, v, log_alpha, beta, initial_state, gate_z, norm_weight, norm_eps, out, final_state, cu_seqlens, chunk, stream
PyObject* prefill_gated(PyObject*, PyObject* const* x, Py_ssize_t nargs) {
    NEED(14);
    const Prefill p(x[0], x[1], x[2], x[3], x[4], x[5], x[9], x[10], x[11], at::kBFloat16);
    const Arg z(x[6], at::kBFloat16), w(x[7], at::kFloat);
    int chunk;
    float eps;
    gdn_stream_t s;
    REFUSE_UNLESS(p.ok && z.ok && w.ok && z.sizes() == p.out.sizes() && w.is({p.dv}) && float_of(x[8], &eps) && int_of(x[12], &chunk) &&
                  stream_of(x[13], &s));
    return call(gdn_chunk_prefill_gated, p.q.ptr<void>(), p.k.ptr<void>(), p.v.ptr<void>(), p.a.ptr<float>(), p.b.ptr<float>(),
                p.s0.ptr<float>(), z.ptr<void>(), w.ptr<float>(), eps, p.out.ptr<void>(), p.fin.ptr<float>(), p.cu.ptr<int32_t>(), p.B, p.T,
                p.H, p.dk, p.dv, chunk, s);
}

// q, k, v, log_alpha, beta, state, out, stream
PyObject* decode(PyObject*, PyObject* const* x, Py_ssize_t nargs) {
    NEED(8);
    const Arg q(x[0], at::kBFloat16), k(x[1], at::kBFloat16), v(x[2], at::kBFloat16), a(x[3], at::kFloat), b(x[4], at::kFloat),
        st(x[5], at::kFloat), out(x[6], at::kBFloat16);
    gdn_stream_t s;
    REFUSE_UNLESS(q.ok && k.ok && v.ok && a.ok && b.ok && st.ok && out.ok && q.dim() == 3 && v.dim() == 3 && stream_of(x[7], &s));
    const auto qs = q.sizes();
    const int64_t dv = v.sizes()[2];
    REFUSE_UNLESS(k.sizes() == qs && v.is({qs[0], qs[1], dv}) && out.sizes() == v.sizes() && a.is({qs[0], qs[1]}) && b.is({qs[0], qs[1]}) &&
                  st.is({qs[0], qs[1], qs[2], dv}) && qs[0] <= INT32_MAX && qs[1] <= INT32_MAX);
    return call(gdn_decode_step, q.ptr<void>(), k.ptr<void>(), v.ptr<void>(), a.ptr<float>(), b.ptr<float>(), st.ptr<float>(),
                out.ptr<void>(), (int)qs[0], (int)qs[1], (int)qs[2], (int)dv, s);
}

// q, k, v, out, cu_seqlens, scale, stream
PyObject* attention(PyObject*, PyObject* const* x, Py_ssize_t nargs) {
    NEED(7);
    const Arg q(x[0], at::kBFloat16), k(x[1], at::kBFloat16), v(x[2], at::kBFloat16), out(x[3], at::kBFloat16), cu(x[4], at::kInt, true);
    float scale;
    gdn_stream_t s;
    const int64_t nd = cu.t ? 3 : 4;
    REFUSE_UNLESS(q.ok && k.ok && v.ok && out.ok && cu.ok && q.dim() == nd && k.dim() == nd && float_of(x[5], &scale) && stream_of(x[6], &s));
    const auto qs = q.sizes(), ks = k.sizes();
    REFUSE_UNLESS(v.sizes() == ks && out.sizes() == qs && qs.slice(0, nd - 2) == ks.slice(0, nd - 2) && qs[nd - 1] == ks[nd - 1]);
    const int64_t B = cu.t ? cu.t->numel() - 1 : qs[0];
    REFUSE_UNLESS(B <= INT32_MAX && qs[nd - 3] <= INT32_MAX && qs[nd - 2] <= INT32_MAX);
    return call(gdn_attn_causal_prefill, q.ptr<void>(), k.ptr<void>(), v.ptr<void>(), out.ptr<void>(), cu.ptr<int32_t>(), (int)B,
                (int)qs[nd - 3], (int)qs[nd - 2], (int)ks[nd - 2], (int)qs[nd - 1], scale, s);
}

// torch throws when a tensor has no address (inside vmap), no plain sizes (nested tensors) or no device to ask for its stream:
// an exception must not leave a function that the interpreter called.
template <PyObject* (*F)(PyObject*, PyObject* const*, Py_ssize_t)>
PyObject* guarded(PyObject* self, PyObject* const* x, Py_ssize_t nargs) {
    try {
        return F(self, x, nargs);
    } catch (const c10::Error& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    }
    return nullptr;
}

#define FAST(name, ...) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(guarded<__VA_ARGS__>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("gdn_chunk_prefill", prefill<gdn_chunk_prefill, at::kBFloat16>),
    FAST("gdn_chunk_prefill_f32", prefill<f32_entry, at::kFloat>),
    FAST("gdn_chunk_prefill_bf16_simt", prefill<gdn_chunk_prefill_bf16_simt, at::kBFloat16>),
    FAST("gdn_chunk_prefill_noalloc", prefill<gdn_chunk_prefill_noalloc, at::kBFloat16>),
    FAST("gdn_chunk_prefill_raw", prefill_raw),
    FAST("gdn_chunk_prefill_gated", prefill_gated),
    FAST("gdn_decode_step", decode),
    FAST("gdn_attn_causal_prefill", attention),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", "Argument checks and marshalling of libgdn's entry points.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call() { return PyModule_Create(&module); }
