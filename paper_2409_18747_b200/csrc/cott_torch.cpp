// The calls of cott.py in their plain forms, without the interpreter: argument checks, output and workspace
// allocation and the call into libcott in one native function each.  A training step of a small layer is
// bound by this work: of the 26 to 30 us that the backward call took the host, 17 to 20 were Python's (forward
// 10 of 18, decode step 5 of 9).
//
// Every function does exactly what the Python code behind it in cott.py does for the forms it knows, and
// returns None -- before anything has been allocated or launched -- for all others: tensor subclasses, active
// torch modes, levels of torch.func, unusual argument types, and every argument that the Python code refuses, so that
// errors and rare forms have one implementation, there.  An error status of libcott is returned as an int.
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>
#include <torch/csrc/utils/python_arg_parser.h>
#include <ATen/ATen.h>
#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <algorithm>
#include <cstring>
#include "cott.h"

namespace {

// The library that cott.py has loaded, whichever file that is: the module is linked against none, so that a program
// has one copy of it, with one set of options.
#define COTT_ENTRIES(X)                                                                                      \
    X(cott_workspace_bytes_dkdv) X(cott_workspace_bytes_varlen) X(cott_fwd_strided) X(cott_fwd_stateful_strided)  \
    X(cott_bwd_strided) X(cott_bwd_after_fwd) X(cott_bwd_stateful_strided) X(cott_fwd_varlen) X(cott_bwd_varlen)  \
    X(cott_decode_step)
struct Library {
#define X(name) decltype(&::name) name;
    COTT_ENTRIES(X)
#undef X
} lib;

struct Other {};      // (thrown inside this file only: the call is left to the Python code)

// A plain CUDA tensor, or Other.
const at::Tensor& plain(PyObject* o) {
    if (!THPVariable_CheckExact(o)) throw Other();
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || t.is_quantized() || t.is_conj() || t.is_neg()) throw Other();
    const c10::DispatchKeySet ks = t.key_set();
    if (ks.has(c10::DispatchKey::Python) || ks.has(c10::DispatchKey::FuncTorchBatched) || ks.has(c10::DispatchKey::FuncTorchGradWrapper) ||
        ks.has(c10::DispatchKey::Batched) || ks.has(c10::DispatchKey::Functionalize) || !t.has_storage()) throw Other();
    return t;
}
bool none(PyObject* o) { return o == Py_None; }
const at::Tensor& contiguous(PyObject* o) {
    const at::Tensor& t = plain(o);
    if (!t.is_contiguous()) throw Other();
    return t;
}
int truth(PyObject* o) {
    if (o == Py_True) return 1;
    if (o == Py_False) return 0;
    throw Other();
}
cott_dtype dtype_of(const at::Tensor& t) {
    if (t.scalar_type() == at::kBFloat16) return COTT_BF16;
    if (t.scalar_type() == at::kFloat) return COTT_F32;
    throw Other();
}

// Strides of a group of [B,H,N,d] tensors that share them (`dense`: all of them contiguous, no strides needed).
struct Layout {
    cott_strides s;
    bool dense = true;
    void add(const at::Tensor& t, bool first) {
        if (t.dim() != 4) throw Other();
        const auto st = t.strides();
        if (st[3] != 1 && t.size(3) > 1) throw Other();
        if (first) { s.batch = st[0]; s.head = st[1]; s.token = st[2]; }
        else if (s.batch != st[0] || s.head != st[1] || s.token != st[2]) throw Other();
        dense = dense && t.is_contiguous();
    }
    const cott_strides* get() const { return dense ? nullptr : &s; }
};
template <class... T> Layout layout(const at::Tensor& first, const T&... rest) {
    Layout l;
    l.add(first, true);
    (l.add(rest, false), ...);
    return l;
}

cott_scale_params scale(PyObject* m, PyObject* seq_len) {
    cott_scale_params sp;
    sp.m = static_cast<const float*>(contiguous(m).data_ptr());
    sp.seq_len = nullptr;
    sp.seq_len_scalar = 0.f;
    if (none(seq_len)) return sp;
    if (PyFloat_CheckExact(seq_len)) sp.seq_len_scalar = (float)PyFloat_AS_DOUBLE(seq_len);
    else if (PyLong_CheckExact(seq_len)) {
        const double v = PyLong_AsDouble(seq_len);
        if (v == -1.0 && PyErr_Occurred()) { PyErr_Clear(); throw Other(); }
        sp.seq_len_scalar = (float)v;
    } else sp.seq_len = static_cast<const float*>(contiguous(seq_len).data_ptr());
    return sp;
}

at::Tensor empty(at::IntArrayRef shape, const at::Tensor& like, at::ScalarType dt) {
    return at::empty(shape, like.options().dtype(dt).requires_grad(false));
}
at::Tensor room(size_t bytes, const at::Tensor& like) {
    if (bytes == (size_t)-1) throw Other();
    return empty({(int64_t)std::max<size_t>(bytes, 256)}, like, at::kByte);
}
void* ptr(const at::Tensor& t) { return t.data_ptr(); }
float* fptr(const at::Tensor& t) { return static_cast<float*>(t.data_ptr()); }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// (a tensor that came in as an argument goes out as the object that it came in as)
PyObject* wrap(const at::Tensor& t) { return THPVariable_Wrap(t); }

// Runs f with the argument count checked and everything that is not a plain call handed back as None.
template <class F> PyObject* guarded(Py_ssize_t n, Py_ssize_t want, F f) {
    if (n != want) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; }
    // (inside a level of torch.func.grad or jvp even a tensor made from plain ones is a wrapper without storage)
    if (at::impl::torch_function_mode_enabled() || c10::impl::TorchDispatchModeTLS::any_modes_set() ||
        c10::impl::tls_is_dispatch_key_included(c10::DispatchKey::FuncTorchDynamicLayerFrontMode)) Py_RETURN_NONE;
    try {
        return f();
    } catch (const Other&) {
        Py_RETURN_NONE;
    } catch (python_error& e) {
        e.restore();
        return nullptr;
    } catch (const std::exception&) {
        // (an allocation that failed, say: the Python code meets it again and reports it in torch's way)
        Py_RETURN_NONE;
    }
}
// The interpreter lock released while f runs and taken again however it ends: asking for a data pointer may throw.
struct Unlocked {
    PyThreadState* state = PyEval_SaveThread();
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <class F> cott_status without_gil(F f) {
    Unlocked unlocked;
    return f();
}
// The tensors of a tuple or list, held as tensors: another thread may change a list while the lock is released.
void three(PyObject* out, at::Tensor (&o)[3]) {
    if (PyTuple_CheckExact(out) && PyTuple_GET_SIZE(out) == 3) {
        for (int i = 0; i < 3; ++i) o[i] = plain(PyTuple_GET_ITEM(out, i));
    } else if (PyList_CheckExact(out) && PyList_GET_SIZE(out) == 3) {
        for (int i = 0; i < 3; ++i) o[i] = plain(PyList_GET_ITEM(out, i));
    } else throw Other();
}

// q, k, v, m, seq_len, causal, return_state, out, workspace
PyObject* fwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&]() -> PyObject* {
        const at::Tensor &q = plain(a[0]), &k = plain(a[1]), &v = plain(a[2]);
        if (q.dim() != 4 || v.dim() < 1 || v.size(-1) != q.size(3)) throw Other();
        const int B = (int)q.size(0), H = (int)q.size(1), N = (int)q.size(2), d = (int)q.size(3);
        const cott_dtype dt = dtype_of(q);
        const cott_scale_params sp = scale(a[3], a[4]);
        const int causal = truth(a[5]), want_state = truth(a[6]);
        const Layout lq = layout(q, k, v);
        at::Tensor o = none(a[7]) ? at::Tensor() : plain(a[7]);
        if (o.defined()) layout(o);
        at::Tensor ws = none(a[8]) ? at::Tensor() : plain(a[8]);
        const size_t need = ws.defined() ? 0 : lib.cott_workspace_bytes_dkdv(COTT_OP_FWD, dt, B, H, N, d, d, causal);
        if (need == (size_t)-1) throw Other();
        if (!o.defined()) o = at::empty_like(q);
        const Layout lo = layout(o);
        at::Tensor state = want_state ? empty({B, H, d, d}, q, at::kFloat) : at::Tensor();
        if (!ws.defined()) ws = room(need, q);
        void* st = stream();
        const cott_status rc = without_gil([&] {
            return lib.cott_fwd_strided(ptr(q), ptr(k), ptr(v), ptr(o), want_state ? fptr(state) : nullptr, B, H, N, d, causal, dt, lq.get(),
                                    lo.get(), &sp, ptr(ws), (size_t)ws.numel(), st);
        });
        if (rc != COTT_OK) return PyLong_FromLong(rc);
        return want_state ? Py_BuildValue("(NN)", wrap(o), wrap(state)) : wrap(o);
    });
}

// q, k, v, m, seq_len, state_in, return_state, out, workspace
PyObject* fwd_stateful(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 9, [&]() -> PyObject* {
        const at::Tensor &q = plain(a[0]), &k = plain(a[1]), &v = plain(a[2]);
        if (none(a[4]) || q.dim() != 4 || v.dim() < 1 || v.size(-1) != q.size(3)) throw Other();
        const int B = (int)q.size(0), H = (int)q.size(1), N = (int)q.size(2), d = (int)q.size(3);
        const cott_dtype dt = dtype_of(q);
        const cott_scale_params sp = scale(a[3], a[4]);
        at::Tensor state_in = none(a[5]) ? at::Tensor() : contiguous(a[5]);
        if (state_in.defined() && (state_in.scalar_type() != at::kFloat || state_in.sizes() != at::IntArrayRef({B, H, d, d}))) throw Other();
        const int want_state = truth(a[6]);
        const Layout lq = layout(q, k, v);
        at::Tensor o = none(a[7]) ? at::Tensor() : plain(a[7]);
        if (o.defined()) layout(o);
        at::Tensor ws = none(a[8]) ? at::Tensor() : plain(a[8]);
        const size_t need = ws.defined() ? 0 : lib.cott_workspace_bytes_dkdv(COTT_OP_FWD, dt, B, H, N, d, d, 1);
        if (need == (size_t)-1) throw Other();
        if (!o.defined()) o = at::empty_like(q);
        const Layout lo = layout(o);
        at::Tensor state = want_state ? empty({B, H, d, d}, q, at::kFloat) : at::Tensor();
        if (!ws.defined()) ws = room(need, q);
        void* st = stream();
        const cott_status rc = without_gil([&] {
            return lib.cott_fwd_stateful_strided(ptr(q), ptr(k), ptr(v), ptr(o), state_in.defined() ? fptr(state_in) : nullptr,
                                             want_state ? fptr(state) : nullptr, B, H, N, d, dt, lq.get(), lo.get(), &sp, ptr(ws),
                                             (size_t)ws.numel(), st);
        });
        if (rc != COTT_OK) return PyLong_FromLong(rc);
        return want_state ? Py_BuildValue("(NN)", wrap(o), wrap(state)) : wrap(o);
    });
}

// q, k, v, d_o, m, seq_len, causal, workspace, out, fwd_workspace
PyObject* bwd(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&]() -> PyObject* {
        const at::Tensor &q = plain(a[0]), &k = plain(a[1]), &v = plain(a[2]), &d_o = plain(a[3]);
        if (q.dim() != 4 || v.dim() < 1 || v.size(-1) != q.size(3)) throw Other();
        const int B = (int)q.size(0), H = (int)q.size(1), N = (int)q.size(2), d = (int)q.size(3);
        const cott_dtype dt = dtype_of(q);
        const cott_scale_params sp = scale(a[4], a[5]);
        const int causal = truth(a[6]);
        const Layout lq = layout(q, k, v), ld = layout(d_o);
        at::Tensor ws = none(a[7]) ? at::Tensor() : plain(a[7]);
        const bool given = !none(a[8]);
        at::Tensor g[3];
        if (given) {
            three(a[8], g);
            layout(g[0], g[1], g[2]);
        }
        at::Tensor fws = none(a[9]) ? at::Tensor() : plain(a[9]);
        const size_t need = ws.defined() ? 0 : lib.cott_workspace_bytes_dkdv(COTT_OP_BWD, dt, B, H, N, d, d, causal);
        if (need == (size_t)-1) throw Other();
        if (!given) for (int i = 0; i < 3; ++i) g[i] = at::empty_like(q);
        const Layout lg = layout(g[0], g[1], g[2]);
        at::Tensor dm = empty({H}, q, at::kFloat);
        if (!ws.defined()) ws = room(need, q);
        void* st = stream();
        const cott_status rc = without_gil([&] {
            return fws.defined()
                ? lib.cott_bwd_after_fwd(ptr(q), ptr(k), ptr(v), ptr(d_o), ptr(g[0]), ptr(g[1]), ptr(g[2]), fptr(dm), B, H, N, d, causal, dt,
                                     lq.get(), ld.get(), lg.get(), &sp, ptr(fws), ptr(ws), (size_t)ws.numel(), st)
                : lib.cott_bwd_strided(ptr(q), ptr(k), ptr(v), ptr(d_o), ptr(g[0]), ptr(g[1]), ptr(g[2]), fptr(dm), B, H, N, d, causal, dt,
                                   lq.get(), ld.get(), lg.get(), &sp, ptr(ws), (size_t)ws.numel(), st);
        });
        if (rc != COTT_OK) return PyLong_FromLong(rc);
        return Py_BuildValue("(NNNN)", wrap(g[0]), wrap(g[1]), wrap(g[2]), wrap(dm));
    });
}

// q, k, v, d_o, m, seq_len, state_in, d_state_out, return_d_state, workspace, out
PyObject* bwd_stateful(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 11, [&]() -> PyObject* {
        const at::Tensor &q = plain(a[0]), &k = plain(a[1]), &v = plain(a[2]), &d_o = plain(a[3]);
        if (none(a[5]) || q.dim() != 4 || v.dim() < 1 || v.size(-1) != q.size(3)) throw Other();
        const int B = (int)q.size(0), H = (int)q.size(1), N = (int)q.size(2), d = (int)q.size(3);
        const cott_dtype dt = dtype_of(q);
        const cott_scale_params sp = scale(a[4], a[5]);
        at::Tensor s[2];
        for (int i = 0; i < 2; ++i) {
            if (none(a[6 + i])) continue;
            s[i] = contiguous(a[6 + i]);
            if (s[i].scalar_type() != at::kFloat || s[i].sizes() != at::IntArrayRef({B, H, d, d})) throw Other();
        }
        const int want = truth(a[8]);
        const Layout lq = layout(q, k, v), ld = layout(d_o);
        at::Tensor ws = none(a[9]) ? at::Tensor() : plain(a[9]);
        const bool given = !none(a[10]);
        at::Tensor g[3];
        if (given) {
            three(a[10], g);
            layout(g[0], g[1], g[2]);
        }
        const size_t need = ws.defined() ? 0 : lib.cott_workspace_bytes_dkdv(COTT_OP_BWD, dt, B, H, N, d, d, 1);
        if (need == (size_t)-1) throw Other();
        if (!given) { g[0] = at::empty_like(q); g[1] = at::empty_like(k); g[2] = at::empty_like(v); }
        const Layout lg = layout(g[0], g[1], g[2]);
        at::Tensor dm = empty({H}, q, at::kFloat);
        at::Tensor ds = want ? empty({B, H, d, d}, q, at::kFloat) : at::Tensor();
        if (!ws.defined()) ws = room(need, q);
        void* st = stream();
        const cott_status rc = without_gil([&] {
            return lib.cott_bwd_stateful_strided(ptr(q), ptr(k), ptr(v), ptr(d_o), s[0].defined() ? fptr(s[0]) : nullptr,
                                             s[1].defined() ? fptr(s[1]) : nullptr, ptr(g[0]), ptr(g[1]), ptr(g[2]),
                                             want ? fptr(ds) : nullptr, fptr(dm), B, H, N, d, d, dt, lq.get(), nullptr, ld.get(), lg.get(),
                                             nullptr, &sp, ptr(ws), (size_t)ws.numel(), st);
        });
        if (rc != COTT_OK) return PyLong_FromLong(rc);
        PyObject* pd = Py_None;
        if (want) pd = wrap(ds); else Py_INCREF(Py_None);
        return Py_BuildValue("(NNNNN)", wrap(g[0]), wrap(g[1]), wrap(g[2]), pd, wrap(dm));
    });
}

struct PackedCall {
    int B, H, T, d, longest, causal;
    cott_dtype dt;
    cott_scale_params sp;
};
PackedCall packed(PyObject* const* t, int n_t, PyObject* m, PyObject* cu, PyObject* longest, PyObject* seq_len, PyObject* causal) {
    PackedCall c;
    const at::Tensor& q = contiguous(t[0]);
    const at::Tensor& off = contiguous(cu);
    if (off.scalar_type() != at::kInt || off.dim() != 1 || off.numel() < 2 || q.dim() != 3) throw Other();
    for (int i = 1; i < n_t; ++i)
        if (contiguous(t[i]).sizes() != q.sizes()) throw Other();
    c.T = (int)q.size(0); c.H = (int)q.size(1); c.d = (int)q.size(2); c.B = (int)off.numel() - 1;
    c.dt = dtype_of(q);
    c.sp = scale(m, seq_len);
    c.causal = truth(causal);
    if (!PyLong_CheckExact(longest)) throw Other();
    int overflow = 0;
    const long l = PyLong_AsLongAndOverflow(longest, &overflow);
    if (overflow || l < 0 || l > 0x7fffffffL) throw Other();
    c.longest = (int)l;
    return c;
}

// q, k, v, m, cu_seqlens, max_seqlen, seq_len, causal, out, workspace
PyObject* fwd_varlen(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&]() -> PyObject* {
        const PackedCall c = packed(a, 3, a[3], a[4], a[5], a[6], a[7]);
        const at::Tensor &q = plain(a[0]), &k = plain(a[1]), &v = plain(a[2]), &cu = plain(a[4]);
        at::Tensor o = none(a[8]) ? at::Tensor() : plain(a[8]);
        at::Tensor ws = none(a[9]) ? at::Tensor() : plain(a[9]);
        const size_t need = ws.defined() ? 0 : lib.cott_workspace_bytes_varlen(COTT_OP_FWD, c.dt, c.B, c.H, c.T, c.longest, c.d, c.causal);
        if (need == (size_t)-1) throw Other();
        if (!o.defined()) o = at::empty_like(q);
        if (!ws.defined()) ws = room(need, q);
        void* st = stream();
        const cott_status rc = without_gil([&] {
            return lib.cott_fwd_varlen(ptr(q), ptr(k), ptr(v), ptr(o), static_cast<const int*>(ptr(cu)), c.B, c.H, c.T, c.longest, c.d, c.causal,
                                   c.dt, &c.sp, ptr(ws), (size_t)ws.numel(), st);
        });
        if (rc != COTT_OK) return PyLong_FromLong(rc);
        return wrap(o);
    });
}

// q, k, v, d_o, m, cu_seqlens, max_seqlen, seq_len, causal, workspace
PyObject* bwd_varlen(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 10, [&]() -> PyObject* {
        const PackedCall c = packed(a, 4, a[4], a[5], a[6], a[7], a[8]);
        const at::Tensor &q = plain(a[0]), &k = plain(a[1]), &v = plain(a[2]), &d_o = plain(a[3]), &cu = plain(a[5]);
        at::Tensor ws = none(a[9]) ? at::Tensor() : plain(a[9]);
        const size_t need = ws.defined() ? 0 : lib.cott_workspace_bytes_varlen(COTT_OP_BWD, c.dt, c.B, c.H, c.T, c.longest, c.d, c.causal);
        if (need == (size_t)-1) throw Other();
        at::Tensor g[3];
        for (auto& x : g) x = at::empty_like(q);
        at::Tensor dm = empty({c.H}, q, at::kFloat);
        if (!ws.defined()) ws = room(need, q);
        void* st = stream();
        const cott_status rc = without_gil([&] {
            return lib.cott_bwd_varlen(ptr(q), ptr(k), ptr(v), ptr(d_o), ptr(g[0]), ptr(g[1]), ptr(g[2]), fptr(dm),
                                   static_cast<const int*>(ptr(cu)), c.B, c.H, c.T, c.longest, c.d, c.causal, c.dt, &c.sp, ptr(ws),
                                   (size_t)ws.numel(), st);
        });
        if (rc != COTT_OK) return PyLong_FromLong(rc);
        return Py_BuildValue("(NNNN)", wrap(g[0]), wrap(g[1]), wrap(g[2]), wrap(dm));
    });
}

// q, k, v, state, m, seq_len, out
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    return guarded(n, 7, [&]() -> PyObject* {
        const at::Tensor &q = contiguous(a[0]), &k = contiguous(a[1]), &v = contiguous(a[2]), &s = contiguous(a[3]);
        if (none(a[5]) || q.dim() != 3 || v.dim() < 1 || v.size(-1) != q.size(2)) throw Other();
        const int B = (int)q.size(0), H = (int)q.size(1), d = (int)q.size(2);
        if (s.scalar_type() != at::kFloat || s.sizes() != at::IntArrayRef({B, H, d, d})) throw Other();
        const cott_dtype dt = dtype_of(q);
        const cott_scale_params sp = scale(a[4], a[5]);
        at::Tensor o = none(a[6]) ? at::empty_like(v) : plain(a[6]);
        THPObjectPtr po(wrap(o));    // (before the state is updated: nothing may fail after that)
        void* st = stream();
        const cott_status rc = without_gil([&] { return lib.cott_decode_step(ptr(q), ptr(k), ptr(v), fptr(s), ptr(o), B, H, d, dt, &sp, st); });
        return rc == COTT_OK ? po.release() : PyLong_FromLong(rc);
    });
}

// The address of a function of the library by its name, in the order of `entries`.
const char* const entries[] = {
#define X(name) #name,
    COTT_ENTRIES(X)
#undef X
};
constexpr Py_ssize_t kEntries = sizeof(entries) / sizeof(entries[0]);
static_assert(sizeof(Library) == kEntries * sizeof(void*));
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    if (n != kEntries) { PyErr_SetString(PyExc_TypeError, "one address for each of `entries`"); return nullptr; }
    void* addr[kEntries];
    for (Py_ssize_t i = 0; i < n; ++i) {
        addr[i] = PyLong_AsVoidPtr(a[i]);
        if (!addr[i]) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "a null address");
            return nullptr;
        }
    }
    memcpy(&lib, addr, sizeof(lib));
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(fwd), FAST(fwd_stateful), FAST(bwd), FAST(bwd_stateful), FAST(fwd_varlen), FAST(bwd_varlen), FAST(decode_step), FAST(bind),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_cott_torch", "Plain forms of the calls of cott.py.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__cott_torch(void) {
    PyObject* mod = PyModule_Create(&module);
    if (!mod) return nullptr;
    PyObject* names = PyTuple_New(kEntries);
    for (Py_ssize_t i = 0; names && i < kEntries; ++i) {
        PyObject* s = PyUnicode_FromString(entries[i]);
        if (!s) { Py_CLEAR(names); break; }
        PyTuple_SET_ITEM(names, i, s);
    }
    if (!names || PyModule_AddObject(mod, "entries", names) < 0) {
        Py_XDECREF(names);
        Py_DECREF(mod);
        return nullptr;
    }
    return mod;
}
