// The marshalling of the calls that a serving loop makes every iteration, as a CPython extension:
// dtype / shape / contiguity checks, output and scratch tensors from torch's allocator, the current
// stream, and the C ABI call.  binding.py has the same in Python over ctypes, which takes 20 to 33 us a
// call - longer than the kernels of a small step - against 3 to 9 us here (commit 3, attention 4 to 5,
// acceptance and draft step 8 to 9).
//
// Every function returns the call's result, a negative gsd_status as an int (binding.py raises), or
// None when an argument is not the plain case (wrong dtype or shape, another device, a tensor
// subclass, a wrapped tensor of a function transform, a number of another type): binding.py then
// takes its own path, which accepts or refuses the argument as it always did.  The library's
// functions are handed in by address (bind), so that this module calls the library binding.py
// has loaded.
#include <Python.h>
#include <ATen/ATen.h>
#include <ATen/TensorSubclassLikeUtils.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <initializer_list>
#include "gsd_binding.h"

namespace {

struct Table {
    decltype(&gsd_verify_attn) verify_attn;
    decltype(&gsd_verify_attn_workspace_bytes) verify_attn_workspace_bytes;
    decltype(&gsd_accept) accept;
    decltype(&gsd_accept_workspace_bytes) accept_workspace_bytes;
    decltype(&gsd_accept_sampled) accept_sampled;
    decltype(&gsd_accept_sampled_workspace_bytes) accept_sampled_workspace_bytes;
    decltype(&gsd_binding_draft_expand) draft_expand;
    decltype(&gsd_draft_expand_workspace_bytes) draft_expand_workspace_bytes;
    decltype(&gsd_build_mask) build_mask;
    decltype(&gsd_commit_kv) commit_kv;
};
constexpr Py_ssize_t kTable = sizeof(Table) / sizeof(void*);
Table g;       // written under the GIL by bind(), copied under the GIL by every call

// A tensor that the C ABI can take as it is; nullptr otherwise.
const at::Tensor* plain(PyObject* o) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || at::isTensorSubclassLike(t) || !t.is_contiguous()) return nullptr;
    return &t;
}

// Collects the arguments of one call; `ok` turns false at the first that is not the plain case.
struct Args {
    PyObject* const* v;
    bool ok = true;
    int device = -1;

    const at::Tensor* tensor(int i, at::ScalarType dt, int dim) {
        const at::Tensor* t = ok ? plain(v[i]) : nullptr;
        if (!t || t->scalar_type() != dt || t->dim() != dim || (device >= 0 && t->get_device() != device)) {
            ok = false;
            return nullptr;
        }
        device = (int)t->get_device();
        return t;
    }
    const at::Tensor* tensor(int i, at::ScalarType dt, std::initializer_list<int64_t> shape) {
        const at::Tensor* t = tensor(i, dt, (int)shape.size());
        if (t && !t->sizes().equals(at::IntArrayRef(shape))) {
            ok = false;
            return nullptr;
        }
        return t;
    }
    // an optional tensor of which only the address and the size in bytes matter
    const at::Tensor* any_or_none(int i) {
        if (!ok || v[i] == Py_None) return nullptr;
        const at::Tensor* t = plain(v[i]);
        if (!t || (device >= 0 && t->get_device() != device)) ok = false;
        return t;
    }
    int32_t i32(int i) {
        if (!ok) return 0;
        if (!PyLong_CheckExact(v[i])) {
            ok = false;
            return 0;
        }
        int overflow = 0;
        const long x = PyLong_AsLongAndOverflow(v[i], &overflow);
        if (overflow || x < INT32_MIN || x > INT32_MAX) ok = false;
        return (int32_t)x;
    }
    float f32(int i) {
        if (!ok) return 0.f;
        if (!PyFloat_CheckExact(v[i])) {
            ok = false;
            return 0.f;
        }
        return (float)PyFloat_AS_DOUBLE(v[i]);
    }
    // sizes the C ABI holds in 32 bits
    int32_t size(const at::Tensor* t, int d) {
        if (!ok) return 0;
        const int64_t n = t->size(d);
        if (n > INT32_MAX) ok = false;
        return (int32_t)n;
    }
};

template <class T>
T* ptr(const at::Tensor* t) { return t ? static_cast<T*>(t->data_ptr()) : nullptr; }

at::Tensor empty(at::IntArrayRef shape, at::ScalarType dt, int device) {
    return at::empty(shape, at::TensorOptions().dtype(dt).device(c10::Device(c10::kCUDA, (c10::DeviceIndex)device)));
}

// The device made current, its current stream, and the scratch of the call: the caller's or a new one.
struct Call {
    c10::cuda::CUDAGuard guard;
    void* stream;
    at::Tensor own;
    void* ws = nullptr;
    size_t ws_bytes = 0;

    explicit Call(int device) : guard((c10::DeviceIndex)device), stream(c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream()) {}
    void scratch(const at::Tensor* given, size_t need, int device) {
        if (!given && need) own = empty({(int64_t)need}, at::kByte, device);
        const at::Tensor* t = given ? given : need ? &own : nullptr;
        if (t) {
            ws = t->data_ptr();
            ws_bytes = (size_t)t->numel() * t->element_size();
        }
    }
};

template <class F>
int unlocked(F f) {      // (ctypes lets other threads run during a call, too)
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = f();
    Py_END_ALLOW_THREADS
    return rc;
}

PyObject* tuple_of(std::initializer_list<PyObject*> items) {     // takes the references
    PyObject* t = PyTuple_New((Py_ssize_t)items.size());
    Py_ssize_t i = 0;
    for (PyObject* o : items) {
        if (t) PyTuple_SET_ITEM(t, i++, o);
        else Py_XDECREF(o);
    }
    return t;
}

#define GSD_PY_BEGIN(n)                                                                         \
    HANDLE_TH_ERRORS                                                                            \
    if (nargs != (n)) { PyErr_SetString(PyExc_TypeError, "wrong number of arguments"); return nullptr; } \
    Args a{argv};                                                                               \
    const Table lib = g;
#define GSD_PY_PLAIN if (!a.ok) Py_RETURN_NONE
#define GSD_PY_END END_HANDLE_TH_ERRORS

// bind(addresses): one per entry of Table, in its order
PyObject* py_bind(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    if (nargs != kTable) { PyErr_SetString(PyExc_TypeError, "bind: wrong number of addresses"); return nullptr; }
    void* at[kTable];
    for (Py_ssize_t i = 0; i < nargs; ++i) {
        at[i] = PyLong_AsVoidPtr(argv[i]);
        if (PyErr_Occurred()) return nullptr;
    }
    memcpy(&g, at, sizeof g);
    Py_RETURN_NONE;
}

// (q, k_cache, v_cache, draft_k, draft_v, mask, seq_lens, out, scale, num_splits, kernel, workspace, status)
PyObject* py_verify_attn(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    GSD_PY_BEGIN(13)
    const at::Tensor* q = a.tensor(0, at::kBFloat16, 4);
    const at::Tensor* kc = a.tensor(1, at::kBFloat16, 4);
    GSD_PY_PLAIN;
    gsd_attn_params p;
    p.B = a.size(q, 0); p.N = a.size(q, 1); p.Hq = a.size(q, 2); p.D = a.size(q, 3);
    p.Lmax = a.size(kc, 1); p.Hkv = a.size(kc, 2);
    GSD_PY_PLAIN;
    if (kc->size(0) != p.B || kc->size(3) != p.D) Py_RETURN_NONE;
    const at::Tensor* vc = a.tensor(2, at::kBFloat16, {p.B, p.Lmax, p.Hkv, p.D});
    const at::Tensor* dk = a.tensor(3, at::kBFloat16, {p.B, p.N, p.Hkv, p.D});
    const at::Tensor* dv = a.tensor(4, at::kBFloat16, {p.B, p.N, p.Hkv, p.D});
    const at::Tensor* sl = a.tensor(6, at::kInt, {p.B});
    GSD_PY_PLAIN;
    const at::Tensor* mask = plain(argv[5]);
    if (!mask || mask->get_device() != a.device || (mask->scalar_type() != at::kInt && mask->scalar_type() != at::kUInt32) ||
        !mask->sizes().equals({p.B, p.N, (p.N + 31) / 32}))
        Py_RETURN_NONE;
    const at::Tensor* out = argv[7] == Py_None ? nullptr : a.tensor(7, at::kBFloat16, {p.B, p.N, p.Hq, p.D});
    p.softmax_scale = a.f32(8); p.num_splits = a.i32(9); p.kernel = a.i32(10);
    const at::Tensor* ws = a.any_or_none(11);
    const at::Tensor* status = a.any_or_none(12);
    GSD_PY_PLAIN;
    Call c(a.device);
    at::Tensor made;
    if (!out) {
        made = empty(q->sizes(), at::kBFloat16, a.device);
        out = &made;
    }
    c.scratch(ws, ws ? 0 : lib.verify_attn_workspace_bytes(&p), a.device);
    const int rc = unlocked([&] {
        return lib.verify_attn(ptr<void>(q), ptr<void>(kc), ptr<void>(vc), ptr<void>(dk), ptr<void>(dv), ptr<uint32_t>(mask),
                               ptr<int32_t>(sl), ptr<void>(out), &p, c.ws, c.ws_bytes, ptr<int32_t>(status), c.stream);
    });
    if (rc != GSD_OK) return PyLong_FromLong(rc);
    if (!made.defined()) {
        Py_INCREF(argv[7]);
        return argv[7];
    }
    return THPVariable_Wrap(std::move(made));
    GSD_PY_END
}

// The acceptance calls share their graph and their outputs.
struct Graph {
    gsd_accept_params p;
    const at::Tensor *logits, *tok, *pptr, *pidx;
};
bool graph_args(Args& a, int at_tcap, Graph& s) {
    s.logits = a.tensor(0, at::kFloat, 3);
    s.pidx = a.tensor(3, at::kInt, 2);
    if (!a.ok) return false;
    s.p.B = a.size(s.logits, 0); s.p.N = a.size(s.logits, 1); s.p.V = a.size(s.logits, 2);
    s.p.Ecap = a.size(s.pidx, 1);
    s.p.Tcap = a.i32(at_tcap);
    if (!a.ok || s.pidx->size(0) != s.p.B) return a.ok = false;
    if (s.p.Tcap == 0) s.p.Tcap = s.p.N;
    s.tok = a.tensor(1, at::kInt, {s.p.B, s.p.N});
    s.pptr = a.tensor(2, at::kInt, {s.p.B, (int64_t)s.p.N + 1});
    return a.ok && s.p.Tcap > 0;
}
struct Accepted {
    at::Tensor toks, lens, nodes;
    Accepted(const gsd_accept_params& p, bool want_nodes, int device)
        : toks(empty({p.B, p.Tcap}, at::kInt, device)), lens(empty({p.B}, at::kInt, device)) {
        if (want_nodes) nodes = empty({p.B, p.Tcap}, at::kInt, device);
    }
    int32_t* nodes_ptr() { return nodes.defined() ? static_cast<int32_t*>(nodes.data_ptr()) : nullptr; }
    PyObject* result() {
        PyObject* n = nodes.defined() ? THPVariable_Wrap(nodes) : Py_NewRef(Py_None);
        return tuple_of({THPVariable_Wrap(toks), THPVariable_Wrap(lens), n});
    }
};
bool flag(Args& a, int i) {
    if (a.v[i] != Py_True && a.v[i] != Py_False) a.ok = false;
    return a.v[i] == Py_True;
}

// (logits, draft_tokens, parent_ptr, parent_idx, Tcap, want_nodes, workspace, status)
PyObject* py_accept(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    GSD_PY_BEGIN(8)
    Graph s;
    if (!graph_args(a, 4, s)) Py_RETURN_NONE;
    const bool want_nodes = flag(a, 5);
    const at::Tensor* ws = a.any_or_none(6);
    const at::Tensor* status = a.any_or_none(7);
    GSD_PY_PLAIN;
    Call c(a.device);
    Accepted out(s.p, want_nodes, a.device);
    c.scratch(ws, ws ? 0 : std::max<size_t>(lib.accept_workspace_bytes(&s.p), 8), a.device);
    const int rc = unlocked([&] {
        return lib.accept(ptr<float>(s.logits), ptr<int32_t>(s.tok), ptr<int32_t>(s.pptr), ptr<int32_t>(s.pidx),
                          ptr<int32_t>(&out.toks), ptr<int32_t>(&out.lens), out.nodes_ptr(), &s.p, c.ws, c.ws_bytes,
                          ptr<int32_t>(status), c.stream);
    });
    return rc != GSD_OK ? PyLong_FromLong(rc) : out.result();
    GSD_PY_END
}

// (logits, draft_tokens, parent_ptr, parent_idx, draft_q, u_accept, u_sample, draft_logits, Tcap, want_nodes, workspace, status)
PyObject* py_accept_sampled(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    GSD_PY_BEGIN(12)
    Graph s;
    if (!graph_args(a, 8, s)) Py_RETURN_NONE;
    const at::Tensor* dq = a.tensor(4, at::kFloat, {s.p.B, s.p.N});
    const at::Tensor* ua = a.tensor(5, at::kFloat, {s.p.B, s.p.N});
    const at::Tensor* us = a.tensor(6, at::kFloat, {s.p.B});
    const at::Tensor* dl = argv[7] == Py_None ? nullptr : a.tensor(7, at::kFloat, {s.p.B, s.p.N, s.p.V});
    const bool want_nodes = flag(a, 9);
    const at::Tensor* ws = a.any_or_none(10);
    const at::Tensor* status = a.any_or_none(11);
    GSD_PY_PLAIN;
    Call c(a.device);
    Accepted out(s.p, want_nodes, a.device);
    c.scratch(ws, ws ? 0 : std::max<size_t>(lib.accept_sampled_workspace_bytes(&s.p), 8), a.device);
    const int rc = unlocked([&] {
        return lib.accept_sampled(ptr<float>(s.logits), ptr<int32_t>(s.tok), ptr<int32_t>(s.pptr), ptr<int32_t>(s.pidx),
                                  ptr<float>(dl), ptr<float>(dq), ptr<float>(ua), ptr<float>(us), ptr<int32_t>(&out.toks),
                                  ptr<int32_t>(&out.lens), out.nodes_ptr(), &s.p, c.ws, c.ws_bytes, ptr<int32_t>(status),
                                  c.stream);
    });
    return rc != GSD_OK ? PyLong_FromLong(rc) : out.result();
    GSD_PY_END
}

// (logits, frontier, frontier_len, tokens, tree_parent, merge_to, leaf, prob, num_nodes, k, tau, theta_prob, theta_sib,
//  workspace, status)
PyObject* py_draft_expand(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    GSD_PY_BEGIN(15)
    const at::Tensor* logits = a.tensor(0, at::kFloat, 3);
    const at::Tensor* tokens = a.tensor(3, at::kInt, 2);
    GSD_PY_PLAIN;
    gsd_draft_params p;
    p.B = a.size(logits, 0); p.F = a.size(logits, 1); p.V = a.size(logits, 2); p.Ncap = a.size(tokens, 1);
    GSD_PY_PLAIN;
    if (tokens->size(0) != p.B) Py_RETURN_NONE;
    const at::Tensor* frontier = a.tensor(1, at::kInt, {p.B, p.F});
    const at::Tensor* frontier_len = a.tensor(2, at::kInt, {p.B});
    const at::Tensor* parent = a.tensor(4, at::kInt, {p.B, p.Ncap});
    const at::Tensor* merge = a.tensor(5, at::kInt, {p.B, p.Ncap});
    const at::Tensor* leaf = a.tensor(6, at::kByte, {p.B, p.Ncap});
    const at::Tensor* prob = a.tensor(7, at::kFloat, {p.B, p.Ncap});
    const at::Tensor* num_nodes = a.tensor(8, at::kInt, {p.B});
    p.k = a.i32(9); p.tau = a.i32(10); p.theta_prob = a.f32(11); p.theta_sib = a.f32(12);
    const at::Tensor* ws = a.any_or_none(13);
    const at::Tensor* status = a.any_or_none(14);
    GSD_PY_PLAIN;
    if (p.k < 1 || p.k > GSD_DRAFT_MAX_K) Py_RETURN_NONE;
    Call c(a.device);
    at::Tensor nf = empty({p.B, (int64_t)p.F * p.k}, at::kInt, a.device);
    at::Tensor nfl = empty({p.B}, at::kInt, a.device);
    c.scratch(ws, ws ? 0 : std::max<size_t>(lib.draft_expand_workspace_bytes(&p), 8), a.device);
    const int rc = unlocked([&] {
        return lib.draft_expand(ptr<float>(logits), ptr<int32_t>(frontier), ptr<int32_t>(frontier_len), ptr<int32_t>(tokens),
                                ptr<int32_t>(parent), ptr<int32_t>(merge), ptr<uint8_t>(leaf), ptr<float>(prob),
                                ptr<int32_t>(num_nodes), ptr<int32_t>(&nf), ptr<int32_t>(&nfl), &p, c.ws, c.ws_bytes,
                                ptr<int32_t>(status), c.stream);
    });
    return rc != GSD_OK ? PyLong_FromLong(rc) : tuple_of({THPVariable_Wrap(nf), THPVariable_Wrap(nfl)});
    GSD_PY_END
}

// (parent_ptr, parent_idx, out, status)
PyObject* py_build_mask(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    GSD_PY_BEGIN(4)
    const at::Tensor* pptr = a.tensor(0, at::kInt, 2);
    const at::Tensor* pidx = a.tensor(1, at::kInt, 2);
    GSD_PY_PLAIN;
    const int32_t B = a.size(pptr, 0), N = a.size(pptr, 1) - 1, Ecap = a.size(pidx, 1);
    if (!a.ok || N < 1 || pidx->size(0) != B) Py_RETURN_NONE;
    const at::Tensor* status = a.any_or_none(3);
    GSD_PY_PLAIN;
    if (argv[2] != Py_None) Py_RETURN_NONE;
    Call c(a.device);
    at::Tensor out = empty({B, N, (N + 31) / 32}, at::kInt, a.device);
    const int rc = unlocked([&] {
        return lib.build_mask(ptr<int32_t>(pptr), ptr<int32_t>(pidx), ptr<uint32_t>(&out), B, N, Ecap, ptr<int32_t>(status), c.stream);
    });
    return rc != GSD_OK ? PyLong_FromLong(rc) : THPVariable_Wrap(std::move(out));
    GSD_PY_END
}

// (k_cache, v_cache, draft_k, draft_v, accepted_nodes, accepted_len, seq_lens, status); returns 0 when done
PyObject* py_commit_kv(PyObject*, PyObject* const* argv, Py_ssize_t nargs) {
    GSD_PY_BEGIN(8)
    const at::Tensor* kc = a.tensor(0, at::kBFloat16, 4);
    const at::Tensor* dk = a.tensor(2, at::kBFloat16, 4);
    const at::Tensor* nodes = a.tensor(4, at::kInt, 2);
    GSD_PY_PLAIN;
    gsd_commit_params p;
    p.B = a.size(kc, 0); p.Lmax = a.size(kc, 1); p.Hkv = a.size(kc, 2); p.D = a.size(kc, 3);
    p.N = a.size(dk, 1); p.Tcap = a.size(nodes, 1);
    GSD_PY_PLAIN;
    if (nodes->size(0) != p.B || !dk->sizes().equals({p.B, p.N, p.Hkv, p.D})) Py_RETURN_NONE;
    const at::Tensor* vc = a.tensor(1, at::kBFloat16, {p.B, p.Lmax, p.Hkv, p.D});
    const at::Tensor* dv = a.tensor(3, at::kBFloat16, {p.B, p.N, p.Hkv, p.D});
    const at::Tensor* len = a.tensor(5, at::kInt, {p.B});
    const at::Tensor* sl = a.tensor(6, at::kInt, {p.B});
    const at::Tensor* status = a.any_or_none(7);
    GSD_PY_PLAIN;
    Call c(a.device);
    return PyLong_FromLong(unlocked([&] {
        return lib.commit_kv(ptr<void>(kc), ptr<void>(vc), ptr<void>(dk), ptr<void>(dv), ptr<int32_t>(nodes), ptr<int32_t>(len),
                             ptr<int32_t>(sl), &p, ptr<int32_t>(status), c.stream);
    }));
    GSD_PY_END
}

#define GSD_PY_FN(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {GSD_PY_FN(bind), GSD_PY_FN(verify_attn), GSD_PY_FN(accept), GSD_PY_FN(accept_sampled),
                         GSD_PY_FN(draft_expand), GSD_PY_FN(build_mask), GSD_PY_FN(commit_kv), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// (the classes of torch's headers are compiled in: binding.py refuses another version's)
PyMODINIT_FUNC PyInit__native(void) {
    PyObject* m = PyModule_Create(&module_def);
    if (m && PyModule_AddStringConstant(m, "torch_version", GSD_TORCH_VERSION) != 0) Py_CLEAR(m);
    return m;
}
