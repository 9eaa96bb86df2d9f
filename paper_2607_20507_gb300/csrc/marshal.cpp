// marshal.cpp -- the argument marshalling of binding.py's calls as a CPython
// module (_marshal): the same checks, the same outputs and the same C ABI
// calls, without interpreter work between them.  A step on small inputs is
// bound by the host (one call: 22 us through ctypes on the Grace cores, of
// which the kernel launches are 4).
//
// Every function returns the call's result; None when an argument is not what
// the call takes (binding.py then runs its own checks, which say what is
// wrong); or the status, an int, when the library reports an error.  Nothing
// is kept between calls but the workspaces that binding.py hands out.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ops/empty.h>
#include <ATen/ops/empty_like.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <map>
#include <tuple>

#include "cachespec.h"

namespace {

// binding._workspace_of(kind, device_index, bytes, stream) -> (Tensor, whether to keep it)
PyObject* g_workspace_of = nullptr;

// A device tensor of the given type and rank, contiguous, on the device of
// the call; `t` is set to it.
bool need(PyObject* o, at::ScalarType type, int ndim, c10::Device dev, const at::Tensor** t) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::Tensor& x = THPVariable_Unpack(o);
    *t = &x;
    return x.scalar_type() == type && x.dim() == ndim && x.is_cuda() && x.device() == dev && x.is_contiguous();
}

// The first tensor of a call, whose device the others share.
bool first(PyObject* o, at::ScalarType type, int ndim, c10::Device* dev, const at::Tensor** t) {
    if (!THPVariable_CheckExact(o)) return false;
    *dev = THPVariable_Unpack(o).device();
    return need(o, type, ndim, *dev, t);
}

bool logits(PyObject* o, int ndim, c10::Device* dev, const at::Tensor** t) {
    if (!THPVariable_CheckExact(o)) return false;
    const at::ScalarType s = THPVariable_Unpack(o).scalar_type();
    return (s == at::kFloat || s == at::kBFloat16) && first(o, s, ndim, dev, t);
}

bool small_int(PyObject* o, int32_t* v) {
    if (!PyLong_CheckExact(o)) return false;
    int over = 0;
    const long x = PyLong_AsLongAndOverflow(o, &over);
    *v = (int32_t)x;
    return !over && x == *v;
}

bool number(PyObject* o, float* v) {
    if (PyFloat_CheckExact(o)) {
        *v = (float)PyFloat_AS_DOUBLE(o);
        return true;
    }
    int32_t i;
    if (!small_int(o, &i)) return false;
    *v = (float)i;
    return true;
}

// None (the device's current stream) or a stream handle.
bool stream_of(PyObject* o, c10::Device dev, cs_stream_t* s) {
    if (o == Py_None) {
        *s = c10::cuda::getCurrentCUDAStream(dev.index()).stream();
        return true;
    }
    if (!PyLong_CheckExact(o)) return false;
    *s = static_cast<cs_stream_t>(PyLong_AsVoidPtr(o));
    if (!PyErr_Occurred()) return true;
    PyErr_Clear();   // (more than a handle: binding.py passes on its low bits)
    return false;
}

enum Kind { kAttn, kTreeAttn, kAccept, kTreeAccept, kSample, kRoute };
const char* const kKinds[] = {"attn", "tree_attn", "accept", "tree_accept", "sample", "route"};

// Scratch of a call; `hold` is the kept workspace it lies in.
struct Scratch {
    void* ptr = nullptr;
    size_t bytes = 0;
    at::Tensor hold;
};

// The caller's workspace, or the one that binding.py keeps for the size and the stream.
// Asking binding.py runs Python code, in which another thread may come here:
// nothing of the map is held meanwhile.
bool workspace(PyObject* o, Kind kind, c10::Device dev, size_t bytes, cs_stream_t s, Scratch* w) {
    if (o != Py_None) {
        if (!THPVariable_CheckExact(o)) return false;
        w->hold = THPVariable_Unpack(o);
    } else {
        using Key = std::tuple<int, int, size_t, cs_stream_t>;
        static auto* kept = new std::map<Key, at::Tensor>;   // under the interpreter lock
        const Key key{(int)kind, (int)dev.index(), bytes, s};
        const auto it = kept->find(key);
        if (it != kept->end()) {
            w->hold = it->second;
        } else {
            PyObject* r = PyObject_CallFunction(g_workspace_of, "sinK", kKinds[kind], (int)dev.index(), (Py_ssize_t)bytes,
                                                (unsigned long long)reinterpret_cast<uintptr_t>(s));
            if (!r) throw python_error();
            w->hold = THPVariable_Unpack(PyTuple_GET_ITEM(r, 0));
            if (PyTuple_GET_ITEM(r, 1) == Py_True) kept->emplace(key, w->hold);   // (binding.py owns the workspace)
            Py_DECREF(r);
        }
    }
    w->ptr = w->hold.data_ptr();
    w->bytes = w->hold.nbytes();
    return true;
}

// The interpreter lock is not held while outputs are allocated and the library
// launches: an allocation or a launch that waits for the device stops this
// thread only, and a host callback that the device waits for may need the lock.
template <typename F>
cs_status launch(F call) {
    struct Unlocked {
        PyThreadState* const held = PyEval_SaveThread();
        ~Unlocked() { PyEval_RestoreThread(held); }
    } unlocked;
    return call();
}

at::Tensor ints(at::IntArrayRef shape, c10::Device dev) { return at::empty(shape, at::TensorOptions(at::kInt).device(dev)); }

PyObject* status(cs_status st) { return PyLong_FromLong(st); }

// The given output, checked; none given leaves `t` undefined, for make().
bool output(PyObject* o, int ndim, c10::Device dev, at::Tensor* t) {
    if (o == Py_None) return true;
    const at::Tensor* x;
    if (!need(o, at::kInt, ndim, dev, &x)) return false;
    *t = *x;
    return true;
}

void make(at::Tensor* t, at::IntArrayRef shape, c10::Device dev) {
    if (!t->defined()) *t = ints(shape, dev);
}

PyObject* pair(const at::Tensor& a, const at::Tensor& b) {
    return Py_BuildValue("(NN)", THPVariable_Wrap(a), THPVariable_Wrap(b));
}

#define CALL(name, count)                                                              \
    PyObject* name(PyObject*, PyObject* const* a, Py_ssize_t n_args) {                 \
        HANDLE_TH_ERRORS                                                               \
        if (n_args != count) Py_RETURN_NONE;
#define CALL_END                                                                       \
        END_HANDLE_TH_ERRORS                                                           \
    }

// q, k_pages, v_pages, page_table, ctx_lens, n_draft | parents, out, workspace, sm_scale, stream
PyObject* attention(PyObject* const* a, bool tree) {
    const at::Tensor *q, *k, *v, *table, *lens, *par = nullptr, *o;
    c10::Device dev(c10::kCPU);
    int32_t n_draft = 0;
    float scale;
    cs_stream_t s;
    if (!first(a[0], at::kBFloat16, 4, &dev, &q) || !need(a[1], at::kBFloat16, 4, dev, &k) ||
        !need(a[2], at::kBFloat16, 4, dev, &v) || !need(a[3], at::kInt, 2, dev, &table) ||
        !need(a[4], at::kInt, 1, dev, &lens) || v->sizes() != k->sizes() || !number(a[8], &scale) ||
        !stream_of(a[9], dev, &s))
        Py_RETURN_NONE;
    const int64_t rows = q->size(1);
    if (tree) {
        if (!need(a[5], at::kInt, 2, dev, &par) || par->size(0) != q->size(0) || par->size(1) != rows) Py_RETURN_NONE;
    } else if (!small_int(a[5], &n_draft) || rows != n_draft + 1) {
        Py_RETURN_NONE;
    }
    if (a[6] != Py_None && !need(a[6], at::kBFloat16, 4, dev, &o)) Py_RETURN_NONE;
    const cs_attn_dims d{(int32_t)q->size(0), (int32_t)q->size(2), (int32_t)k->size(1), (int32_t)q->size(3),
                         (int32_t)k->size(2), (int32_t)table->size(1), (int32_t)k->size(0), scale};
    Scratch ws;
    size_t bytes = 0;
    if (a[7] == Py_None)
        bytes = tree ? cs_tree_verify_attention_workspace_bytes(&d, (int32_t)rows)
                     : cs_verify_attention_workspace_bytes(&d, n_draft);
    if (!workspace(a[7], tree ? kTreeAttn : kAttn, dev, bytes, s, &ws)) Py_RETURN_NONE;
    at::Tensor out;
    const int32_t *tp = (const int32_t*)table->data_ptr(), *lp = (const int32_t*)lens->data_ptr();
    const cs_status st = launch([&] {
        out = a[6] == Py_None ? at::empty_like(*q) : *o;
        return tree ? cs_tree_verify_attention(&d, q->data_ptr(), k->data_ptr(), v->data_ptr(), tp, lp,
                                               (const int32_t*)par->data_ptr(), (int32_t)rows, out.data_ptr(), ws.ptr,
                                               ws.bytes, s)
                    : cs_verify_attention(&d, q->data_ptr(), k->data_ptr(), v->data_ptr(), tp, lp, n_draft,
                                          out.data_ptr(), ws.ptr, ws.bytes, s);
    });
    if (st != CS_OK) return status(st);
    return a[6] == Py_None ? THPVariable_Wrap(out) : Py_NewRef(a[6]);
}

CALL(verify_attention, 10)
    return attention(a, false);
CALL_END

CALL(tree_verify_attention, 10)
    return attention(a, true);
CALL_END

// target, draft, draft_tokens, uniforms, temperature, out_tokens, out_n_accepted, workspace, stream
CALL(spec_accept, 9)
    const at::Tensor *t, *q = nullptr, *x, *u;
    c10::Device dev(c10::kCPU);
    float T;
    cs_stream_t s;
    if (!logits(a[0], 3, &dev, &t)) Py_RETURN_NONE;
    const int64_t B = t->size(0), k = t->size(1) - 1, V = t->size(2);
    if (a[1] != Py_None && (!need(a[1], t->scalar_type(), 3, dev, &q) || q->size(0) != B || q->size(1) != k || q->size(2) != V))
        Py_RETURN_NONE;
    if (k < 0 || !need(a[2], at::kInt, 2, dev, &x) || !need(a[3], at::kFloat, 2, dev, &u) || !number(a[4], &T) ||
        !stream_of(a[8], dev, &s))
        Py_RETURN_NONE;
    const cs_accept_dims d{(int32_t)B, (int32_t)V, t->scalar_type() == at::kFloat ? CS_F32 : CS_BF16};
    at::Tensor tokens, count;
    Scratch ws;
    const size_t bytes = a[7] == Py_None ? cs_spec_accept_workspace_bytes(&d, (int32_t)k) : 0;
    if (!output(a[5], 2, dev, &tokens) || !output(a[6], 1, dev, &count) ||
        !workspace(a[7], kAccept, dev, bytes, s, &ws))
        Py_RETURN_NONE;
    const cs_status st = launch([&] {
        make(&tokens, {B, k + 1}, dev);
        make(&count, {B}, dev);
        return cs_spec_accept(&d, t->data_ptr(), q ? q->data_ptr() : nullptr, (const int32_t*)x->data_ptr(),
                              (const float*)u->data_ptr(), (int32_t)k, T, (int32_t*)tokens.data_ptr(),
                              (int32_t*)count.data_ptr(), ws.ptr, ws.bytes, s);
    });
    return st != CS_OK ? status(st) : pair(tokens, count);
CALL_END

// target, draft, parents, node_tokens, uniforms, temperature, out_tokens, out_path, out_n_accepted, workspace, stream
CALL(tree_accept, 11)
    const at::Tensor *t, *q = nullptr, *par, *x, *u;
    c10::Device dev(c10::kCPU);
    float T;
    cs_stream_t s;
    if (!logits(a[0], 3, &dev, &t) || (a[1] != Py_None && (!need(a[1], t->scalar_type(), 3, dev, &q) || q->sizes() != t->sizes())) ||
        !need(a[2], at::kInt, 2, dev, &par) || !need(a[3], at::kInt, 2, dev, &x) ||
        !need(a[4], at::kFloat, 2, dev, &u) || !number(a[5], &T) || !stream_of(a[10], dev, &s))
        Py_RETURN_NONE;
    const int64_t B = t->size(0), n = t->size(1);
    for (const at::Tensor* y : {par, x})
        if (y->size(0) != B || y->size(1) != n) Py_RETURN_NONE;
    const cs_accept_dims d{(int32_t)B, (int32_t)t->size(2), t->scalar_type() == at::kFloat ? CS_F32 : CS_BF16};
    at::Tensor tokens, path, count;
    Scratch ws;
    const size_t bytes = a[9] == Py_None ? cs_tree_accept_workspace_bytes(&d, (int32_t)n) : 0;
    if (!output(a[6], 2, dev, &tokens) || !output(a[7], 2, dev, &path) || !output(a[8], 1, dev, &count) ||
        !workspace(a[9], kTreeAccept, dev, bytes, s, &ws))
        Py_RETURN_NONE;
    const cs_status st = launch([&] {
        make(&tokens, {B, n}, dev);
        make(&path, {B, n}, dev);
        make(&count, {B}, dev);
        return cs_tree_accept(&d, t->data_ptr(), q ? q->data_ptr() : nullptr, (const int32_t*)par->data_ptr(),
                              (const int32_t*)x->data_ptr(), (const float*)u->data_ptr(), (int32_t)n, T,
                              (int32_t*)tokens.data_ptr(), (int32_t*)path.data_ptr(), (int32_t*)count.data_ptr(),
                              ws.ptr, ws.bytes, s);
    });
    if (st != CS_OK) return status(st);
    return Py_BuildValue("(NNN)", THPVariable_Wrap(tokens), THPVariable_Wrap(path), THPVariable_Wrap(count));
CALL_END

// logits, uniforms, temperature, out_tokens, workspace, stream
CALL(sample, 6)
    const at::Tensor *z, *u;
    c10::Device dev(c10::kCPU);
    float T;
    cs_stream_t s;
    if (!logits(a[0], 2, &dev, &z) || !need(a[1], at::kFloat, 1, dev, &u) || !number(a[2], &T) ||
        !stream_of(a[5], dev, &s))
        Py_RETURN_NONE;
    const cs_accept_dims d{(int32_t)z->size(0), (int32_t)z->size(1), z->scalar_type() == at::kFloat ? CS_F32 : CS_BF16};
    at::Tensor tokens;
    Scratch ws;
    const size_t bytes = a[4] == Py_None ? cs_sample_workspace_bytes(&d) : 0;
    if (!output(a[3], 1, dev, &tokens) || !workspace(a[4], kSample, dev, bytes, s, &ws)) Py_RETURN_NONE;
    const cs_status st = launch([&] {
        make(&tokens, {z->size(0)}, dev);
        return cs_sample(&d, z->data_ptr(), (const float*)u->data_ptr(), T, (int32_t*)tokens.data_ptr(), ws.ptr,
                         ws.bytes, s);
    });
    return st != CS_OK ? status(st) : THPVariable_Wrap(tokens);
CALL_END

// emb, centroids, inv_norms, tau, workspace, stream (outputs are new)
CALL(route, 6)
    const at::Tensor *e, *c, *inv;
    c10::Device dev(c10::kCPU);
    float tau;
    cs_stream_t s;
    if (!first(a[0], at::kBFloat16, 2, &dev, &e) || !need(a[1], at::kBFloat16, 2, dev, &c) ||
        !need(a[2], at::kFloat, 1, dev, &inv) || !number(a[3], &tau) || !stream_of(a[5], dev, &s) || c->size(0) == 0 ||
        c->size(1) != e->size(1))
        Py_RETURN_NONE;
    const int64_t B = e->size(0);
    const cs_route_dims d{(int32_t)B, (int32_t)c->size(0), (int32_t)e->size(1)};
    Scratch ws;
    const size_t bytes = a[4] == Py_None ? cs_route_workspace_bytes(&d) : 0;
    if (!workspace(a[4], kRoute, dev, bytes, s, &ws)) Py_RETURN_NONE;
    at::Tensor group, best, score;
    const cs_status st = launch([&] {
        make(&group, {B}, dev);
        make(&best, {B}, dev);
        score = at::empty({B}, at::TensorOptions(at::kFloat).device(dev));
        return cs_route(&d, e->data_ptr(), c->data_ptr(), (const float*)inv->data_ptr(), tau,
                        (int32_t*)group.data_ptr(), (int32_t*)best.data_ptr(), (float*)score.data_ptr(), ws.ptr,
                        ws.bytes, s);
    });
    if (st != CS_OK) return status(st);
    return Py_BuildValue("(NNN)", THPVariable_Wrap(group), THPVariable_Wrap(best), THPVariable_Wrap(score));
CALL_END

// new_k, new_v, k_pages, v_pages, page_table, ctx_lens, stream.  True when done.
CALL(kv_append, 7)
    const at::Tensor *nk, *nv, *k, *v, *table, *lens;
    c10::Device dev(c10::kCPU);
    cs_stream_t s;
    if (!first(a[2], at::kBFloat16, 4, &dev, &k) || !need(a[0], at::kBFloat16, 4, dev, &nk) ||
        !need(a[1], at::kBFloat16, 4, dev, &nv) || !need(a[3], at::kBFloat16, 4, dev, &v) ||
        !need(a[4], at::kInt, 2, dev, &table) || !need(a[5], at::kInt, 1, dev, &lens) || !stream_of(a[6], dev, &s) ||
        nk->sizes() != nv->sizes() || k->sizes() != v->sizes() || k->size(1) != nk->size(2) || k->size(3) != nk->size(3))
        Py_RETURN_NONE;
    const int32_t hkv = (int32_t)k->size(1);
    const cs_attn_dims d{(int32_t)nk->size(0), hkv, hkv, (int32_t)k->size(3), (int32_t)k->size(2),
                         (int32_t)table->size(1), (int32_t)k->size(0), 0.f};
    const cs_status st = launch([&] {
        return cs_kv_append(&d, nk->data_ptr(), nv->data_ptr(), k->data_ptr(), v->data_ptr(),
                            (const int32_t*)table->data_ptr(), (const int32_t*)lens->data_ptr(), (int32_t)nk->size(1),
                            s);
    });
    if (st != CS_OK) return status(st);
    Py_RETURN_TRUE;
CALL_END

// ctx_lens, n_accepted, n_draft, stream.  True when done.
CALL(kv_commit, 4)
    const at::Tensor *lens, *n;
    c10::Device dev(c10::kCPU);
    int32_t k;
    cs_stream_t s;
    if (!first(a[0], at::kInt, 1, &dev, &lens) || !need(a[1], at::kInt, 1, dev, &n) || !small_int(a[2], &k) ||
        !stream_of(a[3], dev, &s))
        Py_RETURN_NONE;
    const cs_status st = launch([&] {
        return cs_kv_commit((int32_t)lens->size(0), (int32_t*)lens->data_ptr(), (const int32_t*)n->data_ptr(), k, s);
    });
    if (st != CS_OK) return status(st);
    Py_RETURN_TRUE;
CALL_END

// k_pages, v_pages, page_table, ctx_lens, path, n_accepted, stream.  True when done.
CALL(kv_commit_tree, 7)
    const at::Tensor *k, *v, *table, *lens, *path, *n;
    c10::Device dev(c10::kCPU);
    cs_stream_t s;
    if (!first(a[0], at::kBFloat16, 4, &dev, &k) || !need(a[1], at::kBFloat16, 4, dev, &v) ||
        !need(a[2], at::kInt, 2, dev, &table) || !need(a[3], at::kInt, 1, dev, &lens) ||
        !need(a[4], at::kInt, 2, dev, &path) || !need(a[5], at::kInt, 1, dev, &n) || !stream_of(a[6], dev, &s) ||
        k->sizes() != v->sizes())
        Py_RETURN_NONE;
    const int32_t hkv = (int32_t)k->size(1);
    const cs_attn_dims d{(int32_t)path->size(0), hkv, hkv, (int32_t)k->size(3), (int32_t)k->size(2),
                         (int32_t)table->size(1), (int32_t)k->size(0), 0.f};
    const cs_status st = launch([&] {
        return cs_kv_commit_tree(&d, k->data_ptr(), v->data_ptr(), (const int32_t*)table->data_ptr(),
                                 (int32_t*)lens->data_ptr(), (const int32_t*)path->data_ptr(),
                                 (const int32_t*)n->data_ptr(), (int32_t)path->size(1), s);
    });
    if (st != CS_OK) return status(st);
    Py_RETURN_TRUE;
CALL_END

PyObject* use_workspaces(PyObject*, PyObject* f) {
    Py_XSETREF(g_workspace_of, Py_NewRef(f));
    Py_RETURN_NONE;
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(name)), METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {FAST(verify_attention), FAST(tree_verify_attention), FAST(spec_accept), FAST(tree_accept),
                           FAST(sample), FAST(route), FAST(kv_append), FAST(kv_commit), FAST(kv_commit_tree),
                           {"use_workspaces", use_workspaces, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&g_module); }
