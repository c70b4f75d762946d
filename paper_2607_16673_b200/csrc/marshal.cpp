// Argument marshalling of the Python binding in native code: checks and unpacks torch tensors and calls the C ABI.
//
// One call through ctypes costs 12-17 us of host time, most of it in checking and converting up to 27 arguments one by
// one in Python; a speculative round is three calls, and for a single user its kernels take less than that.  Here a call
// costs about a microsecond on top of its kernel launches.
//
// Every function returns the C entry point's code, or None if an argument is not plainly what the entry point wants (a
// wrong dtype, shape, device or layout, or a number that is no integer): the binding then runs its own checks, which
// name the argument, or converts it.  So does whatever torch throws on the way (a tensor without strides or without
// storage, no device to take a stream of): see guarded().  Nothing is kept between calls but the addresses of the entry points.
#include <Python.h>
#include <torch/csrc/autograd/python_variable.h>
#include <c10/cuda/CUDAStream.h>

#include <initializer_list>

#include "../../include/speca.h"

namespace {

using at::ScalarType;

struct Api {
    decltype(&speca_decode_step) decode_step;
    decltype(&speca_verify_chain) verify_chain;
    decltype(&speca_verify_tree) verify_tree;
    decltype(&speca_verify_tree_noalloc) verify_tree_noalloc;
    decltype(&speca_greedy_accept) greedy_accept;
    decltype(&speca_stochastic_accept) stochastic_accept;
    decltype(&speca_commit) commit;
    decltype(&speca_commit_verify_tree) commit_verify_tree;
    decltype(&speca_commit_conv) commit_conv;
    decltype(&speca_tree_mask_to_parent) tree_mask_to_parent;
    decltype(&speca_prune_tree) prune_tree;
    decltype(&speca_chain_decompose) chain_decompose;
} g_api = {};

enum Name { kLayers, kBatch, kHeads, kDk, kDv, kScale, kMaxDepth, kMaxNodes, kRoute, kRule, kK, kV, kAlpha, kBeta, kU, kOffsets, kTotal, kParent, kNames };
PyObject *g_name[kNames];
const char *const kNameText[kNames] = {"n_layers", "batch", "heads", "d_k", "d_v", "scale", "max_depth", "max_nodes", "route", "rule",
                                       "k", "v", "alpha", "beta", "u", "node_offsets", "total_nodes", "parent"};

// Reads the arguments of one call; `ok` turns false at the first that is not plainly right.
struct Reader {
    bool ok;

    Reader(Py_ssize_t n, Py_ssize_t want) : ok(n == want) {}

    int integer(PyObject *o)
    {
        if (!ok || o == nullptr) { ok = false; return 0; }
        // (numpy's integers among them; a tensor's value would have to be fetched, which int() does in the binding)
        PyObject *i = PyLong_Check(o) ? Py_NewRef(o) : PyIndex_Check(o) && !THPVariable_Check(o) ? PyNumber_Index(o) : nullptr;
        const long v = i != nullptr ? PyLong_AsLong(i) : -1;
        Py_XDECREF(i);
        if (i == nullptr || (v == -1 && PyErr_Occurred()) || v != long(int(v))) { PyErr_Clear(); ok = false; }
        return int(v);
    }
    int attr(PyObject *o, Name n)
    {
        PyObject *x = PyObject_GetAttr(o, g_name[n]);
        const int v = integer(x);
        if (x == nullptr) PyErr_Clear();
        Py_XDECREF(x);
        return v;
    }
    speca_dims dims(PyObject *o)
    {
        speca_dims d;
        d.n_layers = attr(o, kLayers); d.batch = attr(o, kBatch); d.heads = attr(o, kHeads);
        d.d_k = attr(o, kDk); d.d_v = attr(o, kDv);
        d.max_depth = attr(o, kMaxDepth); d.max_nodes = attr(o, kMaxNodes); d.route = attr(o, kRoute); d.rule = attr(o, kRule);
        PyObject *s = PyObject_GetAttr(o, g_name[kScale]);
        d.scale = s != nullptr ? float(PyFloat_AsDouble(s)) : 0.f;
        Py_XDECREF(s);
        if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
        return d;
    }
    const at::Tensor *tensor(PyObject *o, ScalarType type)
    {
        if (!ok || o == nullptr || !THPVariable_Check(o)) { ok = false; return nullptr; }
        const at::Tensor &t = THPVariable_Unpack(o);
        if (!t.is_cuda() || t.scalar_type() != type || !t.is_contiguous()) { ok = false; return nullptr; }
        return &t;
    }
    // device pointer of a tensor of this type and shape; None is a null pointer
    void *ptr(PyObject *o, ScalarType type, std::initializer_list<int64_t> shape)
    {
        if (o == Py_None) return nullptr;
        const at::Tensor *t = tensor(o, type);
        if (t == nullptr || !(t->sizes() == at::IntArrayRef(shape))) { ok = false; return nullptr; }
        return t->data_ptr();
    }
    float *f32(PyObject *o, std::initializer_list<int64_t> s) { return static_cast<float *>(ptr(o, ScalarType::Float, s)); }
    int32_t *i32(PyObject *o, std::initializer_list<int64_t> s) { return static_cast<int32_t *>(ptr(o, ScalarType::Int, s)); }
    uint16_t *bf16(PyObject *o, std::initializer_list<int64_t> s) { return static_cast<uint16_t *>(ptr(o, ScalarType::BFloat16, s)); }
    // bytes of any shape
    struct Bytes { void *ptr; size_t size; };
    Bytes bytes(PyObject *o)
    {
        const at::Tensor *t = tensor(o, ScalarType::Byte);
        return t != nullptr ? Bytes{t->data_ptr(), size_t(t->numel())} : Bytes{nullptr, 0};
    }
    // a tensor whose shape the others are checked against
    const at::Tensor *any(PyObject *o, ScalarType type, int64_t ndim)
    {
        const at::Tensor *t = tensor(o, type);
        if (t != nullptr && t->dim() != ndim) { ok = false; return nullptr; }
        return t;
    }
};

// `f` runs without the interpreter lock and must not throw: addresses are taken before.
template <class F> PyObject *call(const Reader &r, F f)
{
    if (!r.ok) Py_RETURN_NONE;
    int rc = 0;
    void *st = c10::cuda::getCurrentCUDAStream().stream();
    Py_BEGIN_ALLOW_THREADS
    rc = f(st);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
}

// q, k, v, alpha, beta, node_offsets, total_nodes and the state: what every verification starts with
struct Draft {
    float *S;
    uint16_t *q, *k, *v;
    float *alpha, *beta;
    int32_t *offs;
    int T;
    Draft(Reader &r, const speca_dims &d, PyObject *s, PyObject *const *a)
    {
        const int64_t L = d.n_layers, B = d.batch, H = d.heads, dk = d.d_k, dv = d.d_v;
        T = r.integer(a[6]);
        S = r.f32(s, {L, B, H, dv, dk});
        q = r.bf16(a[0], {L, T, H, dk});
        k = r.bf16(a[1], {L, T, H, dk});
        v = r.bf16(a[2], {L, T, H, dv});
        alpha = r.f32(a[3], {L, T, H});
        beta = r.f32(a[4], {L, T, H});
        offs = r.i32(a[5], {B + 1});
    }
};

PyObject *decode_step(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 8);
    if (!r.ok) Py_RETURN_NONE;
    const speca_dims d = r.dims(a[0]);
    const int64_t L = d.n_layers, B = d.batch, H = d.heads, dk = d.d_k, dv = d.d_v;
    float *S = r.f32(a[1], {L, B, H, dv, dk});
    uint16_t *q = r.bf16(a[2], {L, B, H, dk}), *k = r.bf16(a[3], {L, B, H, dk}), *v = r.bf16(a[4], {L, B, H, dv});
    float *alpha = r.f32(a[5], {L, B, H}), *beta = r.f32(a[6], {L, B, H}), *o = r.f32(a[7], {L, B, H, dv});
    return call(r, [&](void *st) { return g_api.decode_step(&d, S, q, k, v, alpha, beta, o, st); });
}

PyObject *verify_chain(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 13);
    if (!r.ok) Py_RETURN_NONE;
    const speca_dims d = r.dims(a[0]);
    const Draft x(r, d, a[1], a + 2);
    float *o = r.f32(a[9], {d.n_layers, x.T, d.heads, d.d_v}), *u = r.f32(a[10], {d.n_layers, x.T, d.heads, d.d_v});
    const Reader::Bytes ws = r.bytes(a[11]);
    int32_t *status = r.i32(a[12], {1});
    return call(r, [&](void *st) {
        return g_api.verify_chain(&d, x.S, x.q, x.k, x.v, x.alpha, x.beta, x.offs, x.T, o, u, ws.ptr, ws.size, status, st);
    });
}

PyObject *verify_tree(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 15);
    if (!r.ok) Py_RETURN_NONE;
    const speca_dims d = r.dims(a[0]);
    const Draft x(r, d, a[1], a + 2);
    int32_t *parent = r.i32(a[9], {x.T}), *depth = r.i32(a[10], {x.T});
    float *o = r.f32(a[11], {d.n_layers, x.T, d.heads, d.d_v}), *u = r.f32(a[12], {d.n_layers, x.T, d.heads, d.d_v});
    const Reader::Bytes ws = r.bytes(a[13]);
    int32_t *status = r.i32(a[14], {1});
    return call(r, [&](void *st) {
        return g_api.verify_tree(&d, x.S, x.q, x.k, x.v, x.alpha, x.beta, x.offs, x.T, parent, depth, o, u, ws.ptr,
                                 ws.size, status, st);
    });
}

PyObject *verify_tree_noalloc(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 14);
    if (!r.ok) Py_RETURN_NONE;
    const speca_dims d = r.dims(a[0]);
    const Draft x(r, d, a[1], a + 2);
    int32_t *parent = r.i32(a[9], {x.T}), *depth = r.i32(a[10], {x.T});
    float *o = r.f32(a[11], {d.n_layers, x.T, d.heads, d.d_v}), *u = r.f32(a[12], {d.n_layers, x.T, d.heads, d.d_v});
    int32_t *status = r.i32(a[13], {1});
    return call(r, [&](void *st) {
        return g_api.verify_tree_noalloc(&d, x.S, x.q, x.k, x.v, x.alpha, x.beta, x.offs, x.T, parent, depth, o, u, status, st);
    });
}

PyObject *greedy_accept(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 11);
    if (!r.ok) Py_RETURN_NONE;
    const int B = r.integer(a[0]), D = r.integer(a[1]);
    const at::Tensor *par_t = r.any(a[3], ScalarType::Int, 1);
    if (!r.ok) Py_RETURN_NONE;
    const int64_t T = par_t->numel();
    const int32_t *par = par_t->const_data_ptr<int32_t>();
    int32_t *offs = r.i32(a[2], {B + 1}), *draft = r.i32(a[4], {T}), *target = r.i32(a[5], {T}), *root = r.i32(a[6], {B}),
            *idx = r.i32(a[7], {B, D}), *len = r.i32(a[8], {B}), *next = r.i32(a[9], {B}), *status = r.i32(a[10], {1});
    return call(r, [&](void *st) {
        return g_api.greedy_accept(B, D, offs, par, draft, target, root, idx, len, next, status, st);
    });
}

PyObject *stochastic_accept(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 10);
    if (!r.ok) Py_RETURN_NONE;
    const int B = r.integer(a[0]), D = r.integer(a[1]);
    const at::Tensor *par_t = r.any(a[3], ScalarType::Int, 1);
    if (!r.ok) Py_RETURN_NONE;
    const int64_t T = par_t->numel();
    const int32_t *par = par_t->const_data_ptr<int32_t>();
    int32_t *offs = r.i32(a[2], {B + 1});
    float *pt = r.f32(a[4], {T}), *pd = r.f32(a[5], {T}), *un = r.f32(a[6], {T});
    int32_t *idx = r.i32(a[7], {B, D}), *len = r.i32(a[8], {B}), *status = r.i32(a[9], {1});
    return call(r, [&](void *st) {
        return g_api.stochastic_accept(B, D, offs, par, pt, pd, un, idx, len, status, st);
    });
}

PyObject *commit(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 12);
    if (!r.ok) Py_RETURN_NONE;
    const speca_dims d = r.dims(a[0]);
    const int64_t L = d.n_layers, B = d.batch, H = d.heads, dk = d.d_k, dv = d.d_v;
    const int T = r.integer(a[7]);
    float *S = r.f32(a[1], {L, B, H, dv, dk});
    uint16_t *k = r.bf16(a[2], {L, T, H, dk}), *v = r.bf16(a[3], {L, T, H, dv});
    float *alpha = r.f32(a[4], {L, T, H}), *beta = r.f32(a[5], {L, T, H});
    int32_t *offs = r.i32(a[6], {B + 1}), *parent = r.i32(a[8], {T}), *idx = r.i32(a[9], {B, d.max_depth}), *len = r.i32(a[10], {B}),
            *status = r.i32(a[11], {1});
    return call(r, [&](void *st) { return g_api.commit(&d, S, k, v, alpha, beta, offs, T, parent, idx, len, status, st); });
}

PyObject *commit_verify_tree(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 18);
    if (!r.ok) Py_RETURN_NONE;
    const speca_dims d = r.dims(a[0]);
    const int64_t L = d.n_layers, B = d.batch, H = d.heads, dk = d.d_k, dv = d.d_v;
    // the previous draft: a dict that holds its tensors for the duration of the call
    uint16_t *pk = nullptr, *pv = nullptr;
    float *pa = nullptr, *pb = nullptr, *pu = nullptr;
    int32_t *po = nullptr, *pp = nullptr;
    int Tp = 0;
    if (a[2] != Py_None) {
        if (!PyDict_CheckExact(a[2])) Py_RETURN_NONE;
        auto item = [&](Name w, bool optional) -> PyObject * {
            PyObject *x = PyDict_GetItemWithError(a[2], g_name[w]);          // borrowed
            if (x == nullptr) {
                PyErr_Clear();
                if (!optional) r.ok = false;
                return Py_None;
            }
            return x;
        };
        Tp = r.integer(item(kTotal, false));
        pk = r.bf16(item(kK, false), {L, Tp, H, dk});
        pv = r.bf16(item(kV, false), {L, Tp, H, dv});
        pa = r.f32(item(kAlpha, false), {L, Tp, H});
        pb = r.f32(item(kBeta, false), {L, Tp, H});
        pu = r.f32(item(kU, true), {L, Tp, H, dv});
        po = r.i32(item(kOffsets, false), {B + 1});
        pp = r.i32(item(kParent, true), {Tp});
    }
    int32_t *idx = r.i32(a[3], {B, d.max_depth}), *len = r.i32(a[4], {B});
    const Draft x(r, d, a[1], a + 5);
    int32_t *parent = r.i32(a[12], {x.T}), *depth = r.i32(a[13], {x.T});
    float *o = r.f32(a[14], {L, x.T, H, dv}), *u = r.f32(a[15], {L, x.T, H, dv});
    const Reader::Bytes ws = r.bytes(a[16]);
    int32_t *status = r.i32(a[17], {1});
    return call(r, [&](void *st) {
        return g_api.commit_verify_tree(&d, x.S, pk, pv, pa, pb, pu, po, Tp, pp, idx, len, x.q, x.k, x.v, x.alpha, x.beta, x.offs, x.T,
                                        parent, depth, o, u, ws.ptr, ws.size, status, st);
    });
}

PyObject *commit_conv(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 7);
    if (!r.ok) Py_RETURN_NONE;
    const at::Tensor *C = r.any(a[0], ScalarType::BFloat16, 4), *idx = r.any(a[4], ScalarType::Int, 2);
    if (!r.ok) Py_RETURN_NONE;
    const int64_t L = C->size(0), B = C->size(1), W = C->size(2), ch = C->size(3), D = idx->size(1);
    const int T = r.integer(a[3]);
    if (idx->size(0) != B || L > INT32_MAX || B > INT32_MAX || W > INT32_MAX || ch > INT32_MAX || D > INT32_MAX) Py_RETURN_NONE;
    uint16_t *x = r.bf16(a[1], {L, T, ch});
    int32_t *offs = r.i32(a[2], {B + 1}), *len = r.i32(a[5], {B}), *status = r.i32(a[6], {1});
    uint16_t *c_ptr = static_cast<uint16_t *>(C->data_ptr());
    const int32_t *idx_ptr = idx->const_data_ptr<int32_t>();
    return call(r, [&](void *st) {
        return g_api.commit_conv(int(L), int(B), int(ch), int(W), int(D), c_ptr, x, offs, T,
                                 idx_ptr, len, status, st);
    });
}

PyObject *tree_mask_to_parent(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 4);
    if (!r.ok) Py_RETURN_NONE;
    const at::Tensor *mask = r.any(a[0], ScalarType::Byte, 3), *par = r.any(a[2], ScalarType::Int, 1);
    if (!r.ok || mask->size(1) != mask->size(2) || mask->size(0) > INT32_MAX || mask->size(1) > INT32_MAX) Py_RETURN_NONE;
    const int64_t B = mask->size(0), N = mask->size(1);
    int32_t *offs = r.i32(a[1], {B + 1}), *status = r.i32(a[3], {1});
    const uint8_t *mask_ptr = mask->const_data_ptr<uint8_t>();
    int32_t *par_ptr = static_cast<int32_t *>(par->data_ptr());
    return call(r, [&](void *st) {
        return g_api.tree_mask_to_parent(int(B), int(N), mask_ptr, offs, par_ptr, status, st);
    });
}

PyObject *prune_tree(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 10);
    if (!r.ok || !(PyFloat_Check(a[1]) || PyLong_Check(a[1]))) Py_RETURN_NONE;
    const int N = r.integer(a[0]), budget = r.integer(a[2]);
    const float tau = float(PyFloat_AsDouble(a[1]));
    if (PyErr_Occurred()) { PyErr_Clear(); Py_RETURN_NONE; }     // an integer beyond every double
    const at::Tensor *offs_t = r.any(a[3], ScalarType::Int, 1), *par_t = r.any(a[4], ScalarType::Int, 1);
    if (!r.ok || offs_t->numel() < 1 || offs_t->numel() > INT32_MAX) Py_RETURN_NONE;
    const int64_t B = offs_t->numel() - 1, T = par_t->numel();
    const int32_t *offs = offs_t->const_data_ptr<int32_t>(), *par = par_t->const_data_ptr<int32_t>();
    float *logp = r.f32(a[5], {T});
    int32_t *oo = r.i32(a[6], {B + 1}), *op = r.i32(a[7], {T}), *oi = r.i32(a[8], {T}), *status = r.i32(a[9], {1});
    return call(r, [&](void *st) {
        return g_api.prune_tree(int(B), N, tau, budget, offs, par, logp, oo, op, oi, status, st);
    });
}

PyObject *chain_decompose(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    Reader r(n, 6);
    if (!r.ok) Py_RETURN_NONE;
    const int N = r.integer(a[0]);
    const at::Tensor *offs_t = r.any(a[1], ScalarType::Int, 1), *par_t = r.any(a[2], ScalarType::Int, 1);
    if (!r.ok || offs_t->numel() < 1 || offs_t->numel() > INT32_MAX) Py_RETURN_NONE;
    const int64_t B = offs_t->numel() - 1, T = par_t->numel();
    const int32_t *offs = offs_t->const_data_ptr<int32_t>(), *par = par_t->const_data_ptr<int32_t>();
    int32_t *head = r.i32(a[3], {T}), *count = r.i32(a[4], {B}), *status = r.i32(a[5], {1});
    return call(r, [&](void *st) {
        return g_api.chain_decompose(int(B), N, offs, par, head, count, status, st);
    });
}

// bind({entry point name without "speca_": address})
PyObject *bind(PyObject *, PyObject *table)
{
    bool ok = PyDict_Check(table);
    auto get = [&](const char *name, auto &f) {
        PyObject *x = ok ? PyDict_GetItemString(table, name) : nullptr;
        void *p = x != nullptr ? PyLong_AsVoidPtr(x) : nullptr;
        if (p == nullptr) ok = false;
        f = reinterpret_cast<std::remove_reference_t<decltype(f)>>(p);
    };
    get("decode_step", g_api.decode_step);
    get("verify_chain", g_api.verify_chain);
    get("verify_tree", g_api.verify_tree);
    get("verify_tree_noalloc", g_api.verify_tree_noalloc);
    get("greedy_accept", g_api.greedy_accept);
    get("stochastic_accept", g_api.stochastic_accept);
    get("commit", g_api.commit);
    get("commit_verify_tree", g_api.commit_verify_tree);
    get("commit_conv", g_api.commit_conv);
    get("tree_mask_to_parent", g_api.tree_mask_to_parent);
    get("prune_tree", g_api.prune_tree);
    get("chain_decompose", g_api.chain_decompose);
    if (!ok) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: an entry point is missing");
        return nullptr;
    }
    Py_RETURN_NONE;
}

// An exception must not leave a C function: to the interpreter it would be std::terminate.
template <PyObject *(*F)(PyObject *, PyObject *const *, Py_ssize_t)>
PyObject *guarded(PyObject *self, PyObject *const *a, Py_ssize_t n)
{
    try {
        return F(self, a, n);
    } catch (...) {
        PyErr_Clear();
        Py_RETURN_NONE;
    }
}
#define FAST(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void *>(&guarded<f>)), METH_FASTCALL, nullptr}
PyMethodDef kMethods[] = {
    FAST(decode_step), FAST(verify_chain), FAST(verify_tree), FAST(verify_tree_noalloc), FAST(greedy_accept),
    FAST(stochastic_accept), FAST(commit), FAST(commit_verify_tree), FAST(commit_conv), FAST(tree_mask_to_parent),
    FAST(prune_tree), FAST(chain_decompose), {"bind", bind, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "speca_marshal", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_speca_marshal()
{
    for (int i = 0; i < kNames; ++i) {
        g_name[i] = PyUnicode_InternFromString(kNameText[i]);
        if (g_name[i] == nullptr) return nullptr;
    }
    return PyModule_Create(&kModule);
}
