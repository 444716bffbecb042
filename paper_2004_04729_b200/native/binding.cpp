// The host side of the calls that a training step makes once per layer, as a CPython extension: argument checks, output
// allocation and the C ABI call in one native step. A small layer's kernels take a few microseconds, and the same work
// through ctypes and `torch.empty` took more than they do (fp32 784 -> 300, batch 128: 15 us of host time per call, two
// kernel launches of it 6.5 us).
//
// Every function returns its result, or an int (the library's negative status), or None where the arguments are not what
// the fast path takes; the Python function of the same name in binding.py then runs its own checks, which name what is
// wrong. No arithmetic of the method happens here.
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>

#include "dbp.h"

namespace {

PyObject *key_dW, *key_dX, *key_db, *key_Delta, *key_nnz;

const at::Tensor *tensor_of(PyObject *o) { return THPVariable_Check(o) ? &THPVariable_Unpack(o) : nullptr; }
bool on_device(const at::Tensor &t) { return t.is_cuda() && t.is_contiguous(); }
bool dtype_of(const at::Tensor &t, int &io) {
    if (t.scalar_type() == at::kFloat) io = DBP_F32;
    else if (t.scalar_type() == at::kBFloat16) io = DBP_BF16;
    else return false;
    return true;
}
at::Tensor empty_on(const at::Tensor &like, at::IntArrayRef shape, at::ScalarType type) {
    return at::detail::empty_cuda(shape, type, like.device(), std::nullopt);
}
void *ptr(const at::Tensor &t) { return t.defined() ? t.data_ptr() : nullptr; }
// steals nothing; None for an undefined tensor
bool put(PyObject *dict, PyObject *key, const at::Tensor &t) {
    PyObject *v = t.defined() ? THPVariable_Wrap(t) : Py_NewRef(Py_None);
    if (!v) return false;
    const int rc = PyDict_SetItem(dict, key, v);
    Py_DECREF(v);
    return rc == 0;
}
PyObject *result(const at::Tensor &dW, const at::Tensor &dX, const at::Tensor &db) {
    PyObject *d = PyDict_New();
    if (d && put(d, key_dW, dW) && put(d, key_dX, dX) && put(d, key_db, db)) return d;
    Py_XDECREF(d);
    return nullptr;
}
PyObject *none() { return Py_NewRef(Py_None); }
// A mask that was set for a call is not left behind on the context when the call does not happen (an output that could not be
// allocated, shapes that do not belong together).
struct MaskUse {
    dbp_ctx *ctx;
    ~MaskUse() { dbp_set_relu_mask(ctx, nullptr); }
};
// Owns a reference until it is released.
struct Owned {
    PyObject *o;
    explicit Owned(PyObject *object) : o(object) {}
    Owned(const Owned &) = delete;
    ~Owned() { Py_XDECREF(o); }
    PyObject *release() {
        PyObject *r = o;
        o = nullptr;
        return r;
    }
};
// Other Python threads run while a call allocates and enqueues (either may block: a full launch queue, a growing pool).
struct NoGil {
    PyThreadState *state = PyEval_SaveThread();
    ~NoGil() { PyEval_RestoreThread(state); }
};

struct Call {
    dbp_ctx *ctx;
    unsigned long long seed;
    float scale;
    const float *delta_in = nullptr;
    dbp_sparse *q = nullptr;
    bool need_dW, need_dX, need_db;
    unsigned flags;
};

int linear(const Call &c, const at::Tensor &delta, const at::Tensor &X, const at::Tensor &W, int io, at::Tensor &dW,
           at::Tensor &dX, at::Tensor &db) {
    NoGil nogil;
    const int64_t B = delta.size(0), N = delta.size(1), K = X.size(1);
    if (c.need_dW) dW = empty_on(delta, {N, K}, at::kFloat);
    if (c.need_dX) dX = empty_on(delta, {B, K}, (c.flags & DBP_DX_F32) ? at::kFloat : delta.scalar_type());
    if (c.need_db) db = empty_on(delta, {N}, at::kFloat);
    return dithered_linear_backward(c.ctx, delta.data_ptr(), X.data_ptr(), W.data_ptr(), io, B, N, K, c.seed, c.scale, c.delta_in,
                                    c.q, static_cast<float *>(ptr(dW)), ptr(dX), static_cast<float *>(ptr(db)), c.flags);
}

// g, argmax: not null where delta is to be routed from a pooled gradient (fp32)
int conv(const Call &c, const at::Tensor &delta, const at::Tensor &X, const at::Tensor &W, int io, int stride, int pad, at::Tensor &dW,
         at::Tensor &dX, at::Tensor &db, const at::Tensor *g = nullptr, const at::Tensor *argmax = nullptr) {
    NoGil nogil;
    const int64_t B = delta.size(0), Co = delta.size(1), Ci = X.size(1), H = X.size(2), Wd = X.size(3), k = W.size(2);
    if (c.need_dW) dW = empty_on(delta, {Co, Ci, k, k}, at::kFloat);
    if (c.need_dX) dX = empty_on(delta, {B, Ci, H, Wd}, (c.flags & DBP_DX_F32) ? at::kFloat : delta.scalar_type());
    if (c.need_db) db = empty_on(delta, {Co}, at::kFloat);
    if (g)
        return dithered_conv_backward_pooled(c.ctx, static_cast<const float *>(g->data_ptr()), static_cast<const int8_t *>(argmax->data_ptr()),
                                             static_cast<float *>(delta.data_ptr()), X.data_ptr(), W.data_ptr(), B, Ci, Co, H, Wd, static_cast<int>(k),
                                             pad, c.seed, c.scale, c.delta_in, c.q, static_cast<float *>(ptr(dW)), ptr(dX), static_cast<float *>(ptr(db)), c.flags);
    return dithered_conv_backward(c.ctx, delta.data_ptr(), X.data_ptr(), W.data_ptr(), io, B, Ci, Co, H, Wd, static_cast<int>(k),
                                  stride, pad, c.seed, c.scale, c.delta_in, c.q, static_cast<float *>(ptr(dW)), ptr(dX),
                                  static_cast<float *>(ptr(db)), c.flags);
}

bool linear_shapes(const at::Tensor &d, const at::Tensor &X, const at::Tensor &W) {
    return d.dim() == 2 && X.dim() == 2 && W.dim() == 2 && X.size(0) == d.size(0) && W.size(0) == d.size(1) && W.size(1) == X.size(1);
}
bool conv_shapes(const at::Tensor &d, const at::Tensor &X, const at::Tensor &W, int64_t stride) {
    return d.dim() == 4 && X.dim() == 4 && W.dim() == 4 && (stride == 1 || stride == 2) && X.size(0) == d.size(0) &&
           W.size(0) == d.size(1) && W.size(1) == X.size(1) && W.size(2) == W.size(3) && X.size(2) % stride == 0 &&
           X.size(3) % stride == 0 && d.size(2) == X.size(2) / stride && d.size(3) == X.size(3) / stride;
}
bool same_kind(const at::Tensor &d, const at::Tensor &X, const at::Tensor &W, int &io) {
    return on_device(d) && on_device(X) && on_device(W) && X.scalar_type() == d.scalar_type() && W.scalar_type() == d.scalar_type() &&
           dtype_of(d, io);
}

// (ctx, delta, X, W, seed, scale, delta_in, sparse address, need_dW, need_dX, need_db, flags[, stride, pad])
PyObject *layer_backward(PyObject *const *a, Py_ssize_t n, bool is_conv) {
    if (n != (is_conv ? 14 : 12)) return none();
    const at::Tensor *d = tensor_of(a[1]), *X = tensor_of(a[2]), *W = tensor_of(a[3]);
    if (!d || !X || !W || a[0] == Py_None) return none();
    Call c;
    c.ctx = static_cast<dbp_ctx *>(PyLong_AsVoidPtr(a[0]));
    c.seed = PyLong_AsUnsignedLongLongMask(a[4]);
    c.scale = static_cast<float>(PyFloat_AsDouble(a[5]));
    if (a[6] != Py_None) {
        const at::Tensor *t = tensor_of(a[6]);
        if (!t) return none();
        c.delta_in = static_cast<const float *>(t->data_ptr());
    }
    if (a[7] != Py_None) c.q = static_cast<dbp_sparse *>(PyLong_AsVoidPtr(a[7]));
    c.need_dW = PyObject_IsTrue(a[8]); c.need_dX = PyObject_IsTrue(a[9]); c.need_db = PyObject_IsTrue(a[10]);
    c.flags = static_cast<unsigned>(PyLong_AsUnsignedLongMask(a[11]));
    const long stride = is_conv ? PyLong_AsLong(a[12]) : 1, pad = is_conv ? PyLong_AsLong(a[13]) : 0;
    if (PyErr_Occurred()) { PyErr_Clear(); return none(); }
    int io;
    if (!same_kind(*d, *X, *W, io) || !(is_conv ? conv_shapes(*d, *X, *W, stride) : linear_shapes(*d, *X, *W))) return none();
    const MaskUse mask_use{c.ctx};
    at::Tensor dW, dX, db;
    const int rc = is_conv ? conv(c, *d, *X, *W, io, static_cast<int>(stride), static_cast<int>(pad), dW, dX, db)
                           : linear(c, *d, *X, *W, io, dW, dX, db);
    return rc ? PyLong_FromLong(rc) : result(dW, dX, db);
}

PyObject *linear_backward(PyObject *, PyObject *const *a, Py_ssize_t n) {
    try { return layer_backward(a, n, false); } catch (const std::exception &e) { PyErr_SetString(PyExc_RuntimeError, e.what()); return nullptr; }
}
PyObject *conv_backward(PyObject *, PyObject *const *a, Py_ssize_t n) {
    try { return layer_backward(a, n, true); } catch (const std::exception &e) { PyErr_SetString(PyExc_RuntimeError, e.what()); return nullptr; }
}

// (ctx, delta, seed, scale, delta_in, sparse address) -> 0
PyObject *quantize(PyObject *, PyObject *const *a, Py_ssize_t n) {
    const at::Tensor *d = n == 6 && a[0] != Py_None ? tensor_of(a[1]) : nullptr;
    int io;
    if (!d || !on_device(*d) || !dtype_of(*d, io)) return none();
    const float *delta_in = nullptr;
    if (a[4] != Py_None) {
        const at::Tensor *t = tensor_of(a[4]);
        if (!t) return none();
        delta_in = static_cast<const float *>(t->data_ptr());
    }
    dbp_ctx *ctx = static_cast<dbp_ctx *>(PyLong_AsVoidPtr(a[0]));
    const unsigned long long seed = PyLong_AsUnsignedLongLongMask(a[2]);
    const float scale = static_cast<float>(PyFloat_AsDouble(a[3]));
    dbp_sparse *q = static_cast<dbp_sparse *>(PyLong_AsVoidPtr(a[5]));
    if (PyErr_Occurred()) { PyErr_Clear(); return none(); }
    int rc;
    {
        NoGil nogil;
        rc = nsd_quantize(ctx, d->data_ptr(), io, d->numel(), seed, scale, delta_in, q);
    }
    return PyLong_FromLong(rc);
}

// (ctx, sparse address, numel, a tensor of the device) -> codes
PyObject *decode(PyObject *, PyObject *const *a, Py_ssize_t n) {
    try {
        const at::Tensor *like = n == 4 && a[0] != Py_None ? tensor_of(a[3]) : nullptr;
        if (!like || !like->is_cuda()) return none();
        dbp_ctx *ctx = static_cast<dbp_ctx *>(PyLong_AsVoidPtr(a[0]));
        const dbp_sparse *q = static_cast<const dbp_sparse *>(PyLong_AsVoidPtr(a[1]));
        const long long numel = PyLong_AsLongLong(a[2]);
        if (PyErr_Occurred() || numel <= 0) { PyErr_Clear(); return none(); }
        at::Tensor codes;
        int rc;
        {
            NoGil nogil;
            codes = empty_on(*like, {numel}, at::kChar);
            rc = nsd_decode_dense(ctx, q, static_cast<int8_t *>(codes.data_ptr()));
        }
        return rc ? PyLong_FromLong(rc) : THPVariable_Wrap(codes);
    } catch (const std::exception &e) { PyErr_SetString(PyExc_RuntimeError, e.what()); return nullptr; }
}

int maxpool(dbp_ctx *ctx, const at::Tensor &g, const at::Tensor &am, at::Tensor &out) {
    NoGil nogil;
    const int64_t B = g.size(0), C = g.size(1), h = g.size(2), w = g.size(3);
    out = empty_on(g, {B, C, 2 * h, 2 * w}, g.scalar_type());
    return dbp_maxpool2x2_backward(ctx, static_cast<const float *>(g.data_ptr()), static_cast<const int8_t *>(am.data_ptr()),
                                   static_cast<float *>(out.data_ptr()), B * C, h, w);
}

// (ctx, g, argmax) -> routed gradient
PyObject *maxpool2x2(PyObject *, PyObject *const *a, Py_ssize_t n) {
    try {
        const at::Tensor *g = n == 3 && a[0] != Py_None ? tensor_of(a[1]) : nullptr, *am = n == 3 ? tensor_of(a[2]) : nullptr;
        if (!g || !am || g->dim() != 4 || !on_device(*g) || !on_device(*am) || g->scalar_type() != at::kFloat) return none();
        at::Tensor out;
        const int rc = maxpool(static_cast<dbp_ctx *>(PyLong_AsVoidPtr(a[0])), *g, *am, out);
        return rc ? PyLong_FromLong(rc) : THPVariable_Wrap(out);
    } catch (const std::exception &e) { PyErr_SetString(PyExc_RuntimeError, e.what()); return nullptr; }
}

// (ctx, mask) -> status
PyObject *set_relu_mask(PyObject *, PyObject *const *a, Py_ssize_t n) {
    const at::Tensor *m = n == 2 && a[0] != Py_None ? tensor_of(a[1]) : nullptr;
    if (!m || !on_device(*m) || m->scalar_type() != at::kByte) return none();
    return PyLong_FromLong(dbp_set_relu_mask(static_cast<dbp_ctx *>(PyLong_AsVoidPtr(a[0])), static_cast<const uint8_t *>(m->data_ptr())));
}

// (ctx, kinds, Xs, Ws, masks, pools, delta_out, scale, seed, first_layer_dX, flags) -> one dict per layer. fp32 networks
// of which nobody asked for delta_z or the sparse structure: the masks are folded into the calls.
PyObject *network(PyObject *const *a, Py_ssize_t n) {
    if (n != 11 || a[0] == Py_None) return none();
    for (int i = 1; i <= 5; ++i)
        if (!PyList_Check(a[i]) || PyList_GET_SIZE(a[i]) != PyList_GET_SIZE(a[1])) return none();
    const Py_ssize_t L = PyList_GET_SIZE(a[1]);
    const at::Tensor *d0 = tensor_of(a[6]);
    if (!d0 || L == 0) return none();
    Call c;
    c.ctx = static_cast<dbp_ctx *>(PyLong_AsVoidPtr(a[0]));
    c.scale = static_cast<float>(PyFloat_AsDouble(a[7]));
    const unsigned long long seed = PyLong_AsUnsignedLongLongMask(a[8]);
    const bool first_dX = PyObject_IsTrue(a[9]);
    c.flags = static_cast<unsigned>(PyLong_AsUnsignedLongMask(a[10]));
    c.need_dW = true;
    c.need_db = false;
    if (PyErr_Occurred()) { PyErr_Clear(); return none(); }
    // everything is checked before the first kernel is enqueued
    struct Layer { bool conv; const at::Tensor *X, *W, *mask, *pool; };
    std::vector<Layer> layers(L);
    for (Py_ssize_t l = 0; l < L; ++l) {
        Layer &y = layers[l];
        PyObject *kind = PyList_GET_ITEM(a[1], l), *mask = PyList_GET_ITEM(a[4], l), *pool = PyList_GET_ITEM(a[5], l);
        if (!PyUnicode_Check(kind)) return none();
        y.conv = PyUnicode_CompareWithASCIIString(kind, "linear") != 0;
        y.X = tensor_of(PyList_GET_ITEM(a[2], l));
        y.W = tensor_of(PyList_GET_ITEM(a[3], l));
        y.mask = mask == Py_None ? nullptr : tensor_of(mask);
        y.pool = pool == Py_None ? nullptr : tensor_of(pool);
        if ((mask != Py_None && !y.mask) || (pool != Py_None && !y.pool) || !y.X || !y.W) return none();
        if (!on_device(*y.X) || !on_device(*y.W) || y.X->scalar_type() != at::kFloat || y.W->scalar_type() != at::kFloat) return none();
        if (y.X->dim() != (y.conv ? 4 : 2) || y.W->dim() != y.X->dim()) return none();
        if (y.mask && (!on_device(*y.mask) || y.mask->scalar_type() != at::kByte)) return none();
        if (y.pool && (!on_device(*y.pool) || y.pool->dim() != 4)) return none();
        // the layer above reads what this one made
        if (l + 1 < L && (!y.mask || (y.conv && y.mask->dim() != 4))) return none();
    }
    if (!on_device(*d0) || d0->scalar_type() != at::kFloat) return none();
    Owned res(PyList_New(L));
    if (!res.o) return nullptr;
    at::Tensor delta = *d0, pooled;                  // pooled: what delta is to be routed from
    for (Py_ssize_t l = L - 1; l >= 0; --l) {
        const Layer &y = layers[l];
        int rc = 0;
        if (!(y.conv ? conv_shapes(delta, *y.X, *y.W, 1) : linear_shapes(delta, *y.X, *y.W)) ||
            (y.mask && y.mask->numel() != delta.numel())) {
            if (l < L - 1) { PyErr_SetString(PyExc_ValueError, "shapes of the layers do not belong to one network"); return nullptr; }
            return none();
        }
        const MaskUse mask_use{c.ctx};
        if (y.mask) rc = dbp_set_relu_mask(c.ctx, static_cast<const uint8_t *>(y.mask->data_ptr()));
        c.seed = dbp_layer_seed(seed, static_cast<int>(l));
        c.need_dX = l > 0 || first_dX;
        at::Tensor dW, dX, db;
        if (!rc)
            rc = y.conv ? conv(c, delta, *y.X, *y.W, DBP_F32, 1, static_cast<int>((y.W->size(2) - 1) / 2), dW, dX, db,
                             pooled.defined() ? &pooled : nullptr, y.pool)
                        : linear(c, delta, *y.X, *y.W, DBP_F32, dW, dX, db);
        if (rc) return PyLong_FromLong(rc);
        Owned d(result(dW, dX, db));
        if (!d.o || PyDict_SetItem(d.o, key_Delta, Py_None) || PyDict_SetItem(d.o, key_nnz, Py_None)) return nullptr;
        PyList_SET_ITEM(res.o, l, d.release());
        if (l == 0) break;
        const Layer &below = layers[l - 1];
        delta = dX;
        pooled.reset();
        if (!y.conv && below.conv) {
            const at::Tensor &s = below.pool ? *below.pool : *below.mask;
            delta = dX.view({below.mask->size(0), below.mask->size(1), s.size(2), s.size(3)});
        }
        if (below.pool) {
            if (delta.dim() != 4 || below.pool->numel() != delta.numel()) {
                PyErr_SetString(PyExc_ValueError, "shapes of a pool and its gradient differ");
                return nullptr;
            }
            pooled = delta;
            delta = empty_on(pooled, {pooled.size(0), pooled.size(1), 2 * pooled.size(2), 2 * pooled.size(3)}, pooled.scalar_type());
        }
    }
    return res.release();
}
PyObject *network_backward(PyObject *, PyObject *const *a, Py_ssize_t n) {
    try { return network(a, n); } catch (const std::exception &e) { PyErr_SetString(PyExc_RuntimeError, e.what()); return nullptr; }
}

#define FAST(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {FAST(linear_backward), FAST(conv_backward), FAST(quantize), FAST(decode), FAST(maxpool2x2),
                         FAST(set_relu_mask), FAST(network_backward), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native(void) {
    key_dW = PyUnicode_InternFromString("dW");
    key_dX = PyUnicode_InternFromString("dX");
    key_db = PyUnicode_InternFromString("db");
    key_Delta = PyUnicode_InternFromString("Delta");
    key_nnz = PyUnicode_InternFromString("nnz");
    return PyModule_Create(&module);
}
