// Argument marshalling from torch tensors to the C ABI of include/speckv.h, natively.
//
// binding.py describes a call's arguments by plain Python objects (Batch, Mlp, StepOutputs) and checks every tensor before
// its address is passed on.  Done in Python, reading and checking the twenty tensors of a step costs more than the step
// takes on the GPU for a small batch (one row, V = 32,000: 42 us of host work for 20 us on the device); the same checks here
// take under one (6.5 us with the launches).  The functions below check exactly what the Python path checks and then call the library; where
// a check fails, where an object is not what it usually is, or where the tensors live on another than the current device
// they return None without having done anything, and the caller takes the Python path, which raises the error (or does the
// call with the device switched).  The library's functions are passed in as addresses, so that the caller decides which
// build of the library is used.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <initializer_list>

#include "speckv.h"

namespace {

struct Ref {  // an owned reference
    PyObject* p;
    explicit Ref(PyObject* q = nullptr) : p(q) {}
    Ref(Ref&& o) noexcept : p(o.p) { o.p = nullptr; }
    Ref(const Ref&) = delete;
    Ref& operator=(const Ref&) = delete;
    ~Ref() { Py_XDECREF(p); }
};

#define NAMES(X)                                                                                                       \
    X(draft_logits) X(target_logits) X(draft_tokens) X(gamma) X(temperature) X(temperature_scalar) X(uniforms)        \
    X(entropy_in_bits) X(flags) X(W1) X(b1) X(W2) X(b2) X(gamma_choices) X(feature_layout) X(score_transform) X(H)    \
    X(C) X(feat) X(scores) X(gamma_next) X(n_accepted) X(out_tokens) X(row_status) X(workspace)
#define X(n) PyObject* s_##n;
NAMES(X)
#undef X

// Raised inside when the call has to take the Python path.
struct Slow {};

using Shape = std::initializer_list<int64_t>;

// A tensor attribute or argument; the owner keeps it alive for the duration of the call (the GIL is held).
const at::Tensor* tensor_of(PyObject* o) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) throw Slow();
    return &THPVariable_Unpack(o);
}
struct Args {
    c10::Device dev{c10::DeviceType::CPU};
    Ref held[32];
    int n_held = 0;

    PyObject* get(PyObject* obj, PyObject* name) {
        PyObject* v = PyObject_GetAttr(obj, name);
        if (!v) { PyErr_Clear(); throw Slow(); }
        if (n_held == 32) { Py_DECREF(v); throw Slow(); }
        held[n_held++].p = v;
        return v;
    }
    const at::Tensor* tensor(PyObject* obj, PyObject* name) { return tensor_of(get(obj, name)); }
    long integer(PyObject* obj, PyObject* name) {
        PyObject* v = get(obj, name);
        if (!PyLong_Check(v)) throw Slow();
        const long x = PyLong_AsLong(v);
        if (x == -1 && PyErr_Occurred()) { PyErr_Clear(); throw Slow(); }
        return x;
    }
    // the address of a buffer of exactly this type and shape, contiguous, on the logits' device
    void* buf(const at::Tensor* t, at::ScalarType dt, Shape shape) const {
        if (!t) return nullptr;
        if (t->device() != dev || t->scalar_type() != dt || !t->is_contiguous() || t->sizes() != at::IntArrayRef(shape)) throw Slow();
        return t->data_ptr();
    }
    void* need(const at::Tensor* t, at::ScalarType dt, Shape shape) const {
        if (!t) throw Slow();
        return buf(t, dt, shape);
    }
};

constexpr auto F32 = at::ScalarType::Float;
constexpr auto I32 = at::ScalarType::Int;

void read_batch(Args& a, PyObject* batch, speckv_batch& c) {
    const at::Tensor* d = a.tensor(batch, s_draft_logits);
    if (!d || d->dim() != 3 || !d->is_cuda()) throw Slow();
    const auto dt = d->scalar_type();
    if (dt != F32 && dt != at::ScalarType::BFloat16) throw Slow();
    const int64_t B = d->size(0), G = d->size(1), V = d->size(2);
    if (B > INT32_MAX || G > INT32_MAX || V > INT32_MAX || (V > 1 && d->stride(2) != 1)) throw Slow();
    a.dev = d->device();
    if (a.dev.index() != c10::cuda::current_device()) throw Slow();
    c.B = static_cast<int32_t>(B);
    c.gamma_max = static_cast<int32_t>(G);
    c.V = static_cast<int32_t>(V);
    c.dtype = dt == F32 ? SPECKV_F32 : SPECKV_BF16;
    c.draft_logits = d->data_ptr();
    c.draft_stride_b = d->stride(0);
    c.draft_stride_pos = d->stride(1);
    if (const at::Tensor* t = a.tensor(batch, s_target_logits)) {
        if (t->device() != a.dev || t->scalar_type() != dt || t->sizes() != at::IntArrayRef({B, G + 1, V}) || (V > 1 && t->stride(2) != 1))
            throw Slow();
        c.target_logits = t->data_ptr();
        c.target_stride_b = t->stride(0);
        c.target_stride_pos = t->stride(1);
    }
    c.draft_tokens = static_cast<int32_t*>(a.buf(a.tensor(batch, s_draft_tokens), I32, {B, G}));
    c.gamma = static_cast<int32_t*>(a.buf(a.tensor(batch, s_gamma), I32, {B}));
    c.temperature = static_cast<float*>(a.buf(a.tensor(batch, s_temperature), F32, {B}));
    c.uniforms = static_cast<float*>(a.buf(a.tensor(batch, s_uniforms), F32, {B, G + 1, 2}));
    PyObject* ts = a.get(batch, s_temperature_scalar);
    if (!PyFloat_Check(ts)) throw Slow();
    c.temperature_scalar = static_cast<float>(PyFloat_AS_DOUBLE(ts));
    PyObject* bits = a.get(batch, s_entropy_in_bits);
    if (!PyBool_Check(bits)) throw Slow();
    c.entropy_in_bits = bits == Py_True;
    c.flags = static_cast<int32_t>(a.integer(batch, s_flags));
}

// The controller; its parameters on the device of the call.  Returns the number of compression features.
int64_t read_mlp(Args& a, PyObject* mlp, speckv_mlp& m) {
    const at::Tensor *w1 = a.tensor(mlp, s_W1), *b1 = a.tensor(mlp, s_b1), *w2 = a.tensor(mlp, s_W2), *b2 = a.tensor(mlp, s_b2);
    PyObject* ch = a.get(mlp, s_gamma_choices);
    const long layout = a.integer(mlp, s_feature_layout), transform = a.integer(mlp, s_score_transform);
    if (!w1 || !b1 || !w2 || !b2 || w1->dim() != 2 || w2->dim() != 2 || !PyTuple_Check(ch) || layout < 0 || layout > 2) throw Slow();
    const int64_t hid = w1->size(0), in = w1->size(1), n_ch = PyTuple_GET_SIZE(ch), out = layout == 2 ? n_ch : w2->size(0);
    if (hid > 1024 || in > 1024 || out > 8 || n_ch < out) throw Slow();
    m.n_hidden = static_cast<int32_t>(hid);
    m.n_in = static_cast<int32_t>(in);
    m.n_out = static_cast<int32_t>(out);
    m.W1 = static_cast<float*>(a.buf(w1, F32, {hid, in}));
    m.b1 = static_cast<float*>(a.buf(b1, F32, {hid}));
    if (layout == 2) {
        m.W2 = static_cast<float*>(a.buf(w2, F32, {1, hid ? hid : in}));
        m.b2 = static_cast<float*>(a.buf(b2, F32, {1}));
    } else {
        m.W2 = static_cast<float*>(a.buf(w2, F32, {out, hid}));
        m.b2 = static_cast<float*>(a.buf(b2, F32, {out}));
    }
    for (int64_t j = 0; j < out; ++j) {
        PyObject* g = PyTuple_GET_ITEM(ch, j);
        if (!PyLong_Check(g)) throw Slow();
        const long x = PyLong_AsLong(g);
        if (x < INT32_MIN || x > INT32_MAX || (x == -1 && PyErr_Occurred())) { PyErr_Clear(); throw Slow(); }
        m.gamma_choices[j] = static_cast<int32_t>(x);
    }
    m.feature_layout = static_cast<int32_t>(layout);
    m.score_transform = static_cast<int32_t>(transform);
    const int64_t n_comp = in - (layout == 0 ? 3 : layout == 1 ? 4 : 5);
    if (n_comp < 0) throw Slow();
    return n_comp;
}

struct Outs {
    float *H, *C, *feat, *scores;
    int32_t *gamma_next, *n_accepted, *out_tokens, *row_status;
    void* ws;
    size_t ws_bytes;
};
using size_fn = speckv_status (*)(const speckv_batch*, size_t*);

void read_workspace(const Args& a, const at::Tensor* w, const speckv_batch& c, size_fn size, void** ws, size_t* bytes) {
    size_t need = 0;
    if (!w || w->device() != a.dev || w->scalar_type() != at::ScalarType::Byte || !w->is_contiguous() || size(&c, &need) != SPECKV_OK ||
        static_cast<size_t>(w->numel()) < need)
        throw Slow();
    *ws = w->data_ptr();
    *bytes = static_cast<size_t>(w->numel());
}
void read_outs(Args& a, PyObject* out, const speckv_batch& c, int n_out, Outs& o) {
    const int64_t B = c.B, G = c.gamma_max;
    o.H = static_cast<float*>(a.buf(a.tensor(out, s_H), F32, {B, G}));
    o.C = static_cast<float*>(a.buf(a.tensor(out, s_C), F32, {B, G}));
    o.feat = static_cast<float*>(a.buf(a.tensor(out, s_feat), F32, {B, 4}));
    o.scores = n_out ? static_cast<float*>(a.buf(a.tensor(out, s_scores), F32, {B, n_out})) : nullptr;
    o.gamma_next = static_cast<int32_t*>(a.buf(a.tensor(out, s_gamma_next), I32, {B}));
    o.n_accepted = static_cast<int32_t*>(a.buf(a.tensor(out, s_n_accepted), I32, {B}));
    o.out_tokens = static_cast<int32_t*>(a.buf(a.tensor(out, s_out_tokens), I32, {B, G + 1}));
    o.row_status = static_cast<int32_t*>(a.buf(a.tensor(out, s_row_status), I32, {B}));
}

template <class F>
F fn_of(PyObject* o) {
    void* p = PyLong_AsVoidPtr(o);
    if (!p) { PyErr_Clear(); throw Slow(); }
    return reinterpret_cast<F>(p);
}
void* stream_of(const Args& a) { return c10::cuda::getCurrentCUDAStream(a.dev.index()).stream(); }

// The library call itself, with the interpreter lock released (a launch may wait for room in the stream's queue).
template <class F>
auto unlocked(F f) {
    struct Lock {
        PyThreadState* s = PyEval_SaveThread();
        ~Lock() { PyEval_RestoreThread(s); }
    } lock;
    return f();
}

// Runs f, which returns a status; None where the Python path has to take over.
template <class F>
PyObject* guarded(F f) {
    try {
        return PyLong_FromLong(f());
    } catch (const Slow&) {
    } catch (const std::exception&) {
        PyErr_Clear();
    }
    Py_RETURN_NONE;
}
bool arity(Py_ssize_t n, Py_ssize_t want) {
    if (n == want) return true;
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return false;
}

// step(fn, size_fn, batch, comp, mlp, out)
PyObject* py_step(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 6)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        speckv_mlp m{};
        Outs o{};
        const auto fn = fn_of<decltype(&speckv_step)>(x[0]);
        read_batch(a, x[2], c);
        const int64_t n_comp = read_mlp(a, x[4], m);
        const at::Tensor* comp = tensor_of(x[3]);
        const float* cp = n_comp > 0 ? static_cast<float*>(a.buf(comp, F32, {c.B, n_comp})) : nullptr;
        read_outs(a, x[5], c, m.n_out, o);
        read_workspace(a, a.tensor(x[5], s_workspace), c, fn_of<size_fn>(x[1]), &o.ws, &o.ws_bytes);
        void* st = stream_of(a);
        return unlocked([&] {
            return fn(&c, cp, &m, o.H, o.C, o.feat, o.scores, o.gamma_next, o.n_accepted, o.out_tokens, o.row_status, o.ws, o.ws_bytes, st);
        });
    });
}
// verify(fn, size_fn, batch, out)
PyObject* py_verify(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 4)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        Outs o{};
        const auto fn = fn_of<decltype(&speckv_verify)>(x[0]);
        read_batch(a, x[2], c);
        read_outs(a, x[3], c, 0, o);
        read_workspace(a, a.tensor(x[3], s_workspace), c, fn_of<size_fn>(x[1]), &o.ws, &o.ws_bytes);
        void* st = stream_of(a);
        return unlocked([&] { return fn(&c, o.n_accepted, o.out_tokens, o.row_status, o.ws, o.ws_bytes, st); });
    });
}
// signals(fn, size_fn, batch, out)
PyObject* py_signals(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 4)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        Outs o{};
        const auto fn = fn_of<decltype(&speckv_signals)>(x[0]);
        read_batch(a, x[2], c);
        read_outs(a, x[3], c, 0, o);
        read_workspace(a, a.tensor(x[3], s_workspace), c, fn_of<size_fn>(x[1]), &o.ws, &o.ws_bytes);
        void* st = stream_of(a);
        return unlocked([&] { return fn(&c, o.H, o.C, o.feat, o.row_status, o.ws, o.ws_bytes, st); });
    });
}
// select_gamma(fn, feat, comp, mlp, scores, gamma_next)
PyObject* py_select_gamma(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 6)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_mlp m{};
        const auto fn = fn_of<decltype(&speckv_select_gamma)>(x[0]);
        const at::Tensor* feat = tensor_of(x[1]);
        if (!feat || feat->dim() != 2 || !feat->is_cuda() || feat->size(0) > INT32_MAX) throw Slow();
        a.dev = feat->device();
        if (a.dev.index() != c10::cuda::current_device()) throw Slow();
        const int64_t B = feat->size(0), n_comp = read_mlp(a, x[3], m);
        const auto* f = static_cast<float*>(a.need(feat, F32, {B, 4}));
        const float* cp = n_comp > 0 ? static_cast<float*>(a.buf(tensor_of(x[2]), F32, {B, n_comp})) : nullptr;
        auto* s = static_cast<float*>(a.need(tensor_of(x[4]), F32, {B, m.n_out}));
        auto* g = static_cast<int32_t*>(a.need(tensor_of(x[5]), I32, {B}));
        void* st = stream_of(a);
        return unlocked([&] { return fn(static_cast<int32_t>(B), f, cp, &m, s, g, st); });
    });
}
// sample(fn, size_fn, batch, uniforms, tokens, row_status, workspace): the last three may be None and are then allocated;
// (status, tokens, row_status)
PyObject* py_sample(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 7)) return nullptr;
    try {
        Args a;
        speckv_batch c{};
        const auto fn = fn_of<decltype(&speckv_sample_draft)>(x[0]);
        const auto size = fn_of<size_fn>(x[1]);
        read_batch(a, x[2], c);
        const int64_t B = c.B, G = c.gamma_max;
        const auto* u = static_cast<float*>(a.need(tensor_of(x[3]), F32, {B, G}));
        const auto opt = at::TensorOptions().device(a.dev);
        at::Tensor tok, st, ws;
        if (const at::Tensor* t = tensor_of(x[4])) tok = *t; else tok = at::empty({B, G}, opt.dtype(I32));
        if (const at::Tensor* t = tensor_of(x[5])) st = *t; else st = at::empty({B}, opt.dtype(I32));
        auto* tp = static_cast<int32_t*>(a.buf(&tok, I32, {B, G}));
        auto* sp = static_cast<int32_t*>(a.buf(&st, I32, {B}));
        if (const at::Tensor* t = tensor_of(x[6])) {
            ws = *t;
        } else {
            size_t need = 0;
            if (size(&c, &need) != SPECKV_OK) throw Slow();
            ws = at::empty({static_cast<int64_t>(need)}, opt.dtype(at::ScalarType::Byte));
        }
        if (ws.dim() != 1) throw Slow();
        void* wp = a.buf(&ws, at::ScalarType::Byte, {ws.numel()});
        void* cs = stream_of(a);
        const int rc = unlocked([&] { return fn(&c, u, tp, sp, wp, static_cast<size_t>(ws.numel()), cs); });
        Ref pt(THPVariable_Wrap(tok)), ps(THPVariable_Wrap(st));
        if (!pt.p || !ps.p) return nullptr;
        return Py_BuildValue("(iOO)", rc, pt.p, ps.p);
    } catch (const Slow&) {
    } catch (const std::exception&) {
        PyErr_Clear();
    }
    Py_RETURN_NONE;
}

// ---- vocabulary-sharded step: the same checks as binding.py's calls (type, contiguity, device) ----
template <class T>
T* plain(const Args& a, const at::Tensor* t, at::ScalarType dt) {
    if (!t) return nullptr;
    if (t->device() != a.dev || t->scalar_type() != dt || !t->is_contiguous()) throw Slow();
    return static_cast<T*>(t->data_ptr());
}
constexpr auto F64 = at::ScalarType::Double;
constexpr auto U8 = at::ScalarType::Byte;
long long_of(PyObject* o) {
    if (!PyLong_Check(o)) throw Slow();
    const long v = PyLong_AsLong(o);
    if (v < 0 || v > INT32_MAX) { PyErr_Clear(); throw Slow(); }
    return v;
}
void read_ws(const Args& a, PyObject* o, void** ws, size_t* bytes) {
    const at::Tensor* t = tensor_of(o);
    if (!t) throw Slow();
    *ws = plain<void>(a, t, U8);
    *bytes = static_cast<size_t>(t->numel());
}

// shard_sweep(fn, batch, v_begin, state, tokl, workspace)
PyObject* py_shard_sweep(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 6)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        void* ws;
        size_t bytes;
        const auto fn = fn_of<decltype(&speckv_shard_sweep)>(x[0]);
        read_batch(a, x[1], c);
        const long v0 = long_of(x[2]);
        auto* state = plain<float>(a, tensor_of(x[3]), F32);
        auto* tokl = plain<float>(a, tensor_of(x[4]), F32);
        read_ws(a, x[5], &ws, &bytes);
        void* st = stream_of(a);
        return unlocked([&] { return fn(&c, v0, state, tokl, ws, bytes, st); });
    });
}
// shard_finish(fn, batch, n_shards, shard_width, V_total, all_state, all_tokl, comp, mlp, out, row_info)
PyObject* py_shard_finish(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 11)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        speckv_mlp m{};
        const auto fn = fn_of<decltype(&speckv_shard_finish)>(x[0]);
        read_batch(a, x[1], c);
        const long ns = long_of(x[2]), width = long_of(x[3]), total = long_of(x[4]);
        const auto* state = plain<float>(a, tensor_of(x[5]), F32);
        const auto* tokl = plain<float>(a, tensor_of(x[6]), F32);
        const auto* comp = plain<float>(a, tensor_of(x[7]), F32);
        const bool has_mlp = x[8] != Py_None;
        if (has_mlp) read_mlp(a, x[8], m);
        PyObject* o = x[9];
        auto f = [&](PyObject* name) { return plain<float>(a, a.tensor(o, name), F32); };
        auto i = [&](PyObject* name) { return plain<int32_t>(a, a.tensor(o, name), I32); };
        float *H = f(s_H), *C = f(s_C), *feat = f(s_feat), *scores = f(s_scores);
        int32_t *gn = i(s_gamma_next), *na = i(s_n_accepted), *ot = i(s_out_tokens), *rs = i(s_row_status);
        void* info = plain<void>(a, tensor_of(x[10]), U8);
        void* st = stream_of(a);
        return unlocked([&] {
            return fn(&c, static_cast<int32_t>(ns), static_cast<int32_t>(width), static_cast<int32_t>(total), state, tokl, comp,
                      has_mlp ? &m : nullptr, H, C, feat, scores, gn, na, ot, rs, info, st);
        });
    });
}
// shard_draw_sums(fn, batch, row_info, weight, workspace)
PyObject* py_shard_draw_sums(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 5)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        void* ws;
        size_t bytes;
        const auto fn = fn_of<decltype(&speckv_shard_draw_sums)>(x[0]);
        read_batch(a, x[1], c);
        const void* info = plain<void>(a, tensor_of(x[2]), U8);
        auto* w = plain<double>(a, tensor_of(x[3]), F64);
        read_ws(a, x[4], &ws, &bytes);
        void* st = stream_of(a);
        return unlocked([&] { return fn(&c, info, w, ws, bytes, st); });
    });
}
// shard_draw_pick(fn, batch, v_begin, rank, n_shards, row_info, all_weight, out_tokens, workspace)
PyObject* py_shard_draw_pick(PyObject*, PyObject* const* x, Py_ssize_t n) {
    if (!arity(n, 9)) return nullptr;
    return guarded([&] {
        Args a;
        speckv_batch c{};
        void* ws;
        size_t bytes;
        const auto fn = fn_of<decltype(&speckv_shard_draw_pick)>(x[0]);
        read_batch(a, x[1], c);
        const long v0 = long_of(x[2]), rank = long_of(x[3]), ns = long_of(x[4]);
        const void* info = plain<void>(a, tensor_of(x[5]), U8);
        const auto* w = plain<double>(a, tensor_of(x[6]), F64);
        auto* ot = plain<int32_t>(a, tensor_of(x[7]), I32);
        read_ws(a, x[8], &ws, &bytes);
        void* st = stream_of(a);
        return unlocked([&] { return fn(&c, v0, static_cast<int32_t>(rank), static_cast<int32_t>(ns), info, w, ot, ws, bytes, st); });
    });
}

#define METHOD(n) {#n, reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_##n)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    METHOD(step), METHOD(verify), METHOD(signals), METHOD(select_gamma), METHOD(sample), METHOD(shard_sweep), METHOD(shard_finish),
    METHOD(shard_draw_sums), METHOD(shard_draw_pick),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_speckv_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__speckv_torch(void) {
#define X(n) s_##n = PyUnicode_InternFromString(#n);
    NAMES(X)
#undef X
    return PyModule_Create(&module);
}
