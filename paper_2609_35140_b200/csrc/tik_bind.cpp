// CPython module behind binding.py: takes torch tensors, checks them, makes the outputs and the
// scratch, and calls the C entry point of the same name on the current stream.
//
// Every call here is on the critical path of a small decode or prefill step: marshalling the same
// arguments through ctypes (a Python object per pointer, attribute look-ups per tensor, a stream
// object) took ~15 us of host time per call where the kernels behind it run 3 to 20 us, so a rollout
// layer of 12 launches was bound by the host.  Nothing is kept between calls except the
// per-device library context.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <mutex>
#include <string>

#include "../../include/tik.h"

namespace {

PyObject* g_error = nullptr;                 // binding.TikError

// A Python exception is set; unwinds to the entry point.
struct PyError {};

[[noreturn]] void raise(PyObject* type, const std::string& msg) {
    PyErr_SetString(type, msg.c_str());
    throw PyError{};
}
[[noreturn]] void raise_tik(const std::string& msg) { raise(g_error, msg); }

// ---------------------------------------------------------------- per-device context
constexpr int MAX_DEVICES = 64;
std::mutex g_ctx_mutex;
std::atomic<tik_ctx*> g_ctx[MAX_DEVICES];

tik_ctx* context(int device) {
    if (device < 0 || device >= MAX_DEVICES) raise_tik("device ordinal out of range");
    tik_ctx* c = g_ctx[device].load(std::memory_order_acquire);
    if (c) return c;
    std::lock_guard<std::mutex> lock(g_ctx_mutex);
    c = g_ctx[device].load(std::memory_order_acquire);
    if (c) return c;
    const tik_status rc = tik_create(&c, device);
    if (rc != TIK_OK) raise_tik(std::string("tik_create failed: ") + tik_status_str(rc));
    g_ctx[device].store(c, std::memory_order_release);
    return c;
}

int current_device() {
    if (c10::cuda::device_count() < 1) raise_tik("tik needs a CUDA device; there is no CPU path");
    return static_cast<int>(c10::cuda::current_device());
}

// ---------------------------------------------------------------- arguments
struct Args {
    PyObject* const* a;
    Py_ssize_t n;
    Py_ssize_t i = 0;
    PyObject* next() {
        if (i >= n) raise(PyExc_TypeError, "too few arguments");
        return a[i++];
    }
    const at::Tensor& tensor() {
        PyObject* o = next();
        if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string("expected a tensor, got ") + Py_TYPE(o)->tp_name);
        return THPVariable_Unpack(o);
    }
    // nullptr for None
    const at::Tensor* opt() {
        if (i < n && a[i] == Py_None) {
            ++i;
            return nullptr;
        }
        return &tensor();
    }
    int64_t integer() {
        const long long v = PyLong_AsLongLong(next());
        if (v == -1 && PyErr_Occurred()) throw PyError{};
        return v;
    }
    int int32() {
        const int64_t v = integer();
        if (v < INT32_MIN || v > INT32_MAX) raise(PyExc_OverflowError, "integer argument out of range");
        return static_cast<int>(v);
    }
    float real() {
        const double v = PyFloat_AsDouble(next());
        if (v == -1.0 && PyErr_Occurred()) throw PyError{};
        return static_cast<float>(v);
    }
};

void* ptr(const at::Tensor& t) {
    if (!t.is_cuda() || !t.is_contiguous()) raise_tik("tensors must be contiguous CUDA tensors");
    return t.data_ptr();
}
void* ptr(const at::Tensor& t, at::ScalarType type) {
    void* p = ptr(t);
    if (t.scalar_type() != type)
        raise_tik(std::string("expected dtype ") + at::toString(type) + ", got " + at::toString(t.scalar_type()));
    return p;
}
void* ptr(const at::Tensor* t, at::ScalarType type) { return t ? ptr(*t, type) : nullptr; }
void* bf(const at::Tensor& t) { return ptr(t, at::kBFloat16); }
void* bf(const at::Tensor* t) { return ptr(t, at::kBFloat16); }
float* f32(const at::Tensor* t) { return static_cast<float*>(ptr(t, at::kFloat)); }
int32_t* i32(const at::Tensor& t) { return static_cast<int32_t*>(ptr(t, at::kInt)); }
int32_t* i32(const at::Tensor* t) { return t ? i32(*t) : nullptr; }

void want_rank(const at::Tensor& t, int64_t rank) {
    if (t.dim() != rank)
        raise(PyExc_ValueError, "expected a tensor with " + std::to_string(rank) + " dimensions, got " + std::to_string(t.dim()));
}
// an argument of which only one axis' size is read
void want_axis(const at::Tensor& t, int64_t axis) {
    if (t.dim() <= axis) raise(PyExc_IndexError, "axis " + std::to_string(axis) + " of a tensor with " + std::to_string(t.dim()) + " dimensions");
}
int dim(const at::Tensor& t, int64_t i) {
    const int64_t v = t.size(i);
    if (v > INT32_MAX) raise(PyExc_OverflowError, "tensor dimension out of range");
    return static_cast<int>(v);
}

at::Tensor empty(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor& like) {
    if (!like.is_cuda()) raise_tik("tensors must be contiguous CUDA tensors");
    return at::detail::empty_cuda(sizes, type, like.device(), std::nullopt);
}

void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

void check(tik_status rc, const tik_ctx* ctx) {
    if (rc != TIK_OK) raise_tik(std::string(tik_status_str(rc)) + ": " + tik_last_error(ctx));
}

// Runs a C entry point without the interpreter lock (a launch blocks while the launch queue is full).  f reads
// plain values only: whatever inspects a tensor or may raise happens before, under the lock.  An exception that
// leaves f all the same passes with the lock taken back, so that its handler may set a Python error.
template <class F>
tik_status unlocked(F&& f) {
    struct Unlock {
        PyThreadState* state = PyEval_SaveThread();
        ~Unlock() { PyEval_RestoreThread(state); }
    } unlock;
    return f();
}

struct Scratch {
    at::Tensor own;
    void* p = nullptr;
    size_t bytes = 0;
    void use(const at::Tensor& t) {
        p = ptr(t);
        bytes = t.nbytes();
    }
    void make(size_t need, const at::Tensor& like) {
        own = empty({static_cast<int64_t>(need)}, at::kByte, like);
        p = own.data_ptr();
        bytes = need;
    }
};

// Scratch of the full-sequence kernels: None = what the op asks for, False = none, a tensor = that one.
Scratch plan_ws(PyObject* ws, int op, int64_t S, int64_t max_positions, const at::Tensor& like) {
    Scratch s;
    if (ws == Py_False) return s;
    if (ws != Py_None) {
        if (!THPVariable_Check(ws)) raise(PyExc_TypeError, "ws must be a tensor, None or False");
        s.use(THPVariable_Unpack(ws));
        return s;
    }
    const size_t need = tik_workspace_bytes(op, S, 0, 0, 0, max_positions, 0, 0);
    if (need > 0) s.make(need, like);
    return s;
}
Scratch sized_ws(const at::Tensor* ws, size_t need, const at::Tensor& like) {
    Scratch s;
    if (ws) s.use(*ws);
    else s.make(need > 16 ? need : 16, like);
    return s;
}

PyObject* wrap(const at::Tensor* given, at::Tensor& made) {
    return THPVariable_Wrap(given ? *given : made);
}
// `given` or a new tensor of those sizes
const at::Tensor& out_or(const at::Tensor* given, at::Tensor& made, at::IntArrayRef sizes, at::ScalarType type,
                         const at::Tensor& like) {
    if (given) return *given;
    made = empty(sizes, type, like);
    return made;
}

// ---------------------------------------------------------------- entry points (positional, in binding.py's order)

PyObject* attn_train_fwd(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &q = a.tensor(), &k = a.tensor();
    const at::Tensor* v = a.opt();
    const at::Tensor& cu = a.tensor();
    const int max_seqlen = a.int32();
    const float scale = a.real();
    const at::Tensor *o_in = a.opt(), *lse = a.opt();
    PyObject* ws_in = a.next();
    want_rank(q, 3);
    want_axis(k, 1);
    at::Tensor made;
    const at::Tensor& o = out_or(o_in, made, q.sizes(), q.scalar_type(), q);
    const int S = static_cast<int>(cu.numel() - 1);
    const Scratch ws = plan_ws(ws_in, TIK_OP_ATTN_TRAIN_FWD, S, max_seqlen, q);
    void *qp = bf(q), *kp = bf(k), *vp = bf(v), *op = bf(o), *st = stream();
    float* lp = f32(lse);
    int32_t* cp = i32(cu);
    const int Hq = dim(q, 1), Hkv = dim(k, 1), d = dim(q, 2);
    const int64_t tot = q.size(0);
    check(unlocked([&] { return tik_attn_train_fwd(ctx, qp, kp, vp, op, lp, cp, S, tot, max_seqlen, Hq, Hkv, d, scale, ws.p,
                                                   ws.bytes, st); }), ctx);
    return wrap(o_in, made);
}

PyObject* attn_train_bwd(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &q = a.tensor(), &k = a.tensor(), &v = a.tensor();
    const at::Tensor *o = a.opt(), *d_o = a.opt(), *lse = a.opt();
    const at::Tensor& cu = a.tensor();
    const int max_seqlen = a.int32();
    const float scale = a.real();
    const at::Tensor* ws_in = a.opt();
    want_rank(q, 3);
    want_axis(k, 1);
    const int64_t tot = q.size(0);
    const int Hq = dim(q, 1), Hkv = dim(k, 1), d = dim(q, 2), S = static_cast<int>(cu.numel() - 1);
    const Scratch ws = sized_ws(ws_in, tik_workspace_bytes(TIK_OP_ATTN_TRAIN_BWD, tot, Hq, Hkv, d, 0, 0, 0), q);
    at::Tensor dq = empty(q.sizes(), q.scalar_type(), q), dk = empty(k.sizes(), k.scalar_type(), k),
               dv = empty(v.sizes(), v.scalar_type(), v);
    void *qp = bf(q), *kp = bf(k), *vp = bf(v), *op = bf(o), *gp = bf(d_o), *dqp = bf(dq), *dkp = bf(dk), *dvp = bf(dv), *st = stream();
    float* lp = f32(lse);
    int32_t* cp = i32(cu);
    check(unlocked([&] { return tik_attn_train_bwd(ctx, qp, kp, vp, op, gp, lp, dqp, dkp, dvp, cp, S, tot, max_seqlen, Hq, Hkv,
                                                   d, scale, ws.p, ws.bytes, st); }), ctx);
    PyObject *a0 = THPVariable_Wrap(dq), *a1 = THPVariable_Wrap(dk), *a2 = THPVariable_Wrap(dv);
    return Py_BuildValue("(NNN)", a0, a1, a2);
}

// caches, block table and what they say about the layout
struct Cache {
    void *k, *v;
    int32_t* table;
    int max_blocks, num_pages, Hkv, page, d;
};
Cache cache_of(const at::Tensor& kc, const at::Tensor& vc, const at::Tensor& table) {
    want_rank(kc, 4);
    want_axis(table, 1);
    return {bf(kc), bf(vc), i32(table), dim(table, 1), dim(kc, 0), dim(kc, 1), dim(kc, 2), dim(kc, 3)};
}

PyObject* kv_cache_write(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor& k = a.tensor();
    const at::Tensor *v = a.opt(), *cu = a.opt();
    const at::Tensor &lens = a.tensor(), &kc = a.tensor(), &vc = a.tensor(), &table = a.tensor();
    want_axis(k, 0);
    const Cache c = cache_of(kc, vc, table);
    void *kp = bf(k), *vp = bf(v), *st = stream();
    int32_t *cp = i32(cu), *lp = i32(lens);
    const int S = static_cast<int>(lens.numel());
    const int64_t n = k.size(0);
    check(unlocked([&] { return tik_kv_cache_write(ctx, kp, vp, cp, lp, c.k, c.v, c.table, c.max_blocks, S, n, c.Hkv, c.d,
                                                   c.page, c.num_pages, st); }), ctx);
    Py_RETURN_NONE;
}

PyObject* qk_norm_rope_kv_write(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &q = a.tensor(), &k = a.tensor();
    const at::Tensor *v = a.opt(), *wq = a.opt(), *wk = a.opt();
    const float eps = a.real();
    const at::Tensor &cs = a.tensor(), &cu = a.tensor();
    const at::Tensor *lens = a.opt(), *kc = a.opt(), *vc = a.opt(), *table = a.opt();
    want_rank(q, 3);
    want_axis(k, 1);
    want_axis(cs, 0);
    if (kc) want_axis(*kc, 2);
    if (table) want_axis(*table, 1);
    const int Hq = dim(q, 1), Hkv = dim(k, 1), d = dim(q, 2), page = kc ? dim(*kc, 2) : 0, pages = kc ? dim(*kc, 0) : 0;
    const int max_blocks = table ? dim(*table, 1) : 0, S = static_cast<int>(cu.numel() - 1);
    void *qp = bf(q), *kp = bf(k), *vp = bf(v), *wqp = bf(wq), *wkp = bf(wk), *kcp = bf(kc), *vcp = bf(vc), *st = stream();
    const float* csp = f32(&cs);
    int32_t *cp = i32(cu), *lp = i32(lens), *tp = i32(table);
    const int64_t n = q.size(0);
    const int max_pos = dim(cs, 0);
    check(unlocked([&] { return tik_qk_norm_rope_kv_write(ctx, qp, kp, vp, wqp, wkp, eps, csp, max_pos, cp, lp, kcp, vcp, tp,
                                                          max_blocks, S, n, Hq, Hkv, d, page, pages, st); }), ctx);
    Py_RETURN_NONE;
}

PyObject* rmsnorm(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &x = a.tensor(), &w = a.tensor();
    const float eps = a.real();
    const at::Tensor *res = a.opt(), *y_in = a.opt();
    want_rank(x, 2);
    at::Tensor made;
    const at::Tensor& y = out_or(y_in, made, x.sizes(), x.scalar_type(), x);
    void *xp = bf(x), *rp = bf(res), *wp = bf(w), *yp = bf(y), *st = stream();
    const int64_t T = x.size(0);
    const int H = dim(x, 1);
    check(unlocked([&] { return tik_rmsnorm(ctx, xp, rp, wp, yp, eps, T, H, st); }), ctx);
    return wrap(y_in, made);
}

PyObject* swiglu(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor& gu = a.tensor();
    const at::Tensor* out_in = a.opt();
    want_rank(gu, 2);
    at::Tensor made;
    const int64_t T = gu.size(0);
    const int inter = dim(gu, 1) / 2;
    const at::Tensor& out = out_or(out_in, made, {T, inter}, at::kBFloat16, gu);
    void *gp = bf(gu), *op = bf(out), *st = stream();
    check(unlocked([&] { return tik_swiglu(ctx, gp, op, T, inter, st); }), ctx);
    return wrap(out_in, made);
}

PyObject* linear(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &x = a.tensor(), &w = a.tensor();
    const at::Tensor* y_in = a.opt();
    want_rank(x, 2);
    want_axis(w, 0);
    at::Tensor made;
    const int64_t T = x.size(0);
    const int K = dim(x, 1), N = dim(w, 0);
    const at::Tensor& y = out_or(y_in, made, {T, N}, at::kBFloat16, x);
    void *xp = bf(x), *wp = bf(w), *yp = bf(y), *st = stream();
    check(unlocked([&] { return tik_linear(ctx, xp, wp, yp, T, K, N, st); }), ctx);
    return wrap(y_in, made);
}

PyObject* attn_prefill(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor& q = a.tensor();
    const at::Tensor* cu = a.opt();
    const at::Tensor &lens = a.tensor(), &kc = a.tensor(), &vc = a.tensor(), &table = a.tensor();
    const int max_q = a.int32(), max_ctx = a.int32();
    const float scale = a.real();
    const at::Tensor *o_in = a.opt(), *lse = a.opt();
    PyObject* ws_in = a.next();
    want_rank(q, 3);
    const Cache c = cache_of(kc, vc, table);
    at::Tensor made;
    const at::Tensor& o = out_or(o_in, made, q.sizes(), q.scalar_type(), q);
    const int64_t tot = q.size(0);
    const int S = static_cast<int>(lens.numel()), Hq = dim(q, 1), d = dim(q, 2);
    const Scratch ws = plan_ws(ws_in, TIK_OP_ATTN_PREFILL, S, max_ctx, q);
    void *qp = bf(q), *op = bf(o), *st = stream();
    float* lp = f32(lse);
    int32_t *cp = i32(cu), *np = i32(lens);
    check(unlocked([&] { return tik_attn_prefill(ctx, qp, op, lp, cp, np, c.k, c.v, c.table, c.max_blocks, S, tot, max_q,
                                                 max_ctx, Hq, c.Hkv, d, c.page, c.num_pages, scale, ws.p, ws.bytes, st); }), ctx);
    return wrap(o_in, made);
}

PyObject* attn_prefill_kv(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor& q = a.tensor();
    const at::Tensor *k = a.opt(), *v = a.opt(), *cu = a.opt();
    const at::Tensor &lens = a.tensor(), &kc = a.tensor(), &vc = a.tensor(), &table = a.tensor();
    const int max_q = a.int32(), max_ctx = a.int32();
    const float scale = a.real();
    const at::Tensor *o_in = a.opt(), *lse = a.opt();
    PyObject* ws_in = a.next();
    want_rank(q, 3);
    const Cache c = cache_of(kc, vc, table);
    at::Tensor made;
    const at::Tensor& o = out_or(o_in, made, q.sizes(), q.scalar_type(), q);
    const int64_t tot = q.size(0);
    const int S = static_cast<int>(lens.numel()), Hq = dim(q, 1), d = dim(q, 2);
    const Scratch ws = plan_ws(ws_in, TIK_OP_ATTN_PREFILL, S, max_ctx, q);
    void *qp = bf(q), *kp = bf(k), *vp = bf(v), *op = bf(o), *st = stream();
    float* lp = f32(lse);
    int32_t *cp = i32(cu), *np = i32(lens);
    check(unlocked([&] { return tik_attn_prefill_kv(ctx, qp, kp, vp, op, lp, cp, np, c.k, c.v, c.table, c.max_blocks, S,
                                                    tot, max_q, max_ctx, Hq, c.Hkv, d, c.page, c.num_pages, scale, ws.p,
                                                    ws.bytes, st); }), ctx);
    return wrap(o_in, made);
}

PyObject* attn_decode(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &q = a.tensor(), &lens = a.tensor(), &kc = a.tensor(), &vc = a.tensor(), &table = a.tensor();
    const int max_ctx = a.int32();
    const float scale = a.real();
    const at::Tensor *ws_in = a.opt(), *o_in = a.opt(), *lse = a.opt();
    want_rank(q, 3);
    const Cache c = cache_of(kc, vc, table);
    const int B = dim(q, 0), Hq = dim(q, 1), d = dim(q, 2);
    const Scratch ws = sized_ws(ws_in, tik_workspace_bytes(TIK_OP_ATTN_DECODE, B, Hq, c.Hkv, d, max_ctx, 0, 0), q);
    at::Tensor made;
    const at::Tensor& o = out_or(o_in, made, q.sizes(), q.scalar_type(), q);
    void *qp = bf(q), *op = bf(o), *st = stream();
    float* lp = f32(lse);
    int32_t* np = i32(lens);
    check(unlocked([&] { return tik_attn_decode(ctx, qp, op, lp, np, c.k, c.v, c.table, c.max_blocks, B, max_ctx, Hq, c.Hkv, d,
                                                c.page, c.num_pages, scale, ws.p, ws.bytes, st); }), ctx);
    return wrap(o_in, made);
}

PyObject* attn_decode_static(Args a) {
    const at::Tensor &q = a.tensor(), &lens = a.tensor(), &kc = a.tensor(), &vc = a.tensor(), &table = a.tensor();
    const int max_ctx = a.int32();
    const float scale = a.real();
    const at::Tensor& o = a.tensor();
    const at::Tensor *lse = a.opt(), *flags = a.opt();
    want_rank(q, 3);
    const Cache c = cache_of(kc, vc, table);
    const int B = dim(q, 0), Hq = dim(q, 1), d = dim(q, 2);
    void *qp = bf(q), *op = bf(o), *st = stream();
    float* lp = f32(lse);
    int32_t *np = i32(lens), *fp = i32(flags);
    const tik_status rc = unlocked([&] { return tik_attn_decode_static(qp, op, lp, np, c.k, c.v, c.table, c.max_blocks, B, max_ctx,
                                                                       Hq, c.Hkv, d, c.page, c.num_pages, scale, fp, st); });
    return PyLong_FromLong(rc);
}

PyObject* token_logprob(Args a) {
    tik_ctx* ctx = context(current_device());
    const at::Tensor &x = a.tensor(), &w = a.tensor(), &ids = a.tensor();
    const float inv_temperature = a.real();
    const at::Tensor *ws_in = a.opt(), *lp_in = a.opt(), *lse = a.opt();
    want_rank(x, 2);
    want_axis(w, 0);
    const int64_t T = x.size(0);
    const int H = dim(x, 1), V = dim(w, 0);
    const Scratch ws = sized_ws(ws_in, tik_workspace_bytes(TIK_OP_TOKEN_LOGPROB, T, 0, 0, 0, 0, H, V), x);
    at::Tensor made;
    const at::Tensor& lp = out_or(lp_in, made, {T}, at::kFloat, x);
    void *xp = bf(x), *wp = bf(w), *st = stream();
    int32_t* ip = i32(ids);
    float *op = f32(&lp), *sp = f32(lse);
    check(unlocked([&] { return tik_token_logprob(ctx, xp, wp, ip, op, sp, T, H, V, inv_temperature, ws.p, ws.bytes, st); }), ctx);
    return wrap(lp_in, made);
}

PyObject* context_handle(Args a) {           // device ordinal (or None: the current device) -> the context's address
    PyObject* o = a.next();
    int device = current_device();
    if (o != Py_None) {
        --a.i;
        device = a.int32();
    }
    return PyLong_FromVoidPtr(context(device));
}

PyObject* init(Args a) {
    PyObject* e = a.next();
    Py_INCREF(e);
    Py_XSETREF(g_error, e);
    Py_RETURN_NONE;
}

template <PyObject* (*F)(Args)>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
    HANDLE_TH_ERRORS                         // torch's own errors (out of memory among them) keep their types
    try {
        return F(Args{args, n});
    } catch (const PyError&) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

#define TIK_DEF(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(entry<name>)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    TIK_DEF(init), TIK_DEF(context_handle), TIK_DEF(attn_train_fwd), TIK_DEF(attn_train_bwd), TIK_DEF(kv_cache_write),
    TIK_DEF(qk_norm_rope_kv_write), TIK_DEF(rmsnorm), TIK_DEF(swiglu), TIK_DEF(linear), TIK_DEF(attn_prefill),
    TIK_DEF(attn_prefill_kv), TIK_DEF(attn_decode), TIK_DEF(attn_decode_static), TIK_DEF(token_logprob),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_tikbind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tikbind(void) { return PyModule_Create(&module_def); }
