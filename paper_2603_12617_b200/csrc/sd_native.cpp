// The calling thread's part of the hot entry points: what binding.py does for a call on device tensors (look at
// the arguments, allocate the outputs, ask for the stream, call the library), without the interpreter in between.
//
// Every function takes the arguments of its namesake in binding.py and returns a tuple (status, outputs...), or
// None where the arguments are anything but the plain case: exact torch.Tensor objects with storage, on the
// current CUDA device, of the shapes, types and layout that the entry point asks for.  binding.py then takes its
// general way, which raises what there is to raise; so nothing is refused here, and nothing accepted that it
// would refuse.
//
// What it saves, enqueueing one call on the calling thread (outputs allocated, B = 1): step 17.5 us through ctypes,
// 8.0 here; greedy 15.2, 6.0; error feedback 25.4, 12.3.  Of that the launches are 2 to 3 us each.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/sd_verify.h"

namespace {

// Entry points of the library that binding.py has loaded, by address.
struct Library {
    decltype(&sd_verify_feedback) step_f32 = nullptr;
    decltype(&sd_verify_feedback_bf16) step_bf16 = nullptr;
    decltype(&sd_verify_greedy) greedy = nullptr;
    decltype(&sd_verify_error_feedback) errors = nullptr;
    decltype(&sd_verify_feedback_hint) hint = nullptr;
    decltype(&sd_ensemble_feedback) ensemble = nullptr;
    decltype(&sd_lmhead_grad) lmhead = nullptr;
    decltype(&sd_vp_partial) vp_partial = nullptr;
    decltype(&sd_vp_finish) vp_finish = nullptr;
    decltype(&sd_vp_draw) vp_draw = nullptr;
    decltype(&sd_ensemble_workspace_bytes) ensemble_bytes = nullptr;
} lib;

constexpr int kVpRecordBytes = 48;

// A plain tensor: not a subclass, with memory behind it, dense, on the current CUDA device.
const at::Tensor* plain(PyObject* o, c10::DeviceIndex current) {
    if (current < 0 || !THPVariable_CheckExact(o)) return nullptr;
    const at::Tensor& t = THPVariable_Unpack(o);
    // (no tensor that stands for others: traced, batched, lazy, conjugated or negated)
    constexpr c10::DispatchKeySet known({c10::DispatchKey::CUDA, c10::DispatchKey::ADInplaceOrView, c10::DispatchKey::AutogradCUDA,
                                         c10::DispatchKey::AutocastCUDA});
    if (!t.defined() || (t.key_set() | known) != known || !t.has_storage() || t.layout() != at::kStrided || !t.is_cuda() ||
        t.device().index() != current || !t.is_contiguous())
        return nullptr;
    return &t;
}
// The current CUDA device, or -1 where the first argument of a call isn't on one (and there may be no driver to ask).
c10::DeviceIndex device_of(PyObject* o) {
    return THPVariable_CheckExact(o) && THPVariable_Unpack(o).defined() && THPVariable_Unpack(o).is_cuda() ? c10::cuda::current_device() : -1;
}
bool is_shape(const at::Tensor& t, c10::IntArrayRef s) { return t.sizes() == s; }
int logits_code(const at::Tensor& t) {
    return t.scalar_type() == at::kFloat ? SD_DTYPE_F32 : t.scalar_type() == at::kBFloat16 ? SD_DTYPE_BF16 : -1;
}
void* ptr(const at::Tensor& t) { return t.data_ptr(); }
bool small(int64_t v) { return v >= 0 && v < (int64_t)1 << 31; }
// A Python int or float as the C types of the library; false where ctypes would have more to say.
bool as_int(PyObject* o, int* v) {
    if (!PyLong_CheckExact(o)) return false;
    int over = 0;
    const long long x = PyLong_AsLongLongAndOverflow(o, &over);
    if (over || x < INT_MIN || x > INT_MAX) return false;
    *v = (int)x;
    return true;
}
bool as_float(PyObject* o, float* v) {
    if (!PyFloat_CheckExact(o) && !PyLong_CheckExact(o)) return false;
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    *v = (float)x;
    return true;
}
PyObject* none() { Py_RETURN_NONE; }

// The logits and tokens of a step: [B,k+1,V], [B,k,V], [B,k].
struct Step {
    const at::Tensor *T = nullptr, *D = nullptr, *x = nullptr;
    int B = 0, k = 0, V = 0, code = -1;
    c10::DeviceIndex dev = -1;
    bool take(PyObject* t, PyObject* d, PyObject* xs) {
        dev = device_of(t);
        T = plain(t, dev);
        D = T ? plain(d, dev) : nullptr;
        x = D ? plain(xs, dev) : nullptr;
        if (!x || T->dim() != 3) return false;
        const int64_t b = T->size(0), kk = T->size(1) - 1, v = T->size(2);
        if (kk < 1 || !small(b) || !small(kk) || !small(v)) return false;
        B = (int)b; k = (int)kk; V = (int)v;
        code = logits_code(*T);
        return code >= 0 && D->scalar_type() == T->scalar_type() && is_shape(*D, {b, kk, v}) &&
               x->scalar_type() == at::kInt && is_shape(*x, {b, kk});
    }
    const at::Tensor* uniforms(PyObject* o) const {
        const at::Tensor* u = plain(o, dev);
        return u && u->scalar_type() == at::kFloat && is_shape(*u, {(int64_t)B, (int64_t)k + 1}) ? u : nullptr;
    }
    at::Tensor make(c10::IntArrayRef shape, at::ScalarType type) const {
        return at::empty(shape, at::TensorOptions().dtype(type).device(c10::Device(c10::kCUDA, dev)));
    }
    void* stream() const { return c10::cuda::getCurrentCUDAStream(dev).stream(); }
};
size_t bytes_of(const at::Tensor& t) { return (size_t)t.numel() * t.element_size(); }
PyObject* wrap(const at::Tensor& t) {
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}
template <class... A> PyObject* answer(int rc, const A&... outs) {
    constexpr Py_ssize_t n = 1 + sizeof...(A);
    PyObject* r = PyTuple_New(n);
    if (!r) return nullptr;
    PyObject* items[n] = {PyLong_FromLong(rc), wrap(outs)...};
    for (Py_ssize_t i = 0; i < n; ++i) PyTuple_SET_ITEM(r, i, items[i]);
    return r;
}
// Calls `f` without the interpreter's lock, as ctypes does.  Its arguments are evaluated before the lock is given up: a
// tensor's address may have to be made (a lazy copy) or be refused with an exception.  And whatever leaves here leaves
// with the lock.
class Unlocked {
    PyThreadState* const state = PyEval_SaveThread();

public:
    Unlocked() = default;
    Unlocked(const Unlocked&) = delete;
    Unlocked& operator=(const Unlocked&) = delete;
    ~Unlocked() { PyEval_RestoreThread(state); }
};
template <class... P, class... A> int unlocked(int (*f)(P...), A... args) {
    const Unlocked guard;
    return f(args...);
}

// step(T, D, x, u, temperature, want_loss, want_grad) -> rc, accept_len, tokens, loss, grad
PyObject* step(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Step s;
    float tau;
    if (n != 7 || !s.take(a[0], a[1], a[2]) || !as_float(a[4], &tau)) return none();
    const at::Tensor* u = s.uniforms(a[3]);
    if (!u) return none();
    const bool grad = a[6] == Py_True, loss = grad || a[5] == Py_True;
    const at::Tensor len = s.make({s.B}, at::kInt), tokens = s.make({s.B, s.k + 1}, at::kInt);
    const at::Tensor l = loss ? s.make({s.B, s.k}, at::kFloat) : at::Tensor(), g = grad ? at::empty_like(*s.D) : at::Tensor();
    float* const lp = loss ? (float*)ptr(l) : nullptr;
    void* const gp = grad ? ptr(g) : nullptr;
    void* const st = s.stream();
    const int rc = s.code == SD_DTYPE_F32
                       ? unlocked(lib.step_f32, (const float*)ptr(*s.T), (const float*)ptr(*s.D), (const int32_t*)ptr(*s.x),
                            (const float*)ptr(*u),
                                  tau, s.B, s.k, s.V, (int32_t*)ptr(len), (int32_t*)ptr(tokens), lp, (float*)gp, st)
                       : unlocked(lib.step_bf16, (const uint16_t*)ptr(*s.T), (const uint16_t*)ptr(*s.D), (const int32_t*)ptr(*s.x),
                                  (const float*)ptr(*u), tau, s.B, s.k, s.V, (int32_t*)ptr(len), (int32_t*)ptr(tokens), lp, (uint16_t*)gp, st);
    return answer(rc, len, tokens, l, g);
    END_HANDLE_TH_ERRORS
}

// hint(T, D, x, u, temperature, hint, workspace) -> rc, accept_len, tokens, loss, grad, status, hint_err
PyObject* hint(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Step s;
    float tau;
    if (n != 7 || !s.take(a[0], a[1], a[2]) || !as_float(a[4], &tau)) return none();
    const at::Tensor *u = s.uniforms(a[3]), *h = u ? plain(a[5], s.dev) : nullptr, *ws = h ? plain(a[6], s.dev) : nullptr;
    if (!ws || h->scalar_type() != s.D->scalar_type() || !h->sizes().equals(s.D->sizes())) return none();
    const at::Tensor len = s.make({s.B}, at::kInt), tokens = s.make({s.B, s.k + 1}, at::kInt), l = s.make({s.B, s.k}, at::kFloat);
    const at::Tensor g = at::empty_like(*s.D), status = s.make({s.B}, at::kInt), err = s.make({s.B, s.k}, at::kFloat);
    void* const st = s.stream();
    const int rc = unlocked(lib.hint, ptr(*s.T), ptr(*s.D), (const int32_t*)ptr(*s.x), (const float*)ptr(*u), tau, s.B, s.k, s.V, s.code,
                            ptr(*h),
                            (int32_t*)ptr(len), (int32_t*)ptr(tokens), (float*)ptr(l), ptr(g), (float*)ptr(err), (uint32_t*)ptr(status),
                            ptr(*ws), bytes_of(*ws), st);
    return answer(rc, len, tokens, l, g, status, err);
    END_HANDLE_TH_ERRORS
}

// greedy(T, x, want_argmax) -> rc, accept_len, tokens, argmax
PyObject* greedy(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 3) return none();
    Step s;
    s.dev = device_of(a[0]);
    const at::Tensor *T = plain(a[0], s.dev), *x = T ? plain(a[1], s.dev) : nullptr;
    if (!x || T->dim() != 3) return none();
    const int64_t B = T->size(0), k1 = T->size(1), V = T->size(2);
    const int code = logits_code(*T);
    if (code < 0 || k1 < 2 || !small(B) || !small(k1) || !small(V) || x->scalar_type() != at::kInt || !is_shape(*x, {B, k1 - 1}))
        return none();
    const at::Tensor len = s.make({B}, at::kInt), tokens = s.make({B, k1}, at::kInt);
    const at::Tensor best = a[2] == Py_True ? s.make({B, k1}, at::kInt) : at::Tensor();
    int32_t* const bp = best.defined() ? (int32_t*)ptr(best) : nullptr;
    void* const st = s.stream();
    const int rc = unlocked(lib.greedy, ptr(*T), (const int32_t*)ptr(*x), (int)B, (int)k1 - 1, (int)V, code, (int32_t*)ptr(len),
                            (int32_t*)ptr(tokens), bp,
                            nullptr, 0, st);
    return answer(rc, len, tokens, best);
    END_HANDLE_TH_ERRORS
}

// errors(T, D, x, u, temperature, want_loss, want_grad, want_status) -> rc, accept_len, tokens, loss, error_grad, status
PyObject* errors(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Step s;
    float tau;
    if (n != 8 || !s.take(a[0], a[1], a[2]) || !as_float(a[4], &tau)) return none();
    const at::Tensor* u = s.uniforms(a[3]);
    if (!u) return none();
    const at::Tensor len = s.make({s.B}, at::kInt), tokens = s.make({s.B, s.k + 1}, at::kInt);
    const at::Tensor l = a[5] == Py_True ? s.make({s.B, s.k}, at::kFloat) : at::Tensor();
    const at::Tensor g = a[6] == Py_True ? s.make({s.B, s.V}, s.T->scalar_type()) : at::Tensor();
    const at::Tensor status = a[7] == Py_True ? s.make({s.B}, at::kInt) : at::Tensor();
    float* const lp = l.defined() ? (float*)ptr(l) : nullptr;
    void* const gp = g.defined() ? ptr(g) : nullptr;
    uint32_t* const sp = status.defined() ? (uint32_t*)ptr(status) : nullptr;
    void* const st = s.stream();
    const int rc = unlocked(lib.errors, ptr(*s.T), ptr(*s.D), (const int32_t*)ptr(*s.x), (const float*)ptr(*u), tau, s.B, s.k, s.V, s.code,
                            (int32_t*)ptr(len), (int32_t*)ptr(tokens), lp, gp, sp, nullptr, 0, st);
    return answer(rc, len, tokens, l, g, status);
    END_HANDLE_TH_ERRORS
}

// ensemble(T, drafts, temperature, epsilon, cum_loss, want_grad, want_status)
// -> rc, loss, [grad, ...], round_loss, cum_loss, weights, status
PyObject* ensemble(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    float tau, eps;
    if (n != 7 || !(PyList_CheckExact(a[1]) || PyTuple_CheckExact(a[1])) || !as_float(a[2], &tau) || !as_float(a[3], &eps)) return none();
    Step s;
    s.dev = device_of(a[0]);
    const at::Tensor* T = plain(a[0], s.dev);
    const Py_ssize_t N = PySequence_Fast_GET_SIZE(a[1]);
    if (!T || T->dim() != 3 || N < 1 || N > SD_MAX_LEARNERS) return none();
    const int64_t B = T->size(0), k = T->size(1) - 1, V = T->size(2);
    const int code = logits_code(*T);
    if (code < 0 || k < 1 || !small(B) || !small(k) || !small(V)) return none();
    const void* D[SD_MAX_LEARNERS] = {};
    void* G[SD_MAX_LEARNERS] = {};
    for (Py_ssize_t i = 0; i < N; ++i) {
        const at::Tensor* d = plain(PySequence_Fast_GET_ITEM(a[1], i), s.dev);
        if (!d || d->scalar_type() != T->scalar_type() || !is_shape(*d, {B, k, V})) return none();
        D[i] = ptr(*d);
    }
    const double* cum_in = nullptr;
    if (a[4] != Py_None) {
        const at::Tensor* c = plain(a[4], s.dev);
        if (!c || c->scalar_type() != at::kDouble || !is_shape(*c, {(int64_t)N})) return none();
        cum_in = (const double*)ptr(*c);
    }
    const at::Tensor loss = s.make({(int64_t)N, B, k}, at::kFloat), mean = s.make({(int64_t)N}, at::kDouble);
    const at::Tensor cum = s.make({(int64_t)N}, at::kDouble), weights = s.make({(int64_t)N}, at::kFloat);
    const at::Tensor status = a[6] == Py_True ? s.make({B}, at::kInt) : at::Tensor();
    const bool grad = a[5] == Py_True;
    at::Tensor g[SD_MAX_LEARNERS];
    for (Py_ssize_t i = 0; grad && i < N; ++i) {
        g[i] = s.make({B, k, V}, T->scalar_type());
        G[i] = ptr(g[i]);
    }
    // (scratch of the call's own: calls may overlap on the GPU)
    const size_t bytes = lib.ensemble_bytes((int)B, (int)k, (int)V, code, (int)N);
    const at::Tensor ws = bytes ? s.make({(int64_t)bytes}, at::kByte) : at::Tensor();
    void* const wp = bytes ? ptr(ws) : nullptr;
    uint32_t* const sp = status.defined() ? (uint32_t*)ptr(status) : nullptr;
    void* const st = s.stream();
    const int rc = unlocked(lib.ensemble, ptr(*T), D, (int)N, tau, eps, (int)B, (int)k, (int)V, code, cum_in, (float*)ptr(loss),
                            grad ? G : nullptr,
                            (double*)ptr(mean), (double*)ptr(cum), (float*)ptr(weights), sp, wp, bytes, st);
    PyObject* grads = Py_None;
    if (grad) {
        grads = PyList_New(N);
        if (!grads) return nullptr;
        for (Py_ssize_t i = 0; i < N; ++i) PyList_SET_ITEM(grads, i, wrap(g[i]));
    } else {
        Py_INCREF(grads);
    }
    PyObject* r = PyTuple_New(7);
    if (!r) {
        Py_DECREF(grads);
        return nullptr;
    }
    PyTuple_SET_ITEM(r, 0, PyLong_FromLong(rc));
    PyTuple_SET_ITEM(r, 1, wrap(loss));
    PyTuple_SET_ITEM(r, 2, grads);
    PyTuple_SET_ITEM(r, 3, wrap(mean));
    PyTuple_SET_ITEM(r, 4, wrap(cum));
    PyTuple_SET_ITEM(r, 5, wrap(weights));
    PyTuple_SET_ITEM(r, 6, wrap(status));
    return r;
    END_HANDLE_TH_ERRORS
}

// lmhead(grad_logits, hidden) -> rc, dW
PyObject* lmhead(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    if (n != 2) return none();
    Step s;
    s.dev = device_of(a[0]);
    const at::Tensor *g = plain(a[0], s.dev), *x = g ? plain(a[1], s.dev) : nullptr;
    if (!x || g->dim() != 2 || x->dim() != 2 || g->scalar_type() != at::kBFloat16 || x->scalar_type() != at::kBFloat16 ||
        g->size(0) != x->size(0) || !small(g->size(0)) || !small(g->size(1)) || !small(x->size(1)))
        return none();
    const at::Tensor out = s.make({g->size(1), x->size(1)}, at::kFloat);
    void* const st = s.stream();
    const int rc = unlocked(lib.lmhead, (const uint16_t*)ptr(*g), (const uint16_t*)ptr(*x), (int)g->size(0), (int)g->size(1), (int)x->size(1),
                            (float*)ptr(out), nullptr, st);
    return answer(rc, out);
    END_HANDLE_TH_ERRORS
}

// vp_partial(T, D, x, temperature, v_offset, V_total, workspace, out_records) -> rc, records
PyObject* vp_partial(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Step s;
    float tau;
    int off, total;
    if (n != 8 || !s.take(a[0], a[1], a[2]) || !as_float(a[3], &tau) || !as_int(a[4], &off) || !as_int(a[5], &total)) return none();
    const at::Tensor* ws = plain(a[6], s.dev);
    if (!ws) return none();
    at::Tensor rec;
    if (a[7] != Py_None) {
        const at::Tensor* r = plain(a[7], s.dev);
        if (!r || bytes_of(*r) < (size_t)s.B * (s.k + 1) * kVpRecordBytes) return none();
        rec = *r;
    } else {
        rec = s.make({(int64_t)s.B * (s.k + 1), kVpRecordBytes}, at::kByte);
    }
    void* const st = s.stream();
    const int rc = unlocked(lib.vp_partial, ptr(*s.T), ptr(*s.D), (const int32_t*)ptr(*s.x), tau, s.B, s.k, s.V, off, total, s.code,
                            ptr(rec), ptr(*ws),
                            bytes_of(*ws), st);
    return answer(rc, rec);
    END_HANDLE_TH_ERRORS
}

// vp_finish(T, D, x, u, temperature, v_offset, V_total, all_records, n_ranks, rank, workspace, want_loss, want_grad)
// -> rc, accept_len, loss, grad, mass, status
PyObject* vp_finish(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Step s;
    float tau;
    int off, total, ranks, rank;
    if (n != 13 || !s.take(a[0], a[1], a[2]) || !as_float(a[4], &tau) || !as_int(a[5], &off) || !as_int(a[6], &total) ||
        !as_int(a[8], &ranks) || !as_int(a[9], &rank))
        return none();
    const at::Tensor *u = s.uniforms(a[3]), *all = u ? plain(a[7], s.dev) : nullptr, *ws = all ? plain(a[10], s.dev) : nullptr;
    if (!ws || ranks < 1 || bytes_of(*all) != (size_t)ranks * s.B * (s.k + 1) * kVpRecordBytes) return none();
    const at::Tensor len = s.make({s.B}, at::kInt);
    const at::Tensor l = a[11] == Py_True ? s.make({s.B, s.k}, at::kFloat) : at::Tensor();
    const at::Tensor g = a[12] == Py_True ? at::empty_like(*s.D) : at::Tensor();
    const at::Tensor mass = s.make({s.B, 2}, at::kDouble), status = s.make({s.B}, at::kInt);
    float* const lp = l.defined() ? (float*)ptr(l) : nullptr;
    void* const gp = g.defined() ? ptr(g) : nullptr;
    void* const st = s.stream();
    const int rc = unlocked(lib.vp_finish, ptr(*s.T), ptr(*s.D), (const int32_t*)ptr(*s.x), (const float*)ptr(*u), tau, s.B, s.k, s.V, off,
                            total, s.code,
                            ptr(*all), ranks, rank, (int32_t*)ptr(len), lp, gp, (double*)ptr(mass), (uint32_t*)ptr(status), ptr(*ws),
                            bytes_of(*ws), st);
    return answer(rc, len, l, g, mass, status);
    END_HANDLE_TH_ERRORS
}

// vp_draw(T, D, x, u, temperature, v_offset, V_total, accept_len, all_masses, n_ranks, rank, status, workspace) -> rc, tokens
PyObject* vp_draw(PyObject*, PyObject* const* a, Py_ssize_t n) {
    HANDLE_TH_ERRORS
    Step s;
    float tau;
    int off, total, ranks, rank;
    if (n != 13 || !s.take(a[0], a[1], a[2]) || !as_float(a[4], &tau) || !as_int(a[5], &off) || !as_int(a[6], &total) ||
        !as_int(a[9], &ranks) || !as_int(a[10], &rank))
        return none();
    const at::Tensor *u = s.uniforms(a[3]), *len = u ? plain(a[7], s.dev) : nullptr, *mass = len ? plain(a[8], s.dev) : nullptr;
    const at::Tensor *status = mass ? plain(a[11], s.dev) : nullptr, *ws = status ? plain(a[12], s.dev) : nullptr;
    if (!ws || ranks < 1 || mass->scalar_type() != at::kDouble || mass->numel() != (int64_t)ranks * s.B * 2 ||
        len->scalar_type() != at::kInt || len->numel() < s.B || status->scalar_type() != at::kInt || status->numel() < s.B)
        return none();
    const at::Tensor tokens = s.make({s.B, s.k + 1}, at::kInt);
    void* const st = s.stream();
    const int rc = unlocked(lib.vp_draw, ptr(*s.T), ptr(*s.D), (const int32_t*)ptr(*s.x), (const float*)ptr(*u), tau, s.B, s.k, s.V, off,
                            total, s.code,
                            (const int32_t*)ptr(*len), (const double*)ptr(*mass), ranks, rank, (int32_t*)ptr(tokens), (uint32_t*)ptr(*status),
                            ptr(*ws), bytes_of(*ws), st);
    return answer(rc, tokens);
    END_HANDLE_TH_ERRORS
}

// bind(addresses): the entry points in the order of struct Library.
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
    void** const slots[] = {(void**)&lib.step_f32, (void**)&lib.step_bf16, (void**)&lib.greedy,    (void**)&lib.errors,
                            (void**)&lib.hint,     (void**)&lib.ensemble,   (void**)&lib.lmhead,
                            (void**)&lib.vp_partial, (void**)&lib.vp_finish, (void**)&lib.vp_draw, (void**)&lib.ensemble_bytes};
    constexpr Py_ssize_t want = sizeof slots / sizeof slots[0];
    if (n != want) {
        PyErr_SetString(PyExc_TypeError, "bind: wrong number of entry points");
        return nullptr;
    }
    for (Py_ssize_t i = 0; i < want; ++i) {
        void* p = PyLong_AsVoidPtr(a[i]);
        if (!p) {
            if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "bind: an entry point is null");
            return nullptr;
        }
        *slots[i] = p;
    }
    Py_RETURN_NONE;
}

#define SD_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&name)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SD_METHOD(bind),   SD_METHOD(step),       SD_METHOD(hint),      SD_METHOD(greedy),  SD_METHOD(errors), SD_METHOD(ensemble),
                         SD_METHOD(lmhead), SD_METHOD(vp_partial), SD_METHOD(vp_finish), SD_METHOD(vp_draw), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "sd_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit_sd_native(void) { return PyModule_Create(&module); }
