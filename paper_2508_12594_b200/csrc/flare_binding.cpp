// Argument marshalling between torch tensors and the C-ABI of libflare, as a Python extension module.
//
// A small problem takes the GPU a few microseconds per kernel, so what a call costs on the host is most of it: checking
// nine tensors and converting them to C pointers in Python took longer than the kernels ran.  Here a check is a few loads,
// and the convenience calls take their scratch (workspace, statistics) in one allocation.  Measured, host time of a call: float32
// forward of 1024 tokens 45 -> 17 us, training step of 16384 tokens 127 -> 61 us (its launches are most of that).
//
// The module does not link libflare: flare.py loads the library and hands over the addresses of its functions (bind).
#include <torch/csrc/autograd/python_variable.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>

#include <map>
#include <string>

#include "../../include/flare.h"

namespace {

struct Library {
    decltype(&flare_workspace_bytes) workspace_bytes;
    decltype(&flare_encode) encode;
    decltype(&flare_encode_static_scratch) encode_static_scratch;
    decltype(&flare_decode) decode;
    decltype(&flare_forward) forward;
    decltype(&flare_backward) backward;
    decltype(&flare_forward_host) forward_host;
    decltype(&flare_forward_variant) forward_variant;
    decltype(&flare_backward_variant) backward_variant;
    decltype(&flare_spectral_gram) spectral_gram;
    decltype(&flare_spectral_eig) spectral_eig;
} lib{};
PyObject *flare_error = nullptr;   // the exception class (status, where)

// Raised inside the marshalling code after a Python error has been set.
struct PythonError {};

[[noreturn]] void fail(PyObject *type, const std::string &text) {
    PyErr_SetString(type, text.c_str());
    throw PythonError{};
}
void check_status(int rc, const char *where) {
    if (rc == FLARE_OK) return;
    PyObject *e = PyObject_CallFunction(flare_error, "is", rc, where);
    if (e) {
        PyErr_SetObject(flare_error, e);
        Py_DECREF(e);
    }
    throw PythonError{};
}

std::string dtype_name(at::ScalarType t) {
    switch (t) {
        case at::kFloat: return "torch.float32";
        case at::kBFloat16: return "torch.bfloat16";
        case at::kHalf: return "torch.float16";
        case at::kByte: return "torch.uint8";
        default: return c10::toString(t);
    }
}
std::string shape_text(at::IntArrayRef s) {
    std::string r = "(";
    for (size_t i = 0; i < s.size(); ++i) r += std::to_string(s[i]) + (s.size() == 1 ? "," : i + 1 < s.size() ? ", " : "");
    return r + ")";
}

const at::Tensor &tensor(PyObject *o) {
    if (!THPVariable_Check(o)) fail(PyExc_TypeError, "expected a torch tensor");
    return THPVariable_Unpack(o);
}
void check(const at::Tensor &t, at::ScalarType dtype, at::IntArrayRef shape, bool cuda = true) {
    if (cuda && !t.is_cuda()) fail(PyExc_ValueError, "expected a CUDA tensor");
    if (!t.is_contiguous()) fail(PyExc_ValueError, "expected a contiguous tensor");
    if (t.scalar_type() != dtype) fail(PyExc_TypeError, "expected " + dtype_name(dtype) + ", got " + dtype_name(t.scalar_type()));
    if (t.sizes() != shape) fail(PyExc_ValueError, "expected shape " + shape_text(shape) + ", got " + shape_text(t.sizes()));
}

// The tensors of one call: shapes follow from the descriptor, the call's element type from K.
struct Call {
    const flare_desc_t *d;
    at::ScalarType dt;
    void *ptr(PyObject *o, at::ScalarType dtype, at::IntArrayRef shape, bool cuda = true) const {
        if (o == Py_None) return nullptr;
        const at::Tensor &t = tensor(o);
        check(t, dtype, shape, cuda);
        return t.data_ptr();
    }
    void *q(PyObject *o, bool shared = false, bool cuda = true) const {
        return shared ? ptr(o, dt, {d->M, d->D}, cuda) : ptr(o, dt, {d->H, d->M, d->D}, cuda);
    }
    void *tok(PyObject *o, bool cuda = true) const { return ptr(o, dt, {d->B, d->N, d->H, d->D}, cuda); }
    uint8_t *mask(PyObject *o, bool cuda = true) const { return (uint8_t *)ptr(o, at::kByte, {d->B, d->N}, cuda); }
    float *z(PyObject *o) const { return (float *)ptr(o, at::kFloat, {d->B, d->H, d->M, d->D}); }
    float *le(PyObject *o) const { return (float *)ptr(o, at::kFloat, {d->B, d->H, d->M}); }
    float *ld(PyObject *o) const { return (float *)ptr(o, at::kFloat, {d->B, d->N, d->H}); }
    float *dq(PyObject *o, bool shared = false) const {
        return (float *)(shared ? ptr(o, at::kFloat, {d->M, d->D}) : ptr(o, at::kFloat, {d->H, d->M, d->D}));
    }
};
struct Workspace {
    void *p = nullptr;
    size_t n = 0;
    explicit Workspace(PyObject *o) {
        if (o == Py_None) return;
        const at::Tensor &t = tensor(o);
        check(t, at::kByte, t.sizes());
        p = t.data_ptr();
        n = (size_t)t.numel();
    }
};

// A FlareDesc (a ctypes structure: its memory through the buffer protocol).
struct Desc {
    Py_buffer view;
    explicit Desc(PyObject *o) {
        if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) throw PythonError{};
        if (view.len != (Py_ssize_t)sizeof(flare_desc_t)) {
            PyBuffer_Release(&view);
            fail(PyExc_TypeError, "expected a FlareDesc");
        }
    }
    ~Desc() { PyBuffer_Release(&view); }
    Desc(const Desc &) = delete;
    const flare_desc_t *get() const { return (const flare_desc_t *)view.buf; }
};

flare_stream_t stream_of(PyObject *o) {
    if (o == Py_None) return (flare_stream_t)c10::cuda::getCurrentCUDAStream().stream();
    PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
    if (!h) throw PythonError{};
    void *p = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    if (PyErr_Occurred()) throw PythonError{};
    return (flare_stream_t)p;
}

// Every function below takes positional arguments only; the defaults and keyword names are those of the wrappers in flare.py.
template <typename F>
PyObject *guarded(Py_ssize_t got, Py_ssize_t want, F body) {
    if (got != want) {
        PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, got);
        return nullptr;
    }
    try {
        return body();
    } catch (const PythonError &) {
        return nullptr;
    } catch (const std::exception &e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
// Call into the library without the interpreter's lock.
template <typename F>
int unlocked(F call) {
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = call();
    Py_END_ALLOW_THREADS
    return rc;
}

#define BINDING(name, count) PyObject *py_##name(PyObject *, PyObject *const *a, Py_ssize_t n) { return guarded(n, count, [&]() -> PyObject * {
#define BINDING_END Py_RETURN_NONE; }); }

// desc, Q, K, V, key_mask, Z, lse_enc, workspace, stream
BINDING(encode, 9)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *q = c.q(a[1]), *k = c.tok(a[2]), *v = c.tok(a[3]);
    uint8_t *m = c.mask(a[4]);
    float *z = c.z(a[5]), *le = c.le(a[6]);
    const Workspace w(a[7]);
    flare_stream_t st = stream_of(a[8]);
    check_status(unlocked([&] { return lib.encode(c.d, q, k, v, m, z, le, w.p, w.n, st); }), "flare_encode");
BINDING_END

// desc, Q, K, V, key_mask, Z, lse_enc, stream
BINDING(encode_static_scratch, 8)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *q = c.q(a[1]), *k = c.tok(a[2]), *v = c.tok(a[3]);
    uint8_t *m = c.mask(a[4]);
    float *z = c.z(a[5]), *le = c.le(a[6]);
    flare_stream_t st = stream_of(a[7]);
    check_status(unlocked([&] { return lib.encode_static_scratch(c.d, q, k, v, m, z, le, st); }), "flare_encode_static_scratch");
BINDING_END

// desc, Q, K, Z, Y, lse_dec, workspace, stream
BINDING(decode, 8)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *q = c.q(a[1]), *k = c.tok(a[2]);
    float *z = c.z(a[3]);
    void *y = c.tok(a[4]);
    float *ld = c.ld(a[5]);
    const Workspace w(a[6]);
    flare_stream_t st = stream_of(a[7]);
    check_status(unlocked([&] { return lib.decode(c.d, q, k, z, y, ld, w.p, w.n, st); }), "flare_decode");
BINDING_END

// desc, Q, K, V, key_mask, Y, Z, lse_enc, lse_dec, workspace, stream
BINDING(forward, 11)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *q = c.q(a[1]), *k = c.tok(a[2]), *v = c.tok(a[3]);
    uint8_t *m = c.mask(a[4]);
    void *y = c.tok(a[5]);
    float *z = c.z(a[6]), *le = c.le(a[7]), *ld = c.ld(a[8]);
    const Workspace w(a[9]);
    flare_stream_t st = stream_of(a[10]);
    check_status(unlocked([&] { return lib.forward(c.d, q, k, v, m, y, z, le, ld, w.p, w.n, st); }), "flare_forward");
BINDING_END

// desc, Q, K, V, key_mask, Y, dY, Z, lse_enc, lse_dec, dQ, dK, dV, workspace, stream
BINDING(backward, 15)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *q = c.q(a[1]), *k = c.tok(a[2]), *v = c.tok(a[3]);
    uint8_t *m = c.mask(a[4]);
    void *y = c.tok(a[5]), *dy = c.tok(a[6]);
    float *z = c.z(a[7]), *le = c.le(a[8]), *ld = c.ld(a[9]), *dq = c.dq(a[10]);
    void *dk = c.tok(a[11]), *dv = c.tok(a[12]);
    const Workspace w(a[13]);
    flare_stream_t st = stream_of(a[14]);
    check_status(unlocked([&] { return lib.backward(c.d, q, k, v, m, y, dy, z, le, ld, dq, dk, dv, w.p, w.n, st); }), "flare_backward");
BINDING_END

// desc, hQ, hK, hV, hmask, hY, dQ, dK, dV, dmask, dY, workspace, stream
BINDING(forward_host, 13)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *hq = c.q(a[1], false, false), *hk = c.tok(a[2], false), *hv = c.tok(a[3], false);
    uint8_t *hm = c.mask(a[4], false);
    void *hy = c.tok(a[5], false), *q = c.q(a[6]), *k = c.tok(a[7]), *v = c.tok(a[8]);
    uint8_t *m = c.mask(a[9]);
    void *y = c.tok(a[10]);
    const Workspace w(a[11]);
    flare_stream_t st = stream_of(a[12]);
    check_status(unlocked([&] { return lib.forward_host(c.d, hq, hk, hv, hm, hy, q, k, v, m, y, w.p, w.n, st); }), "flare_forward_host");
BINDING_END

// desc, shared, Q_enc, Q_dec, K, V, key_mask, Y, Z, lse_enc, lse_dec, workspace, stream
BINDING(forward_variant, 13)
    Desc desc(a[0]);
    const int shared = PyObject_IsTrue(a[1]);
    const Call c{desc.get(), tensor(a[4]).scalar_type()};
    void *qe = c.q(a[2], shared), *qd = c.q(a[3], shared), *k = c.tok(a[4]), *v = c.tok(a[5]);
    uint8_t *m = c.mask(a[6]);
    void *y = c.tok(a[7]);
    float *z = c.z(a[8]), *le = c.le(a[9]), *ld = c.ld(a[10]);
    const Workspace w(a[11]);
    flare_stream_t st = stream_of(a[12]);
    check_status(unlocked([&] { return lib.forward_variant(c.d, shared, qe, qd, k, v, m, y, z, le, ld, w.p, w.n, st); }), "flare_forward_variant");
BINDING_END

// desc, shared, Q_enc, Q_dec, K, V, key_mask, Y, dY, Z, lse_enc, lse_dec, dQ_enc, dQ_dec, dK, dV, workspace, stream
BINDING(backward_variant, 18)
    Desc desc(a[0]);
    const int shared = PyObject_IsTrue(a[1]);
    const Call c{desc.get(), tensor(a[4]).scalar_type()};
    void *qe = c.q(a[2], shared), *qd = c.q(a[3], shared), *k = c.tok(a[4]), *v = c.tok(a[5]);
    uint8_t *m = c.mask(a[6]);
    void *y = c.tok(a[7]), *dy = c.tok(a[8]);
    float *z = c.z(a[9]), *le = c.le(a[10]), *ld = c.ld(a[11]), *dqe = c.dq(a[12], shared), *dqd = c.dq(a[13], shared);
    void *dk = c.tok(a[14]), *dv = c.tok(a[15]);
    const Workspace w(a[16]);
    flare_stream_t st = stream_of(a[17]);
    check_status(unlocked([&] { return lib.backward_variant(c.d, shared, qe, qd, k, v, m, y, dy, z, le, ld, dqe, dqd, dk, dv, w.p, w.n, st); }),
                 "flare_backward_variant");
BINDING_END

// desc, Q, K, lse_enc, lse_dec, G, workspace, stream
BINDING(spectral_gram, 8)
    Desc desc(a[0]);
    const Call c{desc.get(), tensor(a[2]).scalar_type()};
    void *q = c.q(a[1]), *k = c.tok(a[2]);
    float *le = c.le(a[3]), *ld = c.ld(a[4]);
    float *g = (float *)c.ptr(a[5], at::kFloat, {c.d->B, c.d->H, c.d->M, c.d->M});
    const Workspace w(a[6]);
    flare_stream_t st = stream_of(a[7]);
    check_status(unlocked([&] { return lib.spectral_gram(c.d, q, k, le, ld, g, w.p, w.n, st); }), "flare_spectral_gram");
BINDING_END

// ---- the convenience calls: descriptor from the tensors, outputs and scratch allocated here

flare_desc_t make_desc(const at::Tensor &Q, const at::Tensor &K, double scale) {
    if (Q.dim() != 3 || K.dim() != 4) fail(PyExc_ValueError, "expected Q_lat [H,M,D] and K [B,N,H,D]");
    if (K.size(2) != Q.size(0) || K.size(3) != Q.size(2)) fail(PyExc_ValueError, "Q_lat [H,M,D] and K [B,N,H,D] disagree");
    int dtype;
    switch (K.scalar_type()) {
        case at::kFloat: dtype = FLARE_DTYPE_F32; break;
        case at::kBFloat16: dtype = FLARE_DTYPE_BF16; break;
        case at::kHalf: dtype = FLARE_DTYPE_F16; break;
        default: fail(PyExc_TypeError, "unsupported dtype " + dtype_name(K.scalar_type()));
    }
    return flare_desc_t{(int32_t)K.size(0), (int32_t)K.size(2), (int32_t)K.size(1), (int32_t)Q.size(1), (int32_t)K.size(3), dtype, (float)scale};
}
size_t workspace_bytes(const flare_desc_t &d, int op) {
    const size_t n = lib.workspace_bytes(&d, op);
    if (n == 0) check_status(FLARE_ERR_UNSUPPORTED, "flare_workspace_bytes");
    return n;
}
size_t round256(size_t n) { return (n + 255) & ~(size_t)255; }
// A Python float, or any number that converts to one.
double number(PyObject *o) {
    const double x = PyFloat_AsDouble(o);
    if (x == -1.0 && PyErr_Occurred()) throw PythonError{};
    return x;
}

// Scratch that is dropped when the call returns, with its kernels still queued: allocated on the stream it is used on (none given: the
// current one), so that nothing of another stream takes its place before they have run, or is still at work on it when they start.
at::Tensor scratch(size_t bytes, const at::Tensor &like, PyObject *stream, flare_stream_t st) {
    c10::cuda::OptionalCUDAStreamGuard guard;
    if (stream != Py_None) guard.reset_stream(c10::cuda::getStreamFromExternal((cudaStream_t)st, like.device().index()));
    return at::empty({(int64_t)bytes}, like.options().dtype(at::kByte));
}

// Q, K, V, key_mask, scale, want_stats, stream -> Y, or (Y, Z, lse_enc, lse_dec)
BINDING(call_forward, 7)
    const at::Tensor &Q = tensor(a[0]), &K = tensor(a[1]);
    const flare_desc_t d = make_desc(Q, K, number(a[4]));
    const Call c{&d, K.scalar_type()};
    void *q = c.q(a[0]), *k = c.tok(a[1]), *v = c.tok(a[2]);
    uint8_t *m = c.mask(a[3]);
    const bool stats = PyObject_IsTrue(a[5]) == 1;
    flare_stream_t st = stream_of(a[6]);
    const size_t ws = workspace_bytes(d, FLARE_OP_FORWARD);
    const at::Tensor Y = at::empty({d.B, d.N, d.H, d.D}, K.options());
    const auto f32 = K.options().dtype(at::kFloat);
    if (stats) {
        const at::Tensor Z = at::empty({d.B, d.H, d.M, d.D}, f32), le = at::empty({d.B, d.H, d.M}, f32), ld = at::empty({d.B, d.N, d.H}, f32);
        const at::Tensor w = scratch(ws, K, a[6], st);
        check_status(unlocked([&] { return lib.forward(&d, q, k, v, m, Y.data_ptr(), (float *)Z.data_ptr(), (float *)le.data_ptr(),
                                                       (float *)ld.data_ptr(), w.data_ptr(), ws, st); }), "flare_forward");
        return Py_BuildValue("(NNNN)", THPVariable_Wrap(Y), THPVariable_Wrap(Z), THPVariable_Wrap(le), THPVariable_Wrap(ld));
    }
    // Z lives in the workspace, the statistics (asked for: the encode weights are then as accurate as in training) behind it
    const size_t le_at = round256(ws), ld_at = round256(le_at + 4 * (size_t)d.B * d.H * d.M), total = ld_at + 4 * (size_t)d.B * d.N * d.H;
    const at::Tensor w = scratch(total, K, a[6], st);
    char *base = (char *)w.data_ptr();
    check_status(unlocked([&] { return lib.forward(&d, q, k, v, m, Y.data_ptr(), nullptr, (float *)(base + le_at), (float *)(base + ld_at), base, ws, st); }),
                 "flare_forward");
    return THPVariable_Wrap(Y);
BINDING_END

// Q, K, V, dY, key_mask, scale, stream -> (Y, dQ, dK, dV, workspace: the forward's, and from byte 256 on the backward's)
BINDING(call_forward_backward, 7)
    const at::Tensor &Q = tensor(a[0]), &K = tensor(a[1]);
    const flare_desc_t d = make_desc(Q, K, number(a[5]));
    const Call c{&d, K.scalar_type()};
    void *q = c.q(a[0]), *k = c.tok(a[1]), *v = c.tok(a[2]), *dy = c.tok(a[3]);
    uint8_t *m = c.mask(a[4]);
    flare_stream_t st = stream_of(a[6]);
    // one workspace: the backward starts when the forward is done with it.  But for the header, which keeps what the forward reports: the
    // backward has its own behind it.
    const size_t fwd_bytes = workspace_bytes(d, FLARE_OP_FORWARD), bwd_bytes = workspace_bytes(d, FLARE_OP_BACKWARD), bwd_at = 256;
    const size_t ws = std::max(fwd_bytes, bwd_at + bwd_bytes);
    const at::Tensor Y = at::empty({d.B, d.N, d.H, d.D}, K.options()), dK = at::empty({d.B, d.N, d.H, d.D}, K.options());
    const at::Tensor dV = at::empty({d.B, d.N, d.H, d.D}, K.options()), dQ = at::empty({d.H, d.M, d.D}, K.options().dtype(at::kFloat));
    const size_t z_at = round256(ws), le_at = round256(z_at + 4 * (size_t)d.B * d.H * d.M * d.D), ld_at = round256(le_at + 4 * (size_t)d.B * d.H * d.M);
    const at::Tensor w = scratch(ld_at + 4 * (size_t)d.B * d.N * d.H, K, a[6], st);
    char *base = (char *)w.data_ptr();
    float *z = (float *)(base + z_at), *le = (float *)(base + le_at), *ld = (float *)(base + ld_at);
    check_status(unlocked([&] { return lib.forward(&d, q, k, v, m, Y.data_ptr(), z, le, ld, base, fwd_bytes, st); }), "flare_forward");
    check_status(unlocked([&] { return lib.backward(&d, q, k, v, m, Y.data_ptr(), dy, z, le, ld, (float *)dQ.data_ptr(), dK.data_ptr(), dV.data_ptr(),
                                                    base + bwd_at, bwd_bytes, st); }), "flare_backward");
    return Py_BuildValue("(NNNNN)", THPVariable_Wrap(Y), THPVariable_Wrap(dQ), THPVariable_Wrap(dK), THPVariable_Wrap(dV), THPVariable_Wrap(w));
BINDING_END

// G, eigenvalues, U, sweeps, stream
BINDING(spectral_eig, 5)
    const at::Tensor &G = tensor(a[0]);
    const int64_t M = G.dim() > 0 ? G.size(-1) : 0;
    if (M < 1) fail(PyExc_ValueError, "expected matrices [..., M, M], got shape " + shape_text(G.sizes()));
    // (rows longer than the library takes are left to it to refuse: their square might not even be a number of elements)
    const int64_t matrices = M <= 1024 ? G.numel() / (M * M) : 0;
    const long sweeps = PyLong_AsLong(a[3]);
    if (sweeps == -1 && PyErr_Occurred()) throw PythonError{};
    // (the library is told sizes of G alone: what it writes must have room)
    auto ptr = [](PyObject *o, int64_t least) -> float * {
        if (o == Py_None) return nullptr;
        const at::Tensor &t = tensor(o);
        check(t, at::kFloat, t.sizes());
        if (t.numel() < least) fail(PyExc_ValueError, "expected at least " + std::to_string(least) + " elements, got shape " + shape_text(t.sizes()));
        return (float *)t.data_ptr();
    };
    float *g = ptr(a[0], 0), *ev = ptr(a[1], matrices * M), *u = ptr(a[2], matrices * M * M);
    flare_stream_t st = stream_of(a[4]);
    check_status(unlocked([&] { return lib.spectral_eig((int32_t)matrices, (int32_t)M, g, ev, u, (int32_t)sweeps, st); }), "flare_spectral_eig");
BINDING_END

// bind(addresses: dict name -> int, FlareError)
BINDING(bind, 2)
    auto get = [&](const char *name, auto &slot) {
        PyObject *o = PyDict_GetItemString(a[0], name);
        if (!o) fail(PyExc_KeyError, name);
        slot = (std::remove_reference_t<decltype(slot)>)PyLong_AsVoidPtr(o);
    };
    get("flare_workspace_bytes", lib.workspace_bytes);
    get("flare_encode", lib.encode);
    get("flare_encode_static_scratch", lib.encode_static_scratch);
    get("flare_decode", lib.decode);
    get("flare_forward", lib.forward);
    get("flare_backward", lib.backward);
    get("flare_forward_host", lib.forward_host);
    get("flare_forward_variant", lib.forward_variant);
    get("flare_backward_variant", lib.backward_variant);
    get("flare_spectral_gram", lib.spectral_gram);
    get("flare_spectral_eig", lib.spectral_eig);
    Py_INCREF(a[1]);
    flare_error = a[1];
BINDING_END

#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(bind), METHOD(encode), METHOD(encode_static_scratch), METHOD(decode), METHOD(forward), METHOD(backward),
                         METHOD(forward_host), METHOD(forward_variant), METHOD(backward_variant), METHOD(spectral_gram), METHOD(spectral_eig),
                         METHOD(call_forward), METHOD(call_forward_backward), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_binding", "Argument marshalling for libflare.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module_def); }
