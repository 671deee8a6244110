// Argument marshalling between torch tensors and the C ABI (include/hgrn2.h), in C++.
//
// A call's host side - reading shapes and pointers off the tensors, allocating what was not passed in, asking for the
// current stream - took 9 of the 11 us of a one-token decode call when it was written in Python on ctypes (the
// kernel needs 3); here it takes about 1.  Nothing is computed: every function fills a descriptor, calls the
// library and hands the buffers back.  binding.py documents the functions and their defaults.
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "hgrn2.h"

namespace {

PyObject *g_desc_type = nullptr, *g_error_type = nullptr;   // binding.Desc, binding.Hgrn2Error

struct PyError {};                                           // a Python exception is set

[[noreturn]] void raise(PyObject *type, const char *text)
{
    PyErr_SetString(type, text);
    throw PyError{};
}

void check(hgrn2_status code, const char *what)
{
    if (code == HGRN2_OK) return;
    PyObject *e = PyObject_CallFunction(g_error_type, "is", (int)code, what);
    if (e) {
        PyErr_SetObject(g_error_type, e);
        Py_DECREF(e);
    }
    throw PyError{};
}

bool given(PyObject *x) { return x != Py_None; }

const at::Tensor &tensor(PyObject *x)
{
    if (!THPVariable_Check(x)) raise(PyExc_TypeError, "expected a torch tensor");
    return THPVariable_Unpack(x);
}

void *ptr(const at::Tensor &t)
{
    if (!t.is_cuda()) raise(PyExc_ValueError, "the library takes device pointers: tensor is not on a CUDA device");
    if (!t.is_contiguous()) raise(PyExc_ValueError, "tensors must be contiguous");
    return t.data_ptr();
}
void *ptr(PyObject *x) { return given(x) ? ptr(tensor(x)) : nullptr; }

int32_t io_code(const at::Tensor &t)
{
    if (t.scalar_type() == at::kFloat) return HGRN2_F32;
    if (t.scalar_type() == at::kBFloat16) return HGRN2_BF16;
    PyErr_Format(PyExc_TypeError, "unsupported I/O dtype %s", c10::toString(t.scalar_type()));
    throw PyError{};
}

// Whatever int() takes, cut to 32 bits, as a ctypes field does.
uint32_t bits(PyObject *x)
{
    PyObject *n = PyNumber_Long(x);
    if (!n) throw PyError{};
    const unsigned long v = PyLong_AsUnsignedLongMask(n);
    Py_DECREF(n);
    if (v == (unsigned long)-1 && PyErr_Occurred()) throw PyError{};
    return (uint32_t)v;
}
long integer(PyObject *x) { return (int32_t)bits(x); }
bool truth(PyObject *x)
{
    const int v = PyObject_IsTrue(x);
    if (v < 0) throw PyError{};
    return v != 0;
}

// stream: None = the current stream of the current device, else the handle as an integer
void *stream_of(PyObject *x)
{
    if (!given(x)) return c10::cuda::getCurrentCUDAStream().stream();
    void *s = PyLong_AsVoidPtr(x);
    if (s == nullptr && PyErr_Occurred()) throw PyError{};
    return s;
}

// A buffer that the caller may have passed in.
struct Buffer {
    PyObject *passed;
    at::Tensor made;
    void *p = nullptr;
    Buffer(PyObject *x) : passed(x) { p = ptr(x); }
    bool missing() const { return !given(passed); }
    void make(at::IntArrayRef shape, at::ScalarType type, const at::Tensor &like)
    {
        made = at::empty(shape, at::TensorOptions().dtype(type).device(like.device()));
        p = made.data_ptr();
    }
    PyObject *give() const                                    // new reference
    {
        if (made.defined()) return THPVariable_Wrap(made);
        Py_INCREF(passed);
        return passed;
    }
};

PyObject *pack(std::initializer_list<const Buffer *> bufs, const hgrn2_desc *d)
{
    PyObject *out = PyTuple_New(bufs.size() + (d ? 1 : 0));
    if (!out) throw PyError{};
    Py_ssize_t n = 0;
    for (const Buffer *b : bufs) {
        PyObject *x = b->give();
        if (!x) { Py_DECREF(out); throw PyError{}; }
        PyTuple_SET_ITEM(out, n++, x);
    }
    if (d) {
        PyObject *x = PyObject_CallFunction(g_desc_type, "iiiiiiiI", d->B, d->H, d->N, d->dk, d->dv, d->io, d->chunk, d->flags);
        if (!x) { Py_DECREF(out); throw PyError{}; }
        PyTuple_SET_ITEM(out, n, x);
    }
    return out;
}

enum Kind { kPlain = 0, kPacked = 1, kGated = 2 };

// Sizes of a sequence call: o [B, H, N, dk] (packed: [H, T, dk] and B from the offsets), i [.., dv].
struct Shape {
    hgrn2_desc d;
    int64_t dims[4];
    int nd;
    at::IntArrayRef seq(int64_t width)
    {
        dims[nd - 1] = width;
        return at::IntArrayRef(dims, nd);
    }
};
Shape sequence_shape(long kind, const at::Tensor &o, const at::Tensor &i, PyObject *extra, PyObject *chunk, PyObject *flags)
{
    Shape s;
    s.nd = kind == kPacked ? 3 : 4;
    if (o.dim() != s.nd || i.dim() < 1)
        raise(PyExc_ValueError, kind == kPacked ? "expected tensors of shape [H, T, d]" : "expected tensors of shape [B, H, N, d]");
    for (int k = 0; k < s.nd; ++k) s.dims[k] = o.size(k);
    int64_t B = s.dims[0], H = s.dims[1], N = s.dims[2];
    if (kind == kPacked) {
        const at::Tensor &cu = tensor(extra);
        if (cu.scalar_type() != at::kInt) raise(PyExc_TypeError, "cu_seqlens must be int32");
        B = cu.numel() - 1; H = s.dims[0]; N = s.dims[1];
    }
    s.d = hgrn2_desc{(int32_t)B, (int32_t)H, (int32_t)N, (int32_t)o.size(-1), (int32_t)i.size(-1), io_code(o),
                     (int32_t)integer(chunk), bits(flags)};
    return s;
}

size_t saved_bytes(long kind, const hgrn2_desc *d)
{
    return kind == kPlain ? hgrn2_saved_bytes(d) : kind == kPacked ? hgrn2_saved_bytes_varlen(d) : hgrn2_saved_bytes_gated(d);
}
void make_workspace(Buffer &ws, long kind, const hgrn2_desc *d, const at::Tensor &like)
{
    const size_t n = kind == kPlain ? hgrn2_workspace_bytes(d)
                     : kind == kPacked ? hgrn2_workspace_bytes_varlen(d) : hgrn2_workspace_bytes_gated(d);
    if (n == 0 && kind == kPlain) check(HGRN2_ERR_UNSUPPORTED, "hgrn2_workspace_bytes");
    ws.make({(int64_t)n}, at::kByte, like);
}

template <typename F> PyObject *guarded(F f)
{
    HANDLE_TH_ERRORS
    try {
        return f();
    } catch (const PyError &) {
        return nullptr;
    }
    END_HANDLE_TH_ERRORS
}

bool arity(Py_ssize_t n, Py_ssize_t want)
{
    if (n != want) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return n == want;
}

// The library call itself runs without the interpreter lock, as a ctypes call does.
template <typename F> hgrn2_status unlocked(F f)
{
    PyThreadState *t = PyEval_SaveThread();
    const hgrn2_status s = f();
    PyEval_RestoreThread(t);
    return s;
}

// step(o, f, i, S, y, stream, several) -> y
PyObject *step(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 7)) return nullptr;
    return guarded([&]() -> PyObject * {
        const at::Tensor &o = tensor(a[0]), &i = tensor(a[2]);
        const bool several = truth(a[6]);
        const int nd = several ? 4 : 3;
        if (o.dim() != nd || i.dim() < 1)
            raise(PyExc_ValueError, several ? "expected tensors of shape [B, H, T, d]" : "expected tensors of shape [B, H, d]");
        const int64_t dv = i.size(-1);
        hgrn2_desc d{(int32_t)o.size(0), (int32_t)o.size(1), several ? (int32_t)o.size(2) : 1, (int32_t)o.size(-1), (int32_t)dv,
                     io_code(o), 0, 0};
        Buffer y(a[4]);
        if (y.missing()) {
            if (several) y.make({d.B, d.H, d.N, dv}, o.scalar_type(), o);
            else y.make({d.B, d.H, dv}, o.scalar_type(), o);
        }
        void *po = ptr(o), *pf = ptr(a[1]), *pi = ptr(i), *pS = ptr(a[3]), *st = stream_of(a[5]);
        check(unlocked([&] {
            return several ? hgrn2_step_multi(&d, po, pf, pi, static_cast<float *>(pS), y.p, st)
                           : hgrn2_step(&d, po, pf, pi, static_cast<float *>(pS), y.p, st);
        }), several ? "hgrn2_step_multi" : "hgrn2_step");
        return y.give();
    });
}

// fwd(kind, o, f, i, extra, S0, y, SN, saved, ws, want_final_state, save_for_backward, chunk, flags, stream)
//   -> (y, SN, saved, ws, desc);  extra: cu_seqlens (packed) or beta (gated)
PyObject *fwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 15)) return nullptr;
    return guarded([&]() -> PyObject * {
        const long kind = integer(a[0]);
        const at::Tensor &o = tensor(a[1]), &i = tensor(a[3]);
        Shape s = sequence_shape(kind, o, i, a[4], a[12], a[13]);
        const hgrn2_desc &d = s.d;
        Buffer y(a[6]), SN(a[7]), saved(a[8]), ws(a[9]);
        if (y.missing()) y.make(s.seq(d.dv), o.scalar_type(), o);
        if (SN.missing() && truth(a[10])) SN.make({d.B, d.H, d.dk, d.dv}, at::kFloat, o);
        if (saved.missing() && truth(a[11])) saved.make({std::max<int64_t>((int64_t)saved_bytes(kind, &d), 16)}, at::kByte, o);
        if (ws.missing()) make_workspace(ws, kind, &d, o);
        void *po = ptr(o), *pf = ptr(a[2]), *pi = ptr(i), *px = ptr(a[4]), *pS0 = ptr(a[5]), *st = stream_of(a[14]);
        const float *S0 = static_cast<const float *>(pS0);
        float *pSN = static_cast<float *>(SN.p);
        check(unlocked([&] {
            return kind == kPlain    ? hgrn2_fwd(&d, po, pf, pi, S0, y.p, pSN, saved.p, ws.p, st)
                   : kind == kPacked ? hgrn2_fwd_varlen(&d, po, pf, pi, static_cast<const int32_t *>(px), S0, y.p, pSN, saved.p, ws.p, st)
                                     : hgrn2_fwd_gated(&d, po, pf, pi, static_cast<const float *>(px), S0, y.p, pSN, saved.p, ws.p, st);
        }), kind == kPlain ? "hgrn2_fwd" : kind == kPacked ? "hgrn2_fwd_varlen" : "hgrn2_fwd_gated");
        return pack({&y, &SN, &saved, &ws}, &d);
    });
}

// bwd(kind, o, f, i, extra, S0, dy, dSN, saved, d_o, d_f, d_i, d_beta, dS0, ws, want_dS0, want_d_beta, chunk, flags, stream)
//   -> (d_o, d_f, d_i, [d_beta,] dS0, ws)
PyObject *bwd(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 20)) return nullptr;
    return guarded([&]() -> PyObject * {
        const long kind = integer(a[0]);
        const at::Tensor &o = tensor(a[1]), &i = tensor(a[3]);
        Shape s = sequence_shape(kind, o, i, a[4], a[17], a[18]);
        const hgrn2_desc &d = s.d;
        Buffer d_o(a[9]), d_f(a[10]), d_i(a[11]), d_beta(a[12]), dS0(a[13]), ws(a[14]);
        if (d_o.missing()) d_o.make(o.sizes(), o.scalar_type(), o);
        if (d_f.missing()) {
            const at::Tensor &f = tensor(a[2]);
            d_f.make(f.sizes(), f.scalar_type(), f);
        }
        if (d_i.missing()) d_i.make(i.sizes(), i.scalar_type(), i);
        if (kind == kGated && d_beta.missing() && truth(a[16])) d_beta.make({d.H, d.dk}, at::kFloat, o);
        if (dS0.missing() && truth(a[15])) dS0.make({d.B, d.H, d.dk, d.dv}, at::kFloat, o);
        if (ws.missing()) make_workspace(ws, kind, &d, o);
        void *po = ptr(o), *pf = ptr(a[2]), *pi = ptr(i), *px = ptr(a[4]), *pS0 = ptr(a[5]), *pdy = ptr(a[6]), *pdSN = ptr(a[7]),
             *psaved = ptr(a[8]), *st = stream_of(a[19]);
        const float *S0 = static_cast<const float *>(pS0), *dSN = static_cast<const float *>(pdSN);
        float *pdS0 = static_cast<float *>(dS0.p);
        check(unlocked([&] {
            return kind == kPlain ? hgrn2_bwd(&d, po, pf, pi, S0, pdy, dSN, psaved, d_o.p, d_f.p, d_i.p, pdS0, ws.p, st)
                   : kind == kPacked
                       ? hgrn2_bwd_varlen(&d, po, pf, pi, static_cast<const int32_t *>(px), S0, pdy, dSN, psaved, d_o.p, d_f.p,
                                          d_i.p, pdS0, ws.p, st)
                       : hgrn2_bwd_gated(&d, po, pf, pi, static_cast<const float *>(px), S0, pdy, dSN, psaved, d_o.p, d_f.p,
                                         d_i.p, static_cast<float *>(d_beta.p), pdS0, ws.p, st);
        }), kind == kPlain ? "hgrn2_bwd" : kind == kPacked ? "hgrn2_bwd_varlen" : "hgrn2_bwd_gated");
        return kind == kGated ? pack({&d_o, &d_f, &d_i, &d_beta, &dS0, &ws}, nullptr) : pack({&d_o, &d_f, &d_i, &dS0, &ws}, nullptr);
    });
}

// setup(Desc, Hgrn2Error): the Python types that results and errors are made of
PyObject *setup(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    if (!arity(n, 2)) return nullptr;
    Py_INCREF(a[0]);
    Py_INCREF(a[1]);
    Py_XSETREF(g_desc_type, a[0]);
    Py_XSETREF(g_error_type, a[1]);
    Py_RETURN_NONE;
}

PyMethodDef g_methods[] = {
    {"step", (PyCFunction)(void (*)(void))step, METH_FASTCALL, nullptr},
    {"fwd", (PyCFunction)(void (*)(void))fwd, METH_FASTCALL, nullptr},
    {"bwd", (PyCFunction)(void (*)(void))bwd, METH_FASTCALL, nullptr},
    {"setup", (PyCFunction)(void (*)(void))setup, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&g_module); }
