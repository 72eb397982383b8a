// Native half of the Python binding (hc.py): takes the tensors of a call,
// checks them, and calls libhc. A call through ctypes spent 11 us of host time
// on reading tensor attributes one Python call at a time and on converting
// them; see hc.py for what each function takes. Every function returns the
// hc_status as an int, or raises ValueError / TypeError where an argument is
// not one that the binding passes on. No tensor or pointer outlives its call.
//
// The module is not linked to libhc: bind() takes the handle of the library
// that hc.load_library() opened, and every call goes there. The library's
// error string and device status are its own, so a call into another copy of
// it would lose them.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include "hc.h"

namespace {

// clang-format off
#define HC_CALLS(X) \
    X(hc_mask_compact) X(hc_mask_compact_static) X(hc_sparse_spiral_conv_fwd) \
    X(hc_conv_rulebook) X(hc_mask_compact_rulebook) X(hc_sparse_conv_rulebook_fwd) \
    X(hc_sparse_conv_rulebook_fwd_hint) X(hc_sparse_linear_fwd) X(hc_sparse_group_norm_fwd) \
    X(hc_sparse_conv_gn_fwd) X(hc_conv_rulebook_transpose) X(hc_sparse_conv_rulebook_bwd) \
    X(hc_mask_score_update) X(hc_mask_select_topk) X(hc_kappa_masks) X(hc_gather_rows) \
    X(hc_scatter_dense) X(hc_spiral_conv_fwd)
// clang-format on

struct Library {
#define MEMBER(f) decltype(&::f) f;
    HC_CALLS(MEMBER)
#undef MEMBER
};
Library lib;  // by bind()
bool bound = false;

struct PyError {};  // a Python exception is set

[[noreturn]] void raise(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    throw PyError{};
}

const at::Tensor* tensor_or_none(PyObject* o) {
    if (o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) raise(PyExc_TypeError, "libhc takes torch tensors");
    return &THPVariable_Unpack(o);
}
const at::Tensor& tensor(PyObject* o) {
    const at::Tensor* t = tensor_or_none(o);
    if (!t) raise(PyExc_TypeError, "libhc: a tensor is required, not None");
    return *t;
}

// Device address of a contiguous device tensor (nullptr for None).
void* dev(const at::Tensor* t, bool pinned_ok = false) {
    if (!t) return nullptr;
    if (!t->is_cuda() && !(pinned_ok && t->is_pinned()))
        raise(PyExc_ValueError, "libhc takes device tensors");
    if (!t->is_contiguous()) raise(PyExc_ValueError, "libhc takes contiguous tensors");
    return t->data_ptr();
}
template <typename T = void>
T* ptr(PyObject* o, bool pinned_ok = false) {
    return static_cast<T*>(dev(tensor_or_none(o), pinned_ok));
}

hc_dtype dtype(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return HC_F32;
    if (t.scalar_type() == at::kBFloat16) return HC_BF16;
    raise(PyExc_TypeError, "unsupported dtype");
}

int size(const at::Tensor& t, int64_t dims, int64_t i) {
    if (t.dim() != dims) raise(PyExc_ValueError, "libhc: a tensor has another number of dimensions");
    return (int)t.size(i);
}
int dim(const at::Tensor& t, int64_t i) {
    if (t.dim() <= i) raise(PyExc_IndexError, "libhc: a tensor has too few dimensions");
    return (int)t.size(i);
}
int last(const at::Tensor& t) {
    if (t.dim() < 1) raise(PyExc_ValueError, "libhc: a tensor has no dimensions");
    return (int)t.size(-1);
}
int rows(const at::Tensor& t) {  // of width last(t)
    const int c = last(t);
    if (c == 0) raise(PyExc_ZeroDivisionError, "libhc: rows of no channels");
    return (int)(t.numel() / c);
}

int integer(PyObject* o) {
    const long v = PyLong_AsLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyError{};
    return (int)v;
}
long long integer64(PyObject* o) {
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) throw PyError{};
    return v;
}
float real(PyObject* o) {
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) throw PyError{};
    return (float)v;
}

// None: torch's current stream; else an object with .cuda_stream, or an int.
hc_stream_t stream(PyObject* o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    PyObject* v = PyObject_GetAttrString(o, "cuda_stream");
    if (!v) {
        PyErr_Clear();
        v = PyNumber_Long(o);
        if (!v) throw PyError{};
    }
    const unsigned long long s = PyLong_AsUnsignedLongLong(v);
    Py_DECREF(v);
    if (PyErr_Occurred()) throw PyError{};
    return reinterpret_cast<hc_stream_t>(s);
}

template <int N, class F>
PyObject* entry(PyObject* const* a, Py_ssize_t n, F&& f) {
    if (n != N) {
        PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
        return nullptr;
    }
    if (!bound) {
        PyErr_SetString(PyExc_RuntimeError, "libhc is not bound");
        return nullptr;
    }
    try {
        return PyLong_FromLong(f(a));
    } catch (const PyError&) {
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
    } catch (...) {
        PyErr_SetString(PyExc_RuntimeError, "libhc binding: unknown error");
    }
    return nullptr;
}
// The library call itself, without the interpreter's lock.
template <class F>
int unlocked(F&& f) {
    PyThreadState* st = PyEval_SaveThread();
    const int r = f();
    PyEval_RestoreThread(st);
    return r;
}

using I32 = int32_t;
#define FN(name) PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs)

template <hc_status (*Library::*F)(const uint8_t*, int, int, I32*, I32*, I32*, I32*, hc_stream_t)>
FN(compact) {  // mask, coords, row_of, batch_offsets, count, stream
    return entry<6>(args, nargs, [](PyObject* const* a) {
        const at::Tensor& m = tensor(a[0]);
        const int B = size(m, 2, 0), V = size(m, 2, 1);
        const auto* mask = static_cast<const uint8_t*>(dev(&m));
        I32 *c = ptr<I32>(a[1]), *r = ptr<I32>(a[2]), *o = ptr<I32>(a[3]), *n = ptr<I32>(a[4]);
        const hc_stream_t s = stream(a[5]);
        return unlocked([&] { return (lib.*F)(mask, B, V, c, r, o, n, s); });
    });
}

// x, x_layout, coords, row_of, count, spiral, B, V, W, bias, act, y, stream
FN(sparse_spiral_conv_fwd) {
    return entry<13>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &sp = tensor(a[5]), &W = tensor(a[8]);
        const int L = dim(sp, 1), ci = last(x), co = dim(W, 1);
        const hc_dtype dt = dtype(x);
        const int layout = integer(a[1]), B = integer(a[6]), V = integer(a[7]), act = integer(a[10]);
        void *xp = dev(&x), *Wp = dev(&W), *y = ptr(a[11]);
        I32 *c = ptr<I32>(a[2]), *r = ptr<I32>(a[3]), *n = ptr<I32>(a[4]);
        const auto* spp = static_cast<I32*>(dev(&sp));
        const float* b = ptr<float>(a[9]);
        const hc_stream_t s = stream(a[12]);
        return unlocked([&] {
            return lib.hc_sparse_spiral_conv_fwd(xp, (hc_layout)layout, dt, c, r, n, spp, B, V, L, ci, co,
                                             Wp, b, (hc_act)act, y, s);
        });
    });
}

FN(conv_rulebook) {  // coords, row_of, count, spiral, B, V, x_layout, rulebook, stream
    return entry<9>(args, nargs, [](PyObject* const* a) {
        const at::Tensor& sp = tensor(a[3]);
        const int L = dim(sp, 1), B = integer(a[4]), V = integer(a[5]), layout = integer(a[6]);
        I32 *c = ptr<I32>(a[0]), *r = ptr<I32>(a[1]), *n = ptr<I32>(a[2]), *rb = ptr<I32>(a[7]);
        const auto* spp = static_cast<I32*>(dev(&sp));
        const hc_stream_t s = stream(a[8]);
        return unlocked([&] {
            return lib.hc_conv_rulebook(c, r, n, spp, B, V, L, (hc_layout)layout, rb, s);
        });
    });
}

// mask, spiral, x_layout, coords, row_of, batch_offsets, count, rulebook, stream
FN(mask_compact_rulebook) {
    return entry<9>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &m = tensor(a[0]), &sp = tensor(a[1]);
        const int B = size(m, 2, 0), V = size(m, 2, 1), L = dim(sp, 1), layout = integer(a[2]);
        const auto* mask = static_cast<const uint8_t*>(dev(&m));
        const auto* spp = static_cast<I32*>(dev(&sp));
        I32 *c = ptr<I32>(a[3]), *r = ptr<I32>(a[4]), *o = ptr<I32>(a[5]), *n = ptr<I32>(a[6]),
            *rb = ptr<I32>(a[7]);
        const hc_stream_t s = stream(a[8]);
        return unlocked([&] {
            return lib.hc_mask_compact_rulebook(mask, B, V, spp, L, (hc_layout)layout, c, r, o, n, rb, s);
        });
    });
}

// x, rulebook, count, W, bias, act, y, rows_hint (None: the call without a
// row estimate), coords, out, stream
FN(sparse_conv_rulebook_fwd) {
    return entry<11>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &rb = tensor(a[1]), &W = tensor(a[3]);
        const at::Tensor *y = tensor_or_none(a[6]), *out = tensor_or_none(a[9]);
        const int L = size(rb, 2, 0), cap = size(rb, 2, 1), ci = last(x), xr = rows(x),
                  co = dim(W, 1), act = integer(a[5]);
        const int B = out ? dim(*out, 0) : 0, V = out ? dim(*out, 1) : 0;
        const hc_dtype dt = dtype(y ? *y : x);
        void *xp = dev(&x), *Wp = dev(&W), *yp = dev(y), *op = dev(out);
        const auto* rbp = static_cast<I32*>(dev(&rb));
        I32 *n = ptr<I32>(a[2]), *c = ptr<I32>(a[8]);
        const float* b = ptr<float>(a[4]);
        const bool hinted = a[7] != Py_None;
        const long long hint = hinted ? integer64(a[7]) : 0;
        const hc_stream_t s = stream(a[10]);
        return unlocked([&] {
            return hinted ? lib.hc_sparse_conv_rulebook_fwd_hint(xp, dt, xr, rbp, n, cap, L, ci, co, Wp, b,
                                                             (hc_act)act, yp, c, B, V, op, hint, s)
                          : lib.hc_sparse_conv_rulebook_fwd(xp, dt, xr, rbp, n, cap, L, ci, co, Wp, b,
                                                        (hc_act)act, yp, c, B, V, op, s);
        });
    });
}

FN(sparse_linear_fwd) {  // x, count, W, bias, act, y, stream
    return entry<7>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &W = tensor(a[2]);
        const int cap = size(x, 2, 0), ci = size(x, 2, 1), co = dim(W, 1), act = integer(a[4]);
        const hc_dtype dt = dtype(x);
        void *xp = dev(&x), *Wp = dev(&W), *y = ptr(a[5]);
        const I32* n = ptr<I32>(a[1]);
        const float* b = ptr<float>(a[3]);
        const hc_stream_t s = stream(a[6]);
        return unlocked([&] {
            return lib.hc_sparse_linear_fwd(xp, dt, n, cap, ci, co, Wp, b, (hc_act)act, y, s);
        });
    });
}

FN(sparse_group_norm_fwd) {  // x, batch_offsets, G, eps, gamma, beta, act, y, stream
    return entry<9>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &o = tensor(a[1]);
        const int cap = size(x, 2, 0), C = size(x, 2, 1), B = dim(o, 0) - 1, G = integer(a[2]),
                  act = integer(a[6]);
        const float eps = real(a[3]);
        const hc_dtype dt = dtype(x);
        void *xp = dev(&x), *y = ptr(a[7]);
        const auto* op = static_cast<I32*>(dev(&o));
        const float *ga = ptr<float>(a[4]), *be = ptr<float>(a[5]);
        const hc_stream_t s = stream(a[8]);
        return unlocked([&] {
            return lib.hc_sparse_group_norm_fwd(xp, dt, op, B, cap, C, G, eps, ga, be, (hc_act)act, y, s);
        });
    });
}

// x, rulebook, count, W, bias, coords, batch_offsets, G, eps, gamma, beta, act, y, stream
FN(sparse_conv_gn_fwd) {
    return entry<14>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &rb = tensor(a[1]), &W = tensor(a[3]), &o = tensor(a[6]),
                         &y = tensor(a[12]);
        const int L = size(rb, 2, 0), cap = size(rb, 2, 1), ci = last(x), xr = rows(x),
                  co = dim(W, 1), B = dim(o, 0) - 1, G = integer(a[7]), act = integer(a[11]);
        const float eps = real(a[8]);
        const hc_dtype dt = dtype(y);
        void *xp = dev(&x), *Wp = dev(&W), *yp = dev(&y);
        const auto* rbp = static_cast<I32*>(dev(&rb));
        const auto* op = static_cast<I32*>(dev(&o));
        const I32 *n = ptr<I32>(a[2]), *c = ptr<I32>(a[5]);
        const float *b = ptr<float>(a[4]), *ga = ptr<float>(a[9]), *be = ptr<float>(a[10]);
        const hc_stream_t s = stream(a[13]);
        return unlocked([&] {
            return lib.hc_sparse_conv_gn_fwd(xp, dt, xr, rbp, n, cap, L, ci, co, Wp, b, c, op, B, G, eps, ga,
                                         be, (hc_act)act, yp, s);
        });
    });
}

FN(conv_rulebook_transpose) {  // rulebook, count, x_rows, row_ptr, taps, stream
    return entry<6>(args, nargs, [](PyObject* const* a) {
        const at::Tensor& rb = tensor(a[0]);
        const int L = size(rb, 2, 0), cap = size(rb, 2, 1), xr = integer(a[2]);
        const auto* rbp = static_cast<I32*>(dev(&rb));
        const I32* n = ptr<I32>(a[1]);
        I32 *p = ptr<I32>(a[3]), *t = ptr<I32>(a[4]);
        const hc_stream_t s = stream(a[5]);
        return unlocked([&] { return lib.hc_conv_rulebook_transpose(rbp, n, cap, L, xr, p, t, s); });
    });
}

// x, rulebook, count, W, y, dy, act, row_ptr, taps, dx, dW, dbias, stream
FN(sparse_conv_rulebook_bwd) {
    return entry<13>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &rb = tensor(a[1]), &W = tensor(a[3]);
        const int L = size(rb, 2, 0), cap = size(rb, 2, 1), ci = last(x), xr = rows(x),
                  co = dim(W, 1), act = integer(a[6]);
        const hc_dtype dt = dtype(x);
        void *xp = dev(&x), *Wp = dev(&W), *y = ptr(a[4]), *dy = ptr(a[5]), *dx = ptr(a[9]);
        const auto* rbp = static_cast<I32*>(dev(&rb));
        const I32 *n = ptr<I32>(a[2]), *p = ptr<I32>(a[7]), *t = ptr<I32>(a[8]);
        float *dW = ptr<float>(a[10]), *db = ptr<float>(a[11]);
        const hc_stream_t s = stream(a[12]);
        return unlocked([&] {
            return lib.hc_sparse_conv_rulebook_bwd(xp, dt, xr, rbp, n, cap, L, ci, co, Wp, y, dy,
                                               (hc_act)act, p, t, dx, dW, db, s);
        });
    });
}

FN(mask_score_update) {  // O, alpha_in, alpha_out, sim, stream
    return entry<5>(args, nargs, [](PyObject* const* a) {
        const at::Tensor& O = tensor(a[0]);
        const int K = size(O, 3, 0), N = size(O, 3, 1), D = size(O, 3, 2);
        const hc_dtype dt = dtype(O);
        void* Op = dev(&O);
        const float* ai = ptr<float>(a[1]);
        float *ao = ptr<float>(a[2]), *sim = ptr<float>(a[3]);
        const hc_stream_t s = stream(a[4]);
        return unlocked([&] { return lib.hc_mask_score_update(Op, dt, K, N, D, ai, ao, sim, s); });
    });
}

FN(mask_select_topk) {  // alpha, kappa, selected, stream
    return entry<4>(args, nargs, [](PyObject* const* a) {
        const at::Tensor& al = tensor(a[0]);
        const int K = dim(al, 0), kappa = integer(a[1]);
        const auto* ap = static_cast<float*>(dev(&al));
        I32* sel = ptr<I32>(a[2]);
        const hc_stream_t s = stream(a[3]);
        return unlocked([&] { return lib.hc_mask_select_topk(ap, K, kappa, sel, s); });
    });
}

FN(kappa_masks) {  // masks, selected, B, out, stream
    return entry<5>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &m = tensor(a[0]), &sel = tensor(a[1]);
        const int K = size(m, 2, 0), V = size(m, 2, 1), kappa = dim(sel, 0), B = integer(a[2]);
        const auto* mp = static_cast<uint8_t*>(dev(&m));
        const auto* sp = static_cast<I32*>(dev(&sel));
        uint8_t* out = ptr<uint8_t>(a[3]);
        const hc_stream_t s = stream(a[4]);
        return unlocked([&] { return lib.hc_kappa_masks(mp, K, V, sp, kappa, B, out, s); });
    });
}

FN(gather_rows) {  // x, coords, count, frames_per_sample, y, stream
    return entry<6>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &y = tensor(a[4]);
        const int B = size(x, 3, 0), V = size(x, 3, 1), C = size(x, 3, 2), fps = integer(a[3]);
        const int cap = dim(y, 0);
        const hc_dtype dt = dtype(x);
        void *xp = dev(&x, true), *yp = dev(&y, true);
        const I32 *c = ptr<I32>(a[1]), *n = ptr<I32>(a[2]);
        const hc_stream_t s = stream(a[5]);
        return unlocked([&] { return lib.hc_gather_rows(xp, dt, B, V, C, c, n, cap, fps, yp, s); });
    });
}

FN(scatter_dense) {  // y, coords, row_of, count, B, V, zero_fill, out, stream
    return entry<9>(args, nargs, [](PyObject* const* a) {
        const at::Tensor& y = tensor(a[0]);
        const int C = last(y), B = integer(a[4]), V = integer(a[5]), zf = integer(a[6]);
        const hc_dtype dt = dtype(y);
        void *yp = dev(&y), *out = ptr(a[7]);
        const I32 *c = ptr<I32>(a[1]), *r = ptr<I32>(a[2]), *n = ptr<I32>(a[3]);
        const hc_stream_t s = stream(a[8]);
        return unlocked([&] { return lib.hc_scatter_dense(yp, dt, c, r, n, B, V, C, zf, out, s); });
    });
}

FN(spiral_conv_fwd) {  // x, spiral, W, bias, act, y, stream
    return entry<7>(args, nargs, [](PyObject* const* a) {
        const at::Tensor &x = tensor(a[0]), &sp = tensor(a[1]), &W = tensor(a[2]);
        const int B = size(x, 3, 0), V = size(x, 3, 1), ci = size(x, 3, 2), L = dim(sp, 1),
                  co = dim(W, 1), act = integer(a[4]);
        const hc_dtype dt = dtype(x);
        void *xp = dev(&x), *Wp = dev(&W), *y = ptr(a[5]);
        const auto* spp = static_cast<I32*>(dev(&sp));
        const float* b = ptr<float>(a[3]);
        const hc_stream_t s = stream(a[6]);
        return unlocked([&] {
            return lib.hc_spiral_conv_fwd(xp, dt, spp, B, V, L, ci, co, Wp, b, (hc_act)act, y, s);
        });
    });
}

#define METHOD(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, nullptr}

PyObject* bind(PyObject*, PyObject* arg) {  // the dlopen handle of libhc, as an int
    void* handle = PyLong_AsVoidPtr(arg);
    if (!handle) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "no library handle");
        return nullptr;
    }
    Library l;
#define LOOK_UP(f)                                                              \
    l.f = reinterpret_cast<decltype(l.f)>(dlsym(handle, #f));                   \
    if (!l.f) {                                                                 \
        PyErr_SetString(PyExc_RuntimeError, "the library does not have " #f);   \
        return nullptr;                                                         \
    }
    HC_CALLS(LOOK_UP)
#undef LOOK_UP
    lib = l;
    bound = true;
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_O, nullptr},
    METHOD("hc_mask_compact", compact<&Library::hc_mask_compact>),
    METHOD("hc_mask_compact_static", compact<&Library::hc_mask_compact_static>),
    METHOD("hc_sparse_spiral_conv_fwd", sparse_spiral_conv_fwd),
    METHOD("hc_conv_rulebook", conv_rulebook),
    METHOD("hc_mask_compact_rulebook", mask_compact_rulebook),
    METHOD("hc_sparse_conv_rulebook_fwd", sparse_conv_rulebook_fwd),
    METHOD("hc_sparse_linear_fwd", sparse_linear_fwd),
    METHOD("hc_sparse_group_norm_fwd", sparse_group_norm_fwd),
    METHOD("hc_sparse_conv_gn_fwd", sparse_conv_gn_fwd),
    METHOD("hc_conv_rulebook_transpose", conv_rulebook_transpose),
    METHOD("hc_sparse_conv_rulebook_bwd", sparse_conv_rulebook_bwd),
    METHOD("hc_mask_score_update", mask_score_update),
    METHOD("hc_mask_select_topk", mask_select_topk),
    METHOD("hc_kappa_masks", kappa_masks),
    METHOD("hc_gather_rows", gather_rows),
    METHOD("hc_scatter_dense", scatter_dense),
    METHOD("hc_spiral_conv_fwd", spiral_conv_fwd),
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_hc_native", nullptr, -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__hc_native() { return PyModule_Create(&module); }
