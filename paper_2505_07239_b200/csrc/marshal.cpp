// Argument marshalling of the calls a serving loop makes on every pass, as a CPython module: checks the tensors, takes
// their addresses and calls the C ABI.  It holds no step of the path; binding.py is the only user and keeps the rarer calls
// in ctypes.
//
// What bounds the smallest layers is host time: 16 bindings, a mask, four launching calls.  Through ctypes a binding took
// 1.6 us, of which the library's own code is 0.1; here it takes 0.27, and a
// stateless call that returns six new tensors 8 us instead of 21.
#include <Python.h>

#include <ATen/core/Tensor.h>
#include <ATen/EmptyTensor.h>
#include <c10/core/Allocator.h>
#include <c10/core/DeviceGuard.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "../../include/comet.h"

namespace {

// Returns false with a Python exception set.
bool refuse(PyObject* type, const char* what) {
    PyErr_SetString(type, what);
    return false;
}

bool as_int(PyObject* o, int64_t* out) {
    *out = PyLong_AsLongLong(o);
    return !(*out == -1 && PyErr_Occurred());
}

bool as_context(PyObject* o, comet_ctx** out) {
    if (o == Py_None) {
        *out = nullptr;
        return true;
    }
    *out = static_cast<comet_ctx*>(PyLong_AsVoidPtr(o));
    return !(*out == nullptr && PyErr_Occurred());
}

// A CUDA stream object, or None for the default stream.
bool as_stream(PyObject* o, void** out) {
    *out = nullptr;
    if (o == Py_None) return true;
    static PyObject* name = PyUnicode_InternFromString("cuda_stream");
    PyObject* v = PyObject_GetAttr(o, name);
    if (!v) return false;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
    return !(*out == nullptr && PyErr_Occurred());
}

const at::Tensor* as_tensor(PyObject* o) {
    if (!THPVariable_Check(o)) {
        PyErr_SetString(PyExc_TypeError, "a torch tensor is expected");
        return nullptr;
    }
    return &THPVariable_Unpack(o);
}

bool device_words(const at::Tensor& t) { return t.is_cuda() && t.is_contiguous() && t.element_size() == 8; }

// The tensors of both parties: contiguous, on the GPU, of a given element size.  The items are this object's own references
// until the call is over: what they came from may make its items on demand (a stacked tensor, any class with __getitem__).
struct Pair {
    PyObject* item[2] = {nullptr, nullptr};
    const at::Tensor* t[2] = {nullptr, nullptr};
    Pair() = default;
    Pair(const Pair&) = delete;
    ~Pair() {
        Py_XDECREF(item[0]);
        Py_XDECREF(item[1]);
    }
    const at::Tensor& operator[](int p) const { return *t[p]; }
};

bool as_pair(PyObject* o, int bytes, Pair& out) {
    static PyObject* const index[2] = {PyLong_FromLong(0), PyLong_FromLong(1)};
    for (int p = 0; p < 2; ++p) {
        if (!(out.item[p] = PyObject_GetItem(o, index[p])) || !(out.t[p] = as_tensor(out.item[p]))) return false;
        if (!out[p].is_cuda() || !out[p].is_contiguous() || out[p].element_size() != bytes)
            return refuse(PyExc_AssertionError, "contiguous CUDA tensors of the documented element size are expected");
    }
    return true;
}

bool same_shape(const Pair& t, const at::Tensor& like) {
    if (t[0].sizes() == like.sizes() && t[1].sizes() == like.sizes()) return true;
    return refuse(PyExc_AssertionError, "the tensors of both parties must have the documented shapes");
}

bool shaped(const Pair& t, std::initializer_list<int64_t> shape) {
    const at::IntArrayRef s(shape);
    if (t[0].sizes() == s && t[1].sizes() == s) return true;
    return refuse(PyExc_AssertionError, "the tensors of both parties must have the documented shapes");
}

uint64_t* words(const at::Tensor& t) { return static_cast<uint64_t*>(t.data_ptr()); }

struct ConstPair {
    const uint64_t* p[2];
    explicit ConstPair(const Pair& t) : p{words(t[0]), words(t[1])} {}
};

// A new contiguous tensor like `like`, on its device, from torch's CUDA allocator and on the current stream as ever, without the
// two dispatched calls of at::empty_like: the six results of a product come 2.4 us sooner.
at::Tensor empty_like(const at::Tensor& like) {
    const c10::DeviceGuard guard(like.device());
    return at::detail::empty_generic(like.sizes(), c10::GetAllocator(c10::DeviceType::CUDA),
                                     c10::DispatchKeySet(c10::DispatchKey::CUDA), like.scalar_type(), std::nullopt);
}

// Two new tensors like `like`, and their addresses.
struct NewPair {
    at::Tensor t[2];
    uint64_t* p[2];
    explicit NewPair(const at::Tensor& like) {
        for (int i = 0; i < 2; ++i) {
            t[i] = empty_like(like);
            p[i] = words(t[i]);
        }
    }
    PyObject* list() const {
        PyObject* l = PyList_New(2);
        for (int i = 0; l && i < 2; ++i) {
            PyObject* o = THPVariable_Wrap(t[i]);
            if (!o) {
                Py_DECREF(l);
                return nullptr;
            }
            PyList_SET_ITEM(l, i, o);
        }
        return l;
    }
};

// (code, list, list, ...): what the Python side unpacks.
PyObject* answer(int code, std::initializer_list<const NewPair*> pairs) {
    PyObject* out = PyTuple_New(1 + (Py_ssize_t)pairs.size());
    if (!out) return nullptr;
    PyTuple_SET_ITEM(out, 0, PyLong_FromLong(code));
    Py_ssize_t i = 1;
    for (const NewPair* p : pairs) {
        PyObject* l = p->list();
        if (!l) {
            Py_DECREF(out);
            return nullptr;
        }
        PyTuple_SET_ITEM(out, i++, l);
    }
    return out;
}

bool counted(Py_ssize_t n, Py_ssize_t want) {
    return n == want || refuse(PyExc_TypeError, "wrong number of arguments");
}

template <typename F>
PyObject* guarded(F&& f) {
    try {
        return f();
    } catch (const std::exception& e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

template <typename F>
int unlocked(F&& f) {
    int code;
    Py_BEGIN_ALLOW_THREADS;
    code = f();
    Py_END_ALLOW_THREADS;
    return code;
}

// bind_shares(context, party, tensor_id, tensor) / load_shares(...) -> code
PyObject* give_shares(PyObject* const* args, Py_ssize_t n, bool bind) {
    return guarded([&]() -> PyObject* {
        comet_ctx* ctx;
        int64_t party, id;
        if (!counted(n, 4) || !as_context(args[0], &ctx) || !as_int(args[1], &party) || !as_int(args[2], &id)) return nullptr;
        const at::Tensor* t = as_tensor(args[3]);
        if (!t) return nullptr;
        if (!t->is_contiguous() || t->element_size() != 8 || (bind && !t->is_cuda())) {
            refuse(PyExc_AssertionError, "a contiguous tensor of 8-byte words is expected");
            return nullptr;
        }
        if (t->dim() != 2) {
            refuse(PyExc_ValueError, "a matrix is expected");
            return nullptr;
        }
        const int64_t rows = t->size(0), cols = t->size(1);
        const uint64_t* ptr = words(*t);
        const int location = t->is_cuda() ? COMET_DEVICE : COMET_HOST;
        return PyLong_FromLong(unlocked([&] {
            return bind ? comet_bind_shares(ctx, (int)party, (int)id, ptr, rows, cols)
                        : comet_load_shares(ctx, (int)party, (int)id, ptr, location, rows, cols);
        }));
    });
}
PyObject* bind_shares(PyObject*, PyObject* const* args, Py_ssize_t n) { return give_shares(args, n, true); }
PyObject* load_shares(PyObject*, PyObject* const* args, Py_ssize_t n) { return give_shares(args, n, false); }

// set_mask(context, host array of bytes) -> (code, active neurons)
PyObject* set_mask(PyObject*, PyObject* const* args, Py_ssize_t n) {
    comet_ctx* ctx;
    if (!counted(n, 2) || !as_context(args[0], &ctx)) return nullptr;
    Py_buffer view;
    if (PyObject_GetBuffer(args[1], &view, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS)) {
        PyErr_Clear();
        refuse(PyExc_AssertionError, "a contiguous array of bytes is expected");
        return nullptr;
    }
    int32_t active = 0;
    int code = 0;
    const bool bytes = view.itemsize == 1 && view.format && std::strcmp(view.format, "B") == 0;
    if (bytes)
        code = unlocked([&] {
            return comet_set_mask(ctx, static_cast<const uint8_t*>(view.buf), COMET_HOST, (int32_t)view.len, &active);
        });
    PyBuffer_Release(&view);
    if (!bytes) {
        refuse(PyExc_AssertionError, "a contiguous array of bytes is expected");
        return nullptr;
    }
    return Py_BuildValue("ii", code, active);
}

// ffn_up(context, tokens), ffn_down(context, tokens), truncate(context, tensor_id) -> code
template <int (*CALL)(comet_ctx*, int32_t)>
PyObject* step(PyObject*, PyObject* const* args, Py_ssize_t n) {
    comet_ctx* ctx;
    int64_t v;
    if (!counted(n, 2) || !as_context(args[0], &ctx) || !as_int(args[1], &v)) return nullptr;
    return PyLong_FromLong(unlocked([&] { return CALL(ctx, (int32_t)v); }));
}
int truncate_call(comet_ctx* ctx, int32_t id) { return comet_truncate(ctx, id); }

// shuffle(stream, X, tau, rho, a, b, bad_index_flag) -> (code, Y, Z)
PyObject* shuffle(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        void* stream;
        Pair X, tau, rho, a, b;
        const at::Tensor* flag = nullptr;
        if (!counted(n, 7) || !as_stream(args[0], &stream) || !as_pair(args[1], 8, X) || !as_pair(args[2], 4, tau) ||
            !as_pair(args[3], 4, rho) || !as_pair(args[4], 8, a) || !as_pair(args[5], 8, b))
            return nullptr;
        if (args[6] != Py_None && !(flag = as_tensor(args[6]))) return nullptr;
        const int64_t rows = X[0].size(0), cols = rows ? X[0].numel() / rows : 0;
        for (int p = 0; p < 2; ++p)
            if (tau[p].scalar_type() != at::kInt || rho[p].scalar_type() != at::kInt) {
                refuse(PyExc_AssertionError, "int32 permutations are expected");
                return nullptr;
            }
        if (!same_shape(X, X[0]) || !shaped(tau, {rows}) || !shaped(rho, {rows}) || !same_shape(a, X[0]) ||
            !same_shape(b, X[0]))
            return nullptr;
        const NewPair Y(X[0]), Z(X[0]);
        const ConstPair x(X), am(a), bm(b);
        const int32_t* t[2] = {static_cast<int32_t*>(tau[0].data_ptr()), static_cast<int32_t*>(tau[1].data_ptr())};
        const int32_t* r[2] = {static_cast<int32_t*>(rho[0].data_ptr()), static_cast<int32_t*>(rho[1].data_ptr())};
        int32_t* f = flag ? static_cast<int32_t*>(flag->data_ptr()) : nullptr;
        const int code = unlocked([&] { return comet_shuffle(stream, x.p, t, r, am.p, bm.p, Y.p, Z.p, rows, cols, f); });
        return answer(code, {&Y, &Z});
    });
}

// invert_permutation(stream, perm, bad_index_flag) -> (code, inverse)
PyObject* invert_permutation(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        void* stream;
        const at::Tensor *perm, *flag = nullptr;
        if (!counted(n, 3) || !as_stream(args[0], &stream) || !(perm = as_tensor(args[1]))) return nullptr;
        if (args[2] != Py_None && !(flag = as_tensor(args[2]))) return nullptr;
        if (!perm->is_cuda() || !perm->is_contiguous() || perm->scalar_type() != at::kInt) {
            refuse(PyExc_AssertionError, "a contiguous int32 CUDA tensor is expected");
            return nullptr;
        }
        const at::Tensor out = empty_like(*perm);
        const int32_t* in = static_cast<int32_t*>(perm->data_ptr());
        int32_t *to = static_cast<int32_t*>(out.data_ptr()), *f = flag ? static_cast<int32_t*>(flag->data_ptr()) : nullptr;
        const int64_t rows = perm->numel();
        const int code = unlocked([&] { return comet_invert_permutation(stream, in, to, rows, f); });
        return Py_BuildValue("iN", code, THPVariable_Wrap(out));
    });
}

// beaver_mul(stream, X, Y, A, B, C) -> (code, D, E, Z)
PyObject* beaver_mul(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        void* stream;
        Pair in[5];
        if (!counted(n, 6) || !as_stream(args[0], &stream)) return nullptr;
        for (int k = 0; k < 5; ++k)
            if (!as_pair(args[1 + k], 8, in[k]) || !same_shape(in[k], in[0][0])) return nullptr;
        const NewPair D(in[0][0]), E(in[0][0]), Z(in[0][0]);
        const ConstPair x(in[0]), y(in[1]), a(in[2]), b(in[3]), c(in[4]);
        const int64_t count = in[0][0].numel();
        const int code = unlocked([&] { return comet_beaver_mul(stream, x.p, y.p, a.p, b.p, c.p, D.p, E.p, Z.p, count); });
        return answer(code, {&D, &E, &Z});
    });
}

// truncate_pair(stream, Z, R, RP, frac_bits) -> (code, M)
PyObject* truncate_pair(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        void* stream;
        int64_t frac;
        Pair z, r, rp;
        if (!counted(n, 5) || !as_stream(args[0], &stream) || !as_pair(args[1], 8, z) || !as_pair(args[2], 8, r) ||
            !as_pair(args[3], 8, rp) || !as_int(args[4], &frac))
            return nullptr;
        if (!same_shape(z, z[0]) || !same_shape(r, z[0]) || !same_shape(rp, z[0])) return nullptr;
        const NewPair M(z[0]);
        const ConstPair rc(r), rpc(rp);
        uint64_t* const zp[2] = {words(z[0]), words(z[1])};
        const int64_t count = z[0].numel();
        const int code = unlocked([&] { return comet_truncate_pair(stream, zp, rc.p, rpc.p, M.p, count, (int32_t)frac); });
        return answer(code, {&M});
    });
}

// add_bias(stream, Z, bias) -> code
PyObject* add_bias(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        void* stream;
        Pair z, bias;
        if (!counted(n, 3) || !as_stream(args[0], &stream) || !as_pair(args[1], 8, z) || !as_pair(args[2], 8, bias))
            return nullptr;
        if (z[0].dim() != 2) {
            refuse(PyExc_ValueError, "a matrix is expected");
            return nullptr;
        }
        const int64_t rows = z[0].size(0), cols = z[0].size(1);
        if (!same_shape(z, z[0]) || !shaped(bias, {cols})) return nullptr;
        uint64_t* const zp[2] = {words(z[0]), words(z[1])};
        const ConstPair b(bias);
        return PyLong_FromLong(unlocked([&] { return comet_add_bias(stream, zp, b.p, rows, cols); }));
    });
}

// beaver_matmul_static(stream, X, A, Y, B, C, Z) -> code
PyObject* beaver_matmul_static(PyObject*, PyObject* const* args, Py_ssize_t n) {
    return guarded([&]() -> PyObject* {
        void* stream;
        Pair t[6];
        if (!counted(n, 7) || !as_stream(args[0], &stream)) return nullptr;
        for (int k = 0; k < 6; ++k)
            if (!as_pair(args[1 + k], 8, t[k])) return nullptr;
        if (t[0][0].dim() != 2 || t[2][0].dim() != 2) {
            refuse(PyExc_ValueError, "matrices are expected");
            return nullptr;
        }
        const int64_t T = t[0][0].size(0), K = t[0][0].size(1), N = t[2][0].size(0);
        if (!shaped(t[0], {T, K}) || !shaped(t[1], {T, K}) || !shaped(t[2], {N, K}) || !shaped(t[3], {N, K}) ||
            !shaped(t[4], {T, N}) || !shaped(t[5], {T, N}))
            return nullptr;
        const ConstPair X(t[0]), A(t[1]), Y(t[2]), B(t[3]), C(t[4]);
        uint64_t* const Z[2] = {words(t[5][0]), words(t[5][1])};
        return PyLong_FromLong(unlocked([&] {
            return comet_beaver_matmul_static(stream, X.p, A.p, Y.p, B.p, C.p, Z, (int32_t)T, (int32_t)K, (int32_t)N);
        }));
    });
}

#define FAST(name, f) {name, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    FAST("bind_shares", bind_shares),
    FAST("load_shares", load_shares),
    FAST("set_mask", set_mask),
    FAST("ffn_up", step<comet_ffn_up>),
    FAST("ffn_down", step<comet_ffn_down>),
    FAST("truncate", step<truncate_call>),
    FAST("shuffle", shuffle),
    FAST("invert_permutation", invert_permutation),
    FAST("beaver_mul", beaver_mul),
    FAST("truncate_pair", truncate_pair),
    FAST("add_bias", add_bias),
    FAST("beaver_matmul_static", beaver_matmul_static),
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
