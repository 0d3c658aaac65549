// Native fast path of the Python binding (binding.py): the calls a user makes on every step, with the checks of the Python
// wrappers done on the tensors themselves.  A short call on the device takes 2 us; the wrapper's Python and ctypes took 2 to 6.
//
// Every function takes the wrapper's arguments and returns the output tensor, or None when anything is not as the fast path
// expects it (a wrong type, layout, device or size, an argument out of range, a status other than OK): the wrapper then goes
// its own way, which raises the error.  Nothing is decided here that the wrapper would decide differently.
// As under ctypes, the library's calls run without the interpreter lock: a launch blocks while its stream's queue is full, and what
// empties the queue may be a Python callback.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "hikonv.h"

namespace {

decltype(&hikonv_conv1d) g_conv1d = nullptr;
decltype(&hikonv_conv1d_dense) g_conv1d_dense = nullptr;
decltype(&hikonv_conv2d) g_conv2d = nullptr;
decltype(&hikonv_conv2d_dense) g_conv2d_dense = nullptr;
decltype(&hikonv_conv2d_workspace_bytes) g_workspace_bytes = nullptr;
decltype(&hikonv_pack) g_pack = nullptr;

// Reads arguments one after the other; `ok` stays true while all are as expected.
struct Args {
    PyObject *const *a;
    Py_ssize_t n, at = 0;
    bool ok = true;

    PyObject *next() {
        if (at >= n) ok = false;
        return at < n ? a[at++] : Py_None;
    }
    long integer() {
        const long v = PyLong_AsLong(next());
        if (v == -1 && PyErr_Occurred()) {
            PyErr_Clear();
            ok = false;
        }
        return v;
    }
    int int32() {
        const long v = integer();
        if (v != (int)v) ok = false;
        return (int)v;
    }
    const at::Tensor *tensor() {
        PyObject *o = next();
        if (!THPVariable_Check(o)) {
            ok = false;
            return nullptr;
        }
        return &THPVariable_Unpack(o);
    }
    // a tensor, or null for None
    const at::Tensor *optional_tensor() {
        if (at < n && a[at] == Py_None) {
            ++at;
            return nullptr;
        }
        return tensor();
    }
    // (shift, lo, hi), or false for None
    bool requant(int *shift, int *lo, int *hi) {
        PyObject *o = next();
        *shift = *lo = *hi = 0;
        if (o == Py_None) return false;
        if (!PyTuple_Check(o) || PyTuple_GET_SIZE(o) != 3) {
            ok = false;
            return false;
        }
        Args inner{&PyTuple_GET_ITEM(o, 0), 3};
        *shift = inner.int32();
        *lo = inner.int32();
        *hi = inner.int32();
        ok = ok && inner.ok;
        return true;
    }
    // a tuple or torch.Size of four sizes
    bool shape4(int64_t (&s)[4]) {
        PyObject *o = next();
        if (!PyTuple_Check(o) || PyTuple_GET_SIZE(o) != 4) return ok = false;
        Args inner{&PyTuple_GET_ITEM(o, 0), 4};
        for (auto &v : s) v = inner.integer();
        return ok = ok && inner.ok;
    }
};

bool plain_cuda(const at::Tensor *t) { return t && t->is_cuda() && t->layout() == at::kStrided && t->is_contiguous(); }
bool codes(const at::Tensor *t) { return plain_cuda(t) && (t->scalar_type() == at::kChar || t->scalar_type() == at::kByte); }
bool fits_int(int64_t v) { return v == (int)v; }
bool output_ok(const at::Tensor &t, int64_t numel, bool bytes, const at::Tensor &like) {
    return plain_cuda(&t) && t.device() == like.device() && t.numel() == numel &&
           (bytes ? t.scalar_type() == at::kChar || t.scalar_type() == at::kByte : t.scalar_type() == at::kInt);
}
at::Tensor empty(at::IntArrayRef sizes, at::ScalarType type, const at::Tensor &like) {
    return at::empty(sizes, at::TensorOptions().dtype(type).device(like.device()));
}
// The stream a call without one runs on: the current stream of the current device, as in the wrappers.
void *current_stream() { return (void *)c10::cuda::getCurrentCUDAStream().stream(); }

// `out` when it was given, else a new Python object for the tensor that was made.
PyObject *result(PyObject *given, const at::Tensor &made) {
    if (given != Py_None) {
        Py_INCREF(given);
        return given;
    }
    return THPVariable_Wrap(made);
}

// Calls into the library with the interpreter lock released.
template <typename F>
int unlocked(F call) {
    int status;
    Py_BEGIN_ALLOW_THREADS
    status = call();
    Py_END_ALLOW_THREADS
    return status;
}

template <typename F>
PyObject *guarded(F f) {
    try {
        if (PyObject *r = f()) return r;
        if (PyErr_Occurred()) return nullptr;
    } catch (const std::exception &) {                   // an allocation that failed, say: the wrapper meets it again
    }
    Py_RETURN_NONE;
}

// conv1d(f, g, p, q, f_signed, g_signed, algo, out)
PyObject *conv1d(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        Args in{a, n};
        const at::Tensor *f = in.tensor(), *g = in.tensor();
        const int p = in.int32(), q = in.int32(), fs = in.int32() != 0, gs = in.int32() != 0, algo = in.int32();
        const at::Tensor *given = in.optional_tensor();
        if (!in.ok || !codes(f) || !codes(g) || !fits_int(g->numel())) return nullptr;
        const int64_t len = f->numel(), n_out = len + g->numel() - 1;
        if (len < 1 || g->numel() < 1) return nullptr;
        at::Tensor made;
        if (!given) made = empty({n_out}, at::kInt, *f);
        const at::Tensor &y = given ? *given : made;
        if (!output_ok(y, n_out, false, *f)) return nullptr;
        const int8_t *f_ptr = (const int8_t *)f->data_ptr(), *g_ptr = (const int8_t *)g->data_ptr();
        const int K = (int)g->numel();
        int32_t *y_ptr = (int32_t *)y.data_ptr();
        void *st = current_stream();
        if (unlocked([&] { return g_conv1d(f_ptr, (size_t)len, g_ptr, K, p, q, fs, gs, y_ptr, algo, nullptr, st); }) != HIKONV_OK) return nullptr;
        return result(a[7], made);
    });
}

// conv1d_dense(f_dense, n, g, p, q, f_signed, g_signed, out)
PyObject *conv1d_dense(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        Args in{a, n};
        const at::Tensor *f = in.tensor();
        const int64_t len = in.integer();
        const at::Tensor *g = in.tensor();
        const int p = in.int32(), q = in.int32(), fs = in.int32() != 0, gs = in.int32() != 0;
        const at::Tensor *given = in.optional_tensor();
        if (!in.ok || !codes(f) || f->scalar_type() != at::kByte || !codes(g) || !fits_int(g->numel())) return nullptr;
        if (len < 1 || g->numel() < 1 || p < 1 || p > 8 || f->numel() * 8 < len * p) return nullptr;
        const int64_t n_out = len + g->numel() - 1;
        at::Tensor made;
        if (!given) made = empty({n_out}, at::kInt, *f);
        const at::Tensor &y = given ? *given : made;
        if (!output_ok(y, n_out, false, *f)) return nullptr;
        const uint8_t *f_ptr = (const uint8_t *)f->data_ptr();
        const int8_t *g_ptr = (const int8_t *)g->data_ptr();
        const int K = (int)g->numel();
        int32_t *y_ptr = (int32_t *)y.data_ptr();
        void *st = current_stream();
        if (unlocked([&] { return g_conv1d_dense(f_ptr, (size_t)len, g_ptr, K, p, q, fs, gs, y_ptr, nullptr, st); }) != HIKONV_OK) return nullptr;
        return result(a[7], made);
    });
}

// pack(in, bits, is_signed, S, N, word_bits)
PyObject *pack(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        Args in{a, n};
        const at::Tensor *x = in.tensor();
        const int bits = in.int32(), is_signed = in.int32() != 0, S = in.int32(), N = in.int32(), word_bits = in.int32();
        if (!in.ok || !codes(x) || N < 1 || (word_bits != 32 && word_bits != 64)) return nullptr;
        const int64_t count = x->numel();
        const at::Tensor words = empty({(count + N - 1) / N}, word_bits == 32 ? at::kInt : at::kLong, *x);
        const int8_t *x_ptr = (const int8_t *)x->data_ptr();
        void *words_ptr = words.data_ptr(), *st = current_stream();
        if (unlocked([&] { return g_pack(x_ptr, (size_t)count, bits, is_signed, S, N, word_bits, words_ptr, st); }) != HIKONV_OK) return nullptr;
        return THPVariable_Wrap(words);
    });
}

// What the 2-D calls share.  B, Ci, H, W and Co, Ci, K, K are known; makes the workspace and the output where none was given.
struct Layer {
    int64_t B, Ci, H, W, Co, K;
    int pad;
    int64_t Ho() const { return H + 2 * pad - K + 1; }
    int64_t Wo() const { return W + 2 * pad - K + 1; }
    bool plausible() const {
        for (int64_t v : {B, Ci, H, W, Co, K})
            if (v < 1 || !fits_int(v)) return false;
        return pad >= 0 && pad < 1 << 20 && Ho() >= 1 && Wo() >= 1;
    }
    bool workspace(const at::Tensor *given, const at::Tensor &like, at::Tensor *made, void **ptr, size_t *bytes) const {
        if (!given) {
            *made = empty({(int64_t)g_workspace_bytes((int)B, (int)Ci, (int)H, (int)W, (int)Co, (int)K, pad)}, at::kByte, like);
            given = made;
        } else if (!plain_cuda(given) || given->device() != like.device()) {
            return false;
        }
        *ptr = given->data_ptr();
        *bytes = (size_t)given->numel() * given->element_size();
        return true;
    }
};

// conv2d(x, w, pad, p, q, x_signed, w_signed, requant, algo, workspace, out, stride)
PyObject *conv2d(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        Args in{a, n};
        const at::Tensor *x = in.tensor(), *w = in.tensor();
        Layer l;
        l.pad = in.int32();
        const int p = in.int32(), q = in.int32(), xs = in.int32() != 0, ws = in.int32() != 0;
        int shift, lo, hi;
        const bool rq = in.requant(&shift, &lo, &hi);
        const int algo = in.int32();
        const at::Tensor *space = in.optional_tensor(), *given = in.optional_tensor();
        const int stride = in.int32();
        if (!in.ok || !codes(x) || !codes(w) || x->dim() != 4 || w->dim() != 4) return nullptr;
        l.B = x->size(0); l.Ci = x->size(1); l.H = x->size(2); l.W = x->size(3);
        l.Co = w->size(0); l.K = w->size(2);
        if (w->size(1) != l.Ci || w->size(3) != l.K || !l.plausible()) return nullptr;
        at::Tensor made_space, made;
        void *space_ptr;
        size_t space_bytes;
        if (!l.workspace(space, *x, &made_space, &space_ptr, &space_bytes)) return nullptr;
        if (!given) made = empty({l.B, l.Co, l.Ho(), l.Wo()}, rq ? at::kChar : at::kInt, *x);
        const at::Tensor &y = given ? *given : made;
        if (!output_ok(y, l.B * l.Co * l.Ho() * l.Wo(), rq, *x)) return nullptr;
        const int8_t *x_ptr = (const int8_t *)x->data_ptr(), *w_ptr = (const int8_t *)w->data_ptr();
        void *y_ptr = y.data_ptr(), *st = current_stream();
        const int status = unlocked([&] {
            return g_conv2d(x_ptr, (int)l.B, (int)l.Ci, (int)l.H, (int)l.W, w_ptr, (int)l.Co, (int)l.K, stride, l.pad, p, q, xs, ws, y_ptr,
                            rq ? 1 : 0, shift, lo, hi, space_ptr, space_bytes, algo, nullptr, st);
        });
        if (status != HIKONV_OK) return nullptr;
        return result(a[10], made);
    });
}

// conv2d_dense(x, x_shape, x_store_bits, w, w_shape, w_store_bits, pad, p, q, x_signed, w_signed, requant, out_store_bits, pool,
//              algo, workspace, out, stride)
PyObject *conv2d_dense(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded([&]() -> PyObject * {
        Args in{a, n};
        const at::Tensor *x = in.tensor();
        int64_t xsh[4], wsh[4];
        in.shape4(xsh);
        const int x_bits = in.int32();
        const at::Tensor *w = in.tensor();
        in.shape4(wsh);
        const int w_bits = in.int32();
        Layer l;
        l.pad = in.int32();
        const int p = in.int32(), q = in.int32(), xs = in.int32() != 0, ws = in.int32() != 0;
        int shift, lo, hi;
        const bool rq = in.requant(&shift, &lo, &hi);
        const int out_bits = in.int32(), pool = in.int32() != 0, algo = in.int32();
        const at::Tensor *space = in.optional_tensor(), *given = in.optional_tensor();
        const int stride = in.int32();
        if (!in.ok || !codes(x) || !codes(w)) return nullptr;
        l.B = xsh[0]; l.Ci = xsh[1]; l.H = xsh[2]; l.W = xsh[3];
        l.Co = wsh[0]; l.K = wsh[2];
        if (wsh[1] != l.Ci || wsh[3] != l.K || !l.plausible()) return nullptr;
        if (x_bits < 1 || x_bits > 8 || w_bits < 1 || w_bits > 8 || out_bits < 1 || out_bits > 8) return nullptr;
        if (x->numel() * 8 < l.B * l.Ci * l.H * l.W * x_bits || w->numel() * 8 < l.Co * l.Ci * l.K * l.K * w_bits) return nullptr;
        const int64_t Hq = pool ? l.Ho() / 2 : l.Ho(), Wq = pool ? l.Wo() / 2 : l.Wo();
        at::Tensor made_space, made;
        void *space_ptr;
        size_t space_bytes;
        if (!l.workspace(space, *x, &made_space, &space_ptr, &space_bytes)) return nullptr;
        const int64_t n_out = rq ? (l.B * l.Co * Hq * Wq * out_bits + 7) / 8 : l.B * l.Co * l.Ho() * l.Wo();
        if (!given)
            made = !rq ? empty({l.B, l.Co, l.Ho(), l.Wo()}, at::kInt, *x)
                 : out_bits == 8 ? empty({l.B, l.Co, Hq, Wq}, at::kChar, *x) : empty({n_out}, at::kByte, *x);
        const at::Tensor &y = given ? *given : made;
        if (!output_ok(y, n_out, rq, *x)) return nullptr;
        const void *x_ptr = x->data_ptr(), *w_ptr = w->data_ptr();
        void *y_ptr = y.data_ptr(), *st = current_stream();
        const int status = unlocked([&] {
            return g_conv2d_dense(x_ptr, x_bits, (int)l.B, (int)l.Ci, (int)l.H, (int)l.W, w_ptr, w_bits, (int)l.Co, (int)l.K, stride, l.pad, p, q,
                                  xs, ws, y_ptr, rq ? out_bits : 32, rq ? 1 : 0, shift, lo, hi, pool, space_ptr, space_bytes, algo, nullptr, st);
        });
        if (status != HIKONV_OK) return nullptr;
        return result(a[16], made);
    });
}

// bind(name, address): the entry points of the library that is loaded.
PyObject *bind(PyObject *, PyObject *args) {
    const char *name;
    unsigned long long address;
    if (!PyArg_ParseTuple(args, "sK", &name, &address)) return nullptr;
    const std::string s(name);
    void *ptr = (void *)(uintptr_t)address;
    if (s == "hikonv_conv1d") g_conv1d = (decltype(g_conv1d))ptr;
    else if (s == "hikonv_conv1d_dense") g_conv1d_dense = (decltype(g_conv1d_dense))ptr;
    else if (s == "hikonv_conv2d") g_conv2d = (decltype(g_conv2d))ptr;
    else if (s == "hikonv_conv2d_dense") g_conv2d_dense = (decltype(g_conv2d_dense))ptr;
    else if (s == "hikonv_conv2d_workspace_bytes") g_workspace_bytes = (decltype(g_workspace_bytes))ptr;
    else if (s == "hikonv_pack") g_pack = (decltype(g_pack))ptr;
    else {
        PyErr_Format(PyExc_ValueError, "no entry point %s", name);
        return nullptr;
    }
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, nullptr},
    {"conv1d", (PyCFunction)(void (*)(void))conv1d, METH_FASTCALL, nullptr},
    {"conv1d_dense", (PyCFunction)(void (*)(void))conv1d_dense, METH_FASTCALL, nullptr},
    {"pack", (PyCFunction)(void (*)(void))pack, METH_FASTCALL, nullptr},
    {"conv2d", (PyCFunction)(void (*)(void))conv2d, METH_FASTCALL, nullptr},
    {"conv2d_dense", (PyCFunction)(void (*)(void))conv2d_dense, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fast", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fast(void) { return PyModule_Create(&module); }
