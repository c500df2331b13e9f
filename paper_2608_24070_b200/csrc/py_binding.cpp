// Native marshalling of the Python binding: takes torch tensors, hands device addresses, sizes and torch's
// current stream to the C ABI (include/slope.h).  Nothing is computed here.  The functions mirror those
// of binding.py, which documents them; each returns the C status.
//
// What bounds a call on a small layer is the host: through ctypes an eager slope_linear_fwd cost 5.8 us for a
// 3.3 us kernel, of which 1.7 us were attribute look-ups and shape tuples in Python and 0.9 us the
// conversion of eleven arguments; here the whole call takes 2.6 us.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <dlfcn.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/slope.h"

// The torch and Python this module was compiled against (build.native_build()); build.py and binding.py look for it in the file.
extern "C" __attribute__((used)) const char slope_native_build[] = SLOPE_NATIVE_BUILD;

namespace {

#define SLOPE_CALLS(X)                                                                                                  \
    X(slope_prune_24) X(slope_double_prune) X(slope_prune_24_double) X(slope_linear_fwd) X(slope_linear_fwd_adapter)    \
    X(slope_linear_bwd_dx) X(slope_linear_bwd_dw_masked) X(slope_adapter_fwd_bwd) X(slope_linear_bwd_dw_adapter)        \
    X(slope_sparse_add) X(slope_update_sparse_matrix) X(slope_prune_nm) X(slope_double_prune_nm) X(slope_apply_mask)    \
    X(slope_dense_linear_fwd) X(slope_dense_linear_bwd_dx) X(slope_dense_linear_bwd_dw)

// the library's entry points, looked up in the handle that binding.lib() loaded
#define SLOPE_POINTER(name) decltype(&::name) p_##name = nullptr;
SLOPE_CALLS(SLOPE_POINTER)

struct Bad {};                    // a Python exception is set

// One call's arguments, read in order.
struct Args {
    PyObject* const* at;
    Py_ssize_t left;

    PyObject* next() {
        if (left <= 0) {
            PyErr_SetString(PyExc_TypeError, "too few arguments");
            throw Bad{};
        }
        --left;
        return *at++;
    }
    const at::Tensor* tensor_or_none() {
        PyObject* o = next();
        if (o == Py_None) return nullptr;
        if (!THPVariable_Check(o)) {
            PyErr_SetString(PyExc_TypeError, "expected a torch tensor or None");
            throw Bad{};
        }
        const at::Tensor& t = THPVariable_Unpack(o);
        if (!t.is_cuda() || !t.is_contiguous()) {
            PyErr_SetString(PyExc_AssertionError, "tensors must be contiguous CUDA tensors");
            throw Bad{};
        }
        return &t;
    }
    const at::Tensor& tensor() {
        const at::Tensor* t = tensor_or_none();
        if (!t) {
            PyErr_SetString(PyExc_TypeError, "expected a torch tensor");
            throw Bad{};
        }
        return *t;
    }
    const at::Tensor& matrix() {
        const at::Tensor& t = tensor();
        if (t.dim() != 2) {
            PyErr_SetString(PyExc_ValueError, "expected a 2-D tensor");
            throw Bad{};
        }
        return t;
    }
    void* ptr() {
        const at::Tensor* t = tensor_or_none();
        return t ? t->data_ptr() : nullptr;
    }
    int integer() {
        const long v = PyLong_AsLong(next());
        if (v == -1 && PyErr_Occurred()) throw Bad{};
        if (v != static_cast<int>(v)) {
            PyErr_SetString(PyExc_OverflowError, "integer argument out of range");
            throw Bad{};
        }
        return static_cast<int>(v);
    }
    float number() {
        const double v = PyFloat_AsDouble(next());
        if (v == -1.0 && PyErr_Occurred()) throw Bad{};
        return static_cast<float>(v);
    }
};

int rows(const at::Tensor& t) { return static_cast<int>(t.size(0)); }
int cols(const at::Tensor& t) { return static_cast<int>(t.size(1)); }
void* stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Runs `body(args)`; C++ exceptions become Python ones.
template <typename Body>
PyObject* guarded(PyObject* const* args, Py_ssize_t n, Body body) {
    try {
        Args a{args, n};
        return PyLong_FromLong(body(a));
    } catch (const Bad&) {
        return nullptr;
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}
template <typename Fn, typename... A>
long call(Fn fn, A... args) {
    void* s = stream();
    slope_status_t st;
    Py_BEGIN_ALLOW_THREADS
    st = fn(args..., s);
    Py_END_ALLOW_THREADS
    return st;
}

#define SLOPE_PY(name) PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n)

SLOPE_PY(slope_prune_24) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& W = a.matrix();
        void *vals = a.ptr(), *meta = a.ptr(), *mask = a.ptr();
        return call(p_slope_prune_24, W.data_ptr(), rows(W), cols(W), vals, meta, mask);
    });
}
SLOPE_PY(slope_double_prune) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& W = a.matrix();
        void *mask1 = a.ptr(), *vals = a.ptr(), *meta = a.ptr(), *mask2 = a.ptr();
        return call(p_slope_double_prune, W.data_ptr(), mask1, rows(W), cols(W), vals, meta, mask2);
    });
}
SLOPE_PY(slope_prune_24_double) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& W = a.matrix();
        void *vals = a.ptr(), *meta = a.ptr(), *mask1 = a.ptr(), *vals_t = a.ptr(), *meta_t = a.ptr(), *mask2 = a.ptr();
        return call(p_slope_prune_24_double, W.data_ptr(), rows(W), cols(W), vals, meta, mask1, vals_t, meta_t, mask2);
    });
}
SLOPE_PY(slope_linear_fwd) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& X = a.matrix();
        void *vals = a.ptr(), *meta = a.ptr();
        const int d_out = a.integer();
        void* Y = a.ptr();
        const at::Tensor* T = a.tensor_or_none();
        void* R = a.ptr();
        return call(p_slope_linear_fwd, X.data_ptr(), rows(X), vals, meta, d_out, cols(X), T ? T->data_ptr() : nullptr, R,
                    T ? cols(*T) : 0, Y);
    });
}
SLOPE_PY(slope_linear_fwd_adapter) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& X = a.matrix();
        void *vals = a.ptr(), *meta = a.ptr();
        const int d_out = a.integer();
        const at::Tensor& L = a.matrix();
        void *R = a.ptr(), *T = a.ptr(), *Y = a.ptr();
        return call(p_slope_linear_fwd_adapter, X.data_ptr(), rows(X), vals, meta, d_out, cols(X), L.data_ptr(), R, cols(L), T,
                    Y);
    });
}
SLOPE_PY(slope_linear_bwd_dx) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& dY = a.matrix();
        void *vals = a.ptr(), *meta = a.ptr();
        const int d_in = a.integer();
        void* dX = a.ptr();
        const at::Tensor* dT = a.tensor_or_none();
        void* L = a.ptr();
        return call(p_slope_linear_bwd_dx, dY.data_ptr(), rows(dY), vals, meta, cols(dY), d_in, dT ? dT->data_ptr() : nullptr, L,
                    dT ? cols(*dT) : 0, dX);
    });
}
SLOPE_PY(slope_linear_bwd_dw_masked) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor &dY = a.matrix(), &X = a.matrix();
        void *mask = a.ptr(), *dWc = a.ptr();
        return call(p_slope_linear_bwd_dw_masked, dY.data_ptr(), X.data_ptr(), rows(dY), cols(dY), cols(X), mask, dWc);
    });
}
SLOPE_PY(slope_adapter_fwd_bwd) {
    return guarded(args, n, [](Args& a) {
        const int phase = a.integer();
        void *X = a.ptr(), *dY = a.ptr(), *L = a.ptr(), *R = a.ptr();
        const int b = a.integer(), d_out = a.integer(), d_in = a.integer(), r = a.integer();
        void *T = a.ptr(), *dT = a.ptr(), *dL = a.ptr(), *dR = a.ptr();
        const at::Tensor* ws = a.tensor_or_none();
        return call(p_slope_adapter_fwd_bwd, phase, X, dY, L, R, b, d_out, d_in, r, T, dT, dL, dR,
                    ws ? ws->data_ptr() : nullptr, ws ? ws->nbytes() : size_t(0));
    });
}
SLOPE_PY(slope_linear_bwd_dw_adapter) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor &dY = a.matrix(), &X = a.matrix(), &T = a.matrix();
        void *dT = a.ptr(), *mask = a.ptr(), *dWc = a.ptr(), *dL = a.ptr(), *dR = a.ptr();
        const at::Tensor& ws = a.tensor();
        return call(p_slope_linear_bwd_dw_adapter, dY.data_ptr(), X.data_ptr(), T.data_ptr(), dT, rows(dY), cols(dY), cols(X),
                    cols(T), mask, dWc, dL, dR, ws.data_ptr(), ws.nbytes());
    });
}
SLOPE_PY(slope_sparse_add) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& A = a.matrix();
        void* B = a.ptr();
        const float beta = a.number(), gamma = a.number();
        void* out = a.ptr();
        return call(p_slope_sparse_add, A.data_ptr(), B, beta, gamma, rows(A), 2 * cols(A), out);
    });
}
SLOPE_PY(slope_update_sparse_matrix) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& vals = a.matrix();
        void *mask = a.ptr(), *meta_t = a.ptr(), *vals_t = a.ptr();
        return call(p_slope_update_sparse_matrix, vals.data_ptr(), mask, meta_t, rows(vals), 2 * cols(vals), vals_t);
    });
}
SLOPE_PY(slope_prune_nm) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& W = a.matrix();
        const int keep = a.integer(), group = a.integer();
        void *out = a.ptr(), *mask = a.ptr();
        return call(p_slope_prune_nm, W.data_ptr(), rows(W), cols(W), keep, group, out, mask);
    });
}
SLOPE_PY(slope_double_prune_nm) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& W = a.matrix();
        void* mask1 = a.ptr();
        const int keep = a.integer(), group = a.integer();
        void *out = a.ptr(), *mask2 = a.ptr();
        return call(p_slope_double_prune_nm, W.data_ptr(), mask1, rows(W), cols(W), keep, group, out, mask2);
    });
}
SLOPE_PY(slope_apply_mask) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor& G = a.matrix();
        void *mask = a.ptr(), *out = a.ptr();
        return call(p_slope_apply_mask, G.data_ptr(), mask, rows(G), cols(G), out);
    });
}
SLOPE_PY(slope_dense_linear_fwd) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor &X = a.matrix(), &W = a.matrix();
        void* Y = a.ptr();
        return call(p_slope_dense_linear_fwd, X.data_ptr(), rows(X), W.data_ptr(), rows(W), cols(X), Y);
    });
}
SLOPE_PY(slope_dense_linear_bwd_dx) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor &dY = a.matrix(), &W = a.matrix();
        void* dX = a.ptr();
        return call(p_slope_dense_linear_bwd_dx, dY.data_ptr(), rows(dY), W.data_ptr(), cols(dY), cols(W), dX);
    });
}
SLOPE_PY(slope_dense_linear_bwd_dw) {
    return guarded(args, n, [](Args& a) {
        const at::Tensor &dY = a.matrix(), &X = a.matrix();
        void* dW = a.ptr();
        return call(p_slope_dense_linear_bwd_dw, dY.data_ptr(), X.data_ptr(), rows(dY), cols(dY), cols(X), dW);
    });
}

// attach(handle): look the entry points up in a loaded libslope.so.
PyObject* attach(PyObject*, PyObject* handle) {
    void* lib = PyLong_AsVoidPtr(handle);
    if (!lib && PyErr_Occurred()) return nullptr;
#define SLOPE_LOOKUP(name)                                                          \
    p_##name = reinterpret_cast<decltype(&::name)>(dlsym(lib, #name));              \
    if (!p_##name) {                                                                \
        PyErr_SetString(PyExc_RuntimeError, "libslope.so does not export " #name);  \
        return nullptr;                                                             \
    }
    SLOPE_CALLS(SLOPE_LOOKUP)
    Py_RETURN_NONE;
}

#define SLOPE_METHOD(name) {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(py_##name)), METH_FASTCALL, nullptr},
PyMethodDef methods[] = {{"attach", attach, METH_O, nullptr}, SLOPE_CALLS(SLOPE_METHOD){nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_slope", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__slope() { return PyModule_Create(&module); }
