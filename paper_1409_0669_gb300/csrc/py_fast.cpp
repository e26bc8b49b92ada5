// Direct calls of the C ABI (include/lak.h) from Python for the common forms: plain
// CUDA tensors on the current device and stream, no explicit configuration, stream or
// workspace.  Each function checks exactly that, calls the ABI with raw pointers and
// returns its result tensor; for anything else -- another device, stride, type, a
// tensor subclass or transform, an empty operand, a missing workspace, an error status
// -- it returns None without side effects, and the caller's Python path (which takes
// every form and raises every error) runs instead.
//
// A call through ctypes spends 4-6 us in argument checks, attribute reads and argument
// conversion beside the 2.7 us of the launch, and torch.empty 7 us more where the
// result is allocated; here the checks take well below a microsecond.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAGraphsC10Utils.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <map>
#include <utility>

#include "lak.h"

namespace {

using at::Tensor;

// Workspaces the Python side allocated, per (device, stream); the tensor is held here
// too.  Touched only with the GIL held.
std::map<std::pair<int, int64_t>, Tensor> &workspaces() {
    static std::map<std::pair<int, int64_t>, Tensor> w;
    return w;
}

struct Where {
    int device;
    int64_t handle;       // raw stream
    void *stream() const { return reinterpret_cast<void *>(handle); }
};

Where here() {
    Where w;
    w.device = c10::cuda::current_device();
    w.handle = reinterpret_cast<int64_t>(
        c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)w.device).stream());
    return w;
}

int storage_of(const Tensor &t) {
    switch (t.scalar_type()) {
    case at::kFloat: return LAK_F32;
    case at::kDouble: return LAK_F64;
    case at::kBFloat16: return LAK_BF16;
    case at::kHalf: return LAK_F16;
    default: return -1;
    }
}

// A plain strided CUDA tensor of the current device with elements
const Tensor *plain(PyObject *o, const Where &w) {
    if (!THPVariable_CheckExact(o)) return nullptr;
    const Tensor &t = THPVariable_Unpack(o);
    if (!t.defined() || !t.is_cuda() || t.layout() != at::kStrided || !t.has_storage()) return nullptr;
    const c10::DispatchKeySet odd({c10::DispatchKey::Python, c10::DispatchKey::FuncTorchBatched,
                                   c10::DispatchKey::FuncTorchGradWrapper, c10::DispatchKey::Functionalize,
                                   c10::DispatchKey::Negative, c10::DispatchKey::Conjugate,
                                   c10::DispatchKey::ZeroTensor});
    if (t.key_set().has_any(odd)) return nullptr;
    if (t.get_device() != w.device || t.numel() == 0) return nullptr;
    return &t;
}

// the same, contiguous and 1-D
const Tensor *vec(PyObject *o, const Where &w) {
    const Tensor *t = plain(o, w);
    if (!t || t->dim() != 1 || (t->numel() > 1 && t->stride(0) != 1)) return nullptr;
    return t;
}

bool same(const Tensor *a, const Tensor *b) { return a && b && a->scalar_type() == b->scalar_type(); }

at::ScalarType acc_type(const Tensor &t) {
    return t.scalar_type() == at::kDouble ? at::kDouble : at::kFloat;
}

bool number(PyObject *o, double *v) {
    *v = PyFloat_AsDouble(o);
    if (*v == -1.0 && PyErr_Occurred()) {
        PyErr_Clear();
        return false;
    }
    return true;
}

// A call's hold on the workspace of its (device, stream).  LAK_CALL gives the GIL up, and
// another thread on the same stream may then replace the kept workspace by a larger one:
// without a reference of the call's own its memory would go back to the allocator, and
// to another tensor of that stream, before the call has launched.
struct Workspace {
    Tensor hold;
    void *ptr() const { return hold.defined() ? hold.data_ptr() : nullptr; }
    size_t bytes() const { return hold.defined() ? (size_t)hold.numel() : 0; }
};

// False if the kept workspace has fewer than `need` bytes
bool workspace(const Where &w, size_t need, Workspace *ws) {
    if (need == 0) return true;
    const auto it = workspaces().find({w.device, w.handle});
    if (it == workspaces().end() || (size_t)it->second.numel() < need) return false;
    ws->hold = it->second;
    return true;
}

PyObject *none() { Py_RETURN_NONE; }

PyObject *given(PyObject *o) {
    Py_INCREF(o);
    return o;
}

// a one-element result: `out` if it fits, a new tensor if it is None
const Tensor *result_of(PyObject *out, const Where &w, at::ScalarType type, const Tensor &like,
                        bool scalar, Tensor *made) {
    if (out == Py_None) {
        *made = scalar ? at::empty({}, like.options().dtype(type)) : at::empty({1}, like.options().dtype(type));
        return made;
    }
    const Tensor *t = plain(out, w);
    return t && t->scalar_type() == type ? t : nullptr;
}

PyObject *give(PyObject *out, const Tensor &made) {
    return out == Py_None ? THPVariable_Wrap(made) : given(out);
}

#define LAK_CALL(expr)              \
    lak_status st;                  \
    Py_BEGIN_ALLOW_THREADS          \
    st = (expr);                    \
    Py_END_ALLOW_THREADS            \
    if (st != LAK_OK) return none()

#define LAK_FAST(name, nargs)                                                          \
    PyObject *name##_impl(PyObject *const *a);                                         \
    PyObject *name(PyObject *, PyObject *const *a, Py_ssize_t n) {                     \
        if (n != nargs) return none();                                                 \
        try {                                                                          \
            return name##_impl(a);                                                     \
        } catch (const std::exception &) {                                             \
            if (PyErr_Occurred()) PyErr_Clear();                                       \
            return none();                                                             \
        }                                                                              \
    }                                                                                  \
    PyObject *name##_impl(PyObject *const *a)

// (x, y)
LAK_FAST(fast_copy, 2) {
    const Where w = here();
    const Tensor *x = vec(a[0], w), *y = vec(a[1], w);
    if (!same(x, y) || x->numel() != y->numel()) return none();
    const int dt = storage_of(*x);
    if (dt < 0) return none();
    void *px = x->data_ptr(), *py = y->data_ptr();
    LAK_CALL(vec_copy(px, py, x->numel(), (lak_dtype)dt, nullptr, w.stream()));
    return given(a[0]);
}

// (x, y, z, alpha)
LAK_FAST(fast_axpy, 4) {
    const Where w = here();
    const Tensor *x = vec(a[0], w), *y = vec(a[1], w), *z = vec(a[2], w);
    double alpha;
    if (!same(x, y) || !same(x, z) || x->numel() != y->numel() || x->numel() != z->numel() ||
        !number(a[3], &alpha))
        return none();
    const int dt = storage_of(*x);
    if (dt < 0) return none();
    void *px = x->data_ptr(), *py = y->data_ptr(), *pz = z->data_ptr();
    LAK_CALL(vec_axpy(px, py, pz, alpha, x->numel(), (lak_dtype)dt, nullptr, w.stream()));
    return given(a[0]);
}

// (x, alpha, y, beta, z)
LAK_FAST(fast_axpby, 5) {
    const Where w = here();
    const Tensor *x = vec(a[0], w), *y = vec(a[2], w), *z = vec(a[4], w);
    double alpha, beta;
    if (!same(x, y) || !same(x, z) || x->numel() != y->numel() || x->numel() != z->numel() ||
        !number(a[1], &alpha) || !number(a[3], &beta))
        return none();
    const int dt = storage_of(*x);
    if (dt < 0) return none();
    void *px = x->data_ptr(), *py = y->data_ptr(), *pz = z->data_ptr();
    LAK_CALL(vec_axpby(px, alpha, py, beta, pz, x->numel(), (lak_dtype)dt, nullptr, w.stream()));
    return given(a[0]);
}

// (x, y, z, alpha, out or None)
LAK_FAST(fast_axpy_norm2, 5) {
    const Where w = here();
    const Tensor *x = vec(a[0], w), *y = vec(a[1], w), *z = vec(a[2], w);
    double alpha;
    if (!same(x, y) || !same(x, z) || x->numel() != y->numel() || x->numel() != z->numel() ||
        !number(a[3], &alpha))
        return none();
    const int dt = storage_of(*x);
    if (dt < 0) return none();
    Workspace ws;
    if (!workspace(w, vec_axpy_norm2_workspace(x->numel(), (lak_dtype)dt, nullptr), &ws))
        return none();
    Tensor made;
    const Tensor *out = result_of(a[4], w, acc_type(*x), *x, false, &made);
    if (!out) return none();
    void *px = x->data_ptr(), *py = y->data_ptr(), *pz = z->data_ptr(), *po = out->data_ptr();
    void *pws = ws.ptr();
    const size_t bytes = ws.bytes();
    LAK_CALL(vec_axpy_norm2(px, py, pz, alpha, po, x->numel(), (lak_dtype)dt, pws, bytes, nullptr, w.stream()));
    return give(a[4], made);
}

// (x, y, out or None, a new result is 0-d)
LAK_FAST(fast_dot, 4) {
    const Where w = here();
    const Tensor *x = vec(a[0], w), *y = vec(a[1], w);
    if (!same(x, y) || x->numel() != y->numel()) return none();
    const int dt = storage_of(*x);
    if (dt < 0) return none();
    Workspace ws;
    if (!workspace(w, vec_dot_workspace(x->numel(), (lak_dtype)dt, nullptr), &ws)) return none();
    Tensor made;
    const Tensor *out = result_of(a[2], w, acc_type(*x), *x, a[3] == Py_True, &made);
    if (!out) return none();
    void *px = x->data_ptr(), *py = y->data_ptr(), *po = out->data_ptr();
    void *pws = ws.ptr();
    const size_t bytes = ws.bytes();
    LAK_CALL(vec_dot(po, px, py, x->numel(), (lak_dtype)dt, pws, bytes, nullptr, w.stream()));
    return give(a[2], made);
}

// (x, y, out or None)
LAK_FAST(fast_dot_compensated, 3) {
    const Where w = here();
    const Tensor *x = vec(a[0], w), *y = vec(a[1], w);
    if (!same(x, y) || x->numel() != y->numel()) return none();
    const int dt = storage_of(*x);
    if (dt < 0 || dt == LAK_F64) return none();
    Workspace ws;
    if (!workspace(w, vec_dot_workspace(x->numel(), (lak_dtype)dt, nullptr), &ws)) return none();
    Tensor made;
    const Tensor *out = result_of(a[2], w, at::kDouble, *x, false, &made);
    if (!out) return none();
    void *px = x->data_ptr(), *py = y->data_ptr();
    double *po = static_cast<double *>(out->data_ptr());
    void *pws = ws.ptr();
    const size_t bytes = ws.bytes();
    LAK_CALL(vec_dot_compensated(po, px, py, x->numel(), (lak_dtype)dt, pws, bytes, nullptr, w.stream()));
    return give(a[2], made);
}

// (A, x, y or None, alpha, beta, transposed)
LAK_FAST(fast_gemv, 6) {
    const Where w = here();
    const Tensor *A = plain(a[0], w), *x = vec(a[1], w);
    double alpha, beta;
    if (!same(A, x) || A->dim() != 2 || !number(a[3], &alpha) || !number(a[4], &beta)) return none();
    const int dt = storage_of(*A);
    if (dt < 0) return none();
    const int64_t m = A->size(0), n = A->size(1), s0 = A->stride(0), s1 = A->stride(1);
    int64_t lda;
    lak_layout layout;
    if (s1 == 1 && (m <= 1 || s0 >= n)) {
        layout = LAK_ROW_MAJOR;
        lda = m > 1 ? s0 : n;
    } else if (s0 == 1 && (n <= 1 || s1 >= m)) {
        layout = LAK_COL_MAJOR;
        lda = n > 1 ? s1 : m;
    } else {
        return none();
    }
    const bool trans = a[5] == Py_True;
    const int64_t rows = trans ? n : m, cols = trans ? m : n;
    const lak_layout as = !trans ? layout : layout == LAK_ROW_MAJOR ? LAK_COL_MAJOR : LAK_ROW_MAJOR;
    if (x->numel() != cols) return none();
    Tensor made;
    const Tensor *y;
    if (a[2] == Py_None) {
        if (beta != 0.0) return none();
    } else {
        y = vec(a[2], w);
        if (!same(y, A) || y->numel() != rows) return none();
    }
    Workspace ws;
    const size_t need = dense_gemv_workspace(rows, cols, as, (lak_dtype)dt, nullptr);
    // a row-major product in a graph has scratch of the graph's own (Python path)
    if (need > 0 && as == LAK_ROW_MAJOR &&
        c10::cuda::currentStreamCaptureStatusMayInitCtx() != c10::cuda::CaptureStatus::None)
        return none();
    if (!workspace(w, need, &ws)) return none();
    if (a[2] == Py_None) {
        made = at::empty({rows}, A->options());
        y = &made;
    }
    void *py = y->data_ptr(), *pA = A->data_ptr(), *px = x->data_ptr();
    void *pws = ws.ptr();
    const size_t bytes = ws.bytes();
    LAK_CALL(alpha == 1.0 && beta == 0.0
                 ? dense_gemv(py, pA, px, rows, cols, lda, as, (lak_dtype)dt, pws, bytes, nullptr, w.stream())
                 : dense_gemv_axpby(py, alpha, pA, px, beta, rows, cols, lda, as, (lak_dtype)dt, pws, bytes,
                                    nullptr, w.stream()));
    return give(a[2], made);
}

// (row_ptr, col_idx, vals, x, y or None, n_cols or None)
LAK_FAST(fast_spmv, 6) {
    const Where w = here();
    const Tensor *rp = vec(a[0], w), *ci = vec(a[1], w), *v = vec(a[2], w), *x = vec(a[3], w);
    if (!rp || !ci || !same(v, x) || rp->scalar_type() != at::kInt || ci->scalar_type() != at::kInt ||
        ci->numel() != v->numel())
        return none();
    const int dt = storage_of(*v);
    const int64_t m = rp->numel() - 1;
    if (dt < 0 || m < 1) return none();
    int64_t n = x->numel();
    if (a[5] != Py_None) {
        n = PyLong_AsLongLong(a[5]);
        if (n == -1 && PyErr_Occurred()) {
            PyErr_Clear();
            return none();
        }
    }
    Tensor made;
    const Tensor *y;
    if (a[4] == Py_None) {
        made = at::empty({m}, v->options());
        y = &made;
    } else {
        y = vec(a[4], w);
        if (!same(y, v) || y->numel() != m) return none();
    }
    const int32_t *prp = static_cast<const int32_t *>(rp->data_ptr());
    const int32_t *pci = static_cast<const int32_t *>(ci->data_ptr());
    void *py = y->data_ptr(), *pv = v->data_ptr(), *px = x->data_ptr();
    LAK_CALL(csr_spmv(py, prp, pci, pv, px, m, n, v->numel(), (lak_dtype)dt, nullptr, w.stream()));
    return give(a[4], made);
}

// (dy, x) -> dy x^T
LAK_FAST(fast_outer, 2) {
    const Where w = here();
    const Tensor *dy = vec(a[0], w), *x = vec(a[1], w);
    if (!same(dy, x)) return none();
    const int dt = storage_of(*dy);
    if (dt < 0) return none();
    const int64_t m = dy->numel(), n = x->numel();
    Tensor made = at::empty({m, n}, dy->options());
    void *po = made.data_ptr(), *pd = dy->data_ptr(), *px = x->data_ptr();
    LAK_CALL(dense_outer(po, pd, px, m, n, n, (lak_dtype)dt, w.stream()));
    return THPVariable_Wrap(made);
}

// (row_ptr, col_idx, dy, x)
LAK_FAST(fast_sampled_outer, 4) {
    const Where w = here();
    const Tensor *rp = vec(a[0], w), *ci = vec(a[1], w), *dy = vec(a[2], w), *x = vec(a[3], w);
    if (!rp || !ci || !same(dy, x) || rp->scalar_type() != at::kInt || ci->scalar_type() != at::kInt)
        return none();
    const int dt = storage_of(*dy);
    const int64_t m = rp->numel() - 1;
    if (dt < 0 || m < 1) return none();
    Tensor made = at::empty({ci->numel()}, dy->options());
    const int32_t *prp = static_cast<const int32_t *>(rp->data_ptr());
    const int32_t *pci = static_cast<const int32_t *>(ci->data_ptr());
    void *po = made.data_ptr(), *pd = dy->data_ptr(), *px = x->data_ptr();
    LAK_CALL(csr_sampled_outer(po, prp, pci, pd, px, m, ci->numel(), (lak_dtype)dt, w.stream()));
    return THPVariable_Wrap(made);
}

// (v, alpha) -> alpha v, alpha a device element
LAK_FAST(fast_scale, 2) {
    const Where w = here();
    const Tensor *v = vec(a[0], w), *alpha = plain(a[1], w);
    if (!v || !alpha || alpha->scalar_type() != acc_type(*v)) return none();
    const int dt = storage_of(*v);
    if (dt < 0) return none();
    Tensor made = at::empty({v->numel()}, v->options());
    void *po = made.data_ptr(), *pv = v->data_ptr(), *pa = alpha->data_ptr();
    LAK_CALL(vec_scale_dev(po, pv, pa, v->numel(), (lak_dtype)dt, w.stream()));
    return THPVariable_Wrap(made);
}

// (device, stream, tensor): the workspace the Python side keeps for them
PyObject *keep_workspace(PyObject *, PyObject *const *a, Py_ssize_t n) {
    if (n != 3 || !THPVariable_Check(a[2])) {
        PyErr_SetString(PyExc_TypeError, "keep_workspace(device, stream, tensor)");
        return nullptr;
    }
    const long long device = PyLong_AsLongLong(a[0]), stream = PyLong_AsLongLong(a[1]);
    if (PyErr_Occurred()) return nullptr;
    workspaces()[{(int)device, (int64_t)stream}] = THPVariable_Unpack(a[2]);
    Py_RETURN_NONE;
}

#define LAK_DEF(name, fn) {name, (PyCFunction)(void (*)(void))fn, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    LAK_DEF("vec_copy", fast_copy),
    LAK_DEF("vec_axpy", fast_axpy),
    LAK_DEF("vec_axpby", fast_axpby),
    LAK_DEF("vec_axpy_norm2", fast_axpy_norm2),
    LAK_DEF("vec_dot", fast_dot),
    LAK_DEF("vec_dot_compensated", fast_dot_compensated),
    LAK_DEF("dense_gemv", fast_gemv),
    LAK_DEF("csr_spmv", fast_spmv),
    LAK_DEF("dense_outer", fast_outer),
    LAK_DEF("csr_sampled_outer", fast_sampled_outer),
    LAK_DEF("vec_scale_dev", fast_scale),
    LAK_DEF("keep_workspace", keep_workspace),
    {nullptr, nullptr, 0, nullptr},
};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fast", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fast(void) {
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "torch_version", LAK_TORCH_VERSION) < 0) Py_CLEAR(m);
    return m;
}
