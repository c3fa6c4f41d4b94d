// fem_marshal.cpp -- argument marshalling of the Python binding's entry points in native code.
//
// One call through ctypes costs about 25 us of host time on an Arm host (checks and pointers of
// five tensors, two host tables, the current stream, an output, 13 converted arguments), more
// than the kernels of all but the largest meshes take; here the same checks take about 1 us.
//
// Every function takes the binding function's arguments by position and either makes the C call
// and returns its result, or returns None without having done anything: some argument is not
// exactly what the call wants (another dtype, shape, device or layout, a table that is no
// contiguous float64 array, a tensor that gives no data pointer, an active torch function mode).
// binding.py then takes its own path, which converts what can be converted and raises the error
// that names the argument otherwise. A failing C call raises through binding._check. The C
// functions' addresses and _check are passed in once (init), so this module links no libfem.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/core/Tensor.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>
#include <initializer_list>

#include "../../include/fem.h"

namespace {

struct NotPlain {};  // thrown where the Python path has to look at the argument

void need(bool ok) {
    if (!ok) throw NotPlain();
}

// ------------------------------------------------------------------ the C functions

struct Functions {
    decltype(&fem_integrate_laplacian) integrate_laplacian;
    decltype(&fem_integrate_laplacian_fields) integrate_laplacian_fields;
    decltype(&fem_integrate_elasticity) integrate_elasticity;
    decltype(&fem_integrate_reaction_diffusion) integrate_reaction_diffusion;
    decltype(&fem_integrate_pointwise) integrate_pointwise;
    decltype(&fem_integrate_laplacian_geom) integrate_laplacian_geom;
    decltype(&fem_adjoint_laplacian) adjoint_laplacian;
    decltype(&fem_build_node2cell) build_node2cell;
    decltype(&fem_gather_nodes) gather_nodes;
    decltype(&fem_node2cell_work_size) node2cell_work_size;
} fn;
PyObject *check = nullptr;  // binding._check(name, status): raises
PyObject *stream_type = nullptr;  // torch.cuda.Stream

// ------------------------------------------------------------------ arguments

// a tensor argument: a CUDA tensor of this dtype, contiguous, with a data pointer
const at::Tensor &tensor(PyObject *o) {
    need(THPVariable_Check(o));
    return THPVariable_Unpack(o);
}
void *pointer(const at::Tensor &t, at::ScalarType dtype, std::initializer_list<int64_t> shape, c10::Device dev) {
    need(t.defined() && !t.unsafeGetTensorImpl()->is_python_dispatch());
    need(t.layout() == c10::kStrided && t.scalar_type() == dtype && t.device() == dev && dev.is_cuda());
    need(t.sizes().equals(c10::IntArrayRef(shape.begin(), shape.size())) && t.is_contiguous());
    return t.numel() ? t.data_ptr() : nullptr;
}

// a host table: a contiguous float64 buffer of rows x cols values (cols 0: a vector), copied
struct Table {
    double v[FEM_MAX_QPTS * 3];
    int64_t rows = 0;
    bool given = false;
    const double *ptr() const { return given ? v : nullptr; }
};
void table(PyObject *o, int64_t rows, int64_t cols, Table &t) {
    if (o == Py_None) return;
    need(PyObject_CheckBuffer(o) && !THPVariable_Check(o));
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS) != 0) {
        PyErr_Clear();
        throw NotPlain();
    }
    const int want = cols == 0 ? 1 : 2;
    bool ok = b.format && std::strcmp(b.format, "d") == 0 && b.ndim == want &&
              (rows < 0 ? b.shape[0] >= 1 && b.shape[0] <= FEM_MAX_QPTS : b.shape[0] == rows) &&
              (cols == 0 || b.shape[1] == cols);
    if (ok) {
        t.rows = b.shape[0];
        t.given = true;
        std::memcpy(t.v, b.buf, size_t(b.len));
    }
    PyBuffer_Release(&b);
    need(ok);
}

struct Rule {
    Table points, weights;
    int nq = 0;
};
void rule(PyObject *qpts, PyObject *qw, int dim, Rule &r) {
    table(qw, -1, 0, r.weights);
    need(r.weights.given);
    r.nq = static_cast<int>(r.weights.rows);
    table(qpts, r.nq, dim, r.points);
}

fem_precision precision(PyObject *o) {
    if (PyUnicode_Check(o)) {
        if (PyUnicode_CompareWithASCIIString(o, "mixed") == 0) return FEM_FP32_MIXED;
        if (PyUnicode_CompareWithASCIIString(o, "fp64") == 0) return FEM_FP64;
        if (PyUnicode_CompareWithASCIIString(o, "fp32") == 0) return FEM_FP32;
        if (PyUnicode_CompareWithASCIIString(o, "fp64_df") == 0) return FEM_FP64_DF;
        throw NotPlain();
    }
    need(PyLong_CheckExact(o));
    const long v = PyLong_AsLong(o);
    need(v >= 0 && v <= 3);
    return static_cast<fem_precision>(v);
}
at::ScalarType value_type(fem_precision p) { return p == FEM_FP64 || p == FEM_FP64_DF ? at::kDouble : at::kFloat; }

fem_stream stream(PyObject *o) {
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream().stream();
    const bool number = PyLong_CheckExact(o);
    if (!number && PyObject_IsInstance(o, stream_type) != 1) {
        PyErr_Clear();
        throw NotPlain();
    }
    PyObject *n = number ? Py_NewRef(o) : PyObject_GetAttrString(o, "cuda_stream");
    if (!n) {
        PyErr_Clear();
        throw NotPlain();
    }
    void *p = PyLong_Check(n) ? PyLong_AsVoidPtr(n) : nullptr;
    const bool ok = PyLong_Check(n) && !PyErr_Occurred();
    Py_DECREF(n);
    if (!ok) {
        PyErr_Clear();
        throw NotPlain();
    }
    return static_cast<fem_stream>(p);
}

int64_t integer(PyObject *o) {
    need(PyLong_CheckExact(o));
    const long long v = PyLong_AsLongLong(o);
    if (PyErr_Occurred()) {
        PyErr_Clear();
        throw NotPlain();
    }
    return v;
}

// an output or workspace: the caller's tensor, or a new one
at::Tensor made(PyObject *o, at::ScalarType dtype, std::initializer_list<int64_t> shape, c10::Device dev) {
    if (o != Py_None) return tensor(o);
    return at::empty(c10::IntArrayRef(shape.begin(), shape.size()), at::TensorOptions().dtype(dtype).device(dev));
}

struct MeshArgs {
    int dim;
    int64_t V, C;
    const double *coords;
    const int32_t *conn;
    c10::Device dev = c10::Device(c10::kCPU);
};
MeshArgs mesh(PyObject *coords, PyObject *conn) {
    const at::Tensor &x = tensor(coords), &c = tensor(conn);
    need(x.dim() == 2 && c.dim() == 2 && (x.size(0) == 2 || x.size(0) == 3) && c.size(0) == x.size(0) + 1);
    MeshArgs m;
    m.dim = static_cast<int>(x.size(0)), m.V = x.size(1), m.C = c.size(1);
    m.dev = x.device();
    m.coords = static_cast<const double *>(pointer(x, at::kDouble, {m.dim, m.V}, m.dev));
    m.conn = static_cast<const int32_t *>(pointer(c, at::kInt, {m.dim + 1, m.C}, m.dev));
    return m;
}

// ------------------------------------------------------------------ calls

// `body` marshals and calls: it returns the status and sets `result` to a new reference. The
// interpreter lock is released around the C call itself (as ctypes does): a launch may block.
template <class Body>
PyObject *guarded(const char *name, Py_ssize_t nargs, Py_ssize_t want, Body body) {
    if (nargs != want) {
        PyErr_Format(PyExc_TypeError, "%s: %zd arguments, %zd wanted", name, nargs, want);
        return nullptr;
    }
    if (at::impl::torch_function_mode_enabled()) Py_RETURN_NONE;
    PyObject *result = nullptr;
    try {
        const fem_status st = body(result);
        if (!result && PyErr_Occurred()) return nullptr;
        if (st != FEM_OK) {
            Py_CLEAR(result);
            PyObject *r = PyObject_CallFunction(check, "si", name, static_cast<int>(st));  // raises
            Py_XDECREF(r);
            if (!PyErr_Occurred()) PyErr_Format(PyExc_RuntimeError, "%s failed with status %d", name, static_cast<int>(st));
            return nullptr;
        }
        return result;
    } catch (...) {  // NotPlain, or a tensor that refused (fake, batched, undefined): the Python path says why
        Py_XDECREF(result);
        if (PyErr_Occurred()) PyErr_Clear();
        Py_RETURN_NONE;
    }
}

template <class F, class... A>
fem_status unlocked(F f, A... a) {
    fem_status st;
    Py_BEGIN_ALLOW_THREADS
    st = f(a...);
    Py_END_ALLOW_THREADS
    return st;
}

// coords, conn, u, K, qpts, qw, out, prec, stream
PyObject *laplacian(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_integrate_laplacian", n, 9, [&](PyObject *&result) {
        const MeshArgs m = mesh(a[0], a[1]);
        const fem_precision p = precision(a[7]);
        const at::ScalarType t = value_type(p);
        Rule q;
        rule(a[4], a[5], m.dim, q);
        void *u = pointer(tensor(a[2]), t, {m.V}, m.dev), *K = pointer(tensor(a[3]), t, {q.nq, m.C}, m.dev);
        const fem_stream s = stream(a[8]);
        const at::Tensor out = made(a[6], t, {m.dim + 1, m.C}, m.dev);
        void *o = pointer(out, t, {m.dim + 1, m.C}, m.dev);
        result = a[6] != Py_None ? Py_NewRef(a[6]) : THPVariable_Wrap(out);
        return unlocked(fn.integrate_laplacian, m.dim, m.C, m.V, m.coords, m.conn, u, K, q.nq, q.points.ptr(),
                        q.weights.ptr(), o, p, s);
    });
}

// coords, conn, u, K, qpts, qw, out, prec, stream
PyObject *laplacian_fields(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_integrate_laplacian_fields", n, 9, [&](PyObject *&result) {
        const MeshArgs m = mesh(a[0], a[1]);
        const fem_precision p = precision(a[7]);
        const at::ScalarType t = value_type(p);
        Rule q;
        rule(a[4], a[5], m.dim, q);
        const at::Tensor &ut = tensor(a[2]);
        need(ut.dim() == 2 && ut.size(0) < (int64_t(1) << 31));
        const int64_t nf = ut.size(0);
        void *u = pointer(ut, t, {nf, m.V}, m.dev), *K = pointer(tensor(a[3]), t, {q.nq, m.C}, m.dev);
        const fem_stream s = stream(a[8]);
        const at::Tensor out = made(a[6], t, {nf, m.dim + 1, m.C}, m.dev);
        void *o = pointer(out, t, {nf, m.dim + 1, m.C}, m.dev);
        result = a[6] != Py_None ? Py_NewRef(a[6]) : THPVariable_Wrap(out);
        return unlocked(fn.integrate_laplacian_fields, m.dim, m.C, m.V, m.coords, m.conn, static_cast<int>(nf), u, K,
                        q.nq, q.points.ptr(), q.weights.ptr(), o, p, s);
    });
}

// coords, conn, u, lam, mu, qpts, qw, out, prec, stream
PyObject *elasticity(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_integrate_elasticity", n, 10, [&](PyObject *&result) {
        const MeshArgs m = mesh(a[0], a[1]);
        const fem_precision p = precision(a[8]);
        const at::ScalarType t = value_type(p);
        Rule q;
        rule(a[5], a[6], m.dim, q);
        void *u = pointer(tensor(a[2]), t, {m.dim, m.V}, m.dev);
        void *lam = pointer(tensor(a[3]), t, {q.nq, m.C}, m.dev), *mu = pointer(tensor(a[4]), t, {q.nq, m.C}, m.dev);
        const fem_stream s = stream(a[9]);
        const int64_t rows = (m.dim + 1) * m.dim;
        const at::Tensor out = made(a[7], t, {rows, m.C}, m.dev);
        void *o = pointer(out, t, {rows, m.C}, m.dev);
        result = a[7] != Py_None ? Py_NewRef(a[7]) : THPVariable_Wrap(out);
        return unlocked(fn.integrate_elasticity, m.dim, m.C, m.V, m.coords, m.conn, u, lam, mu, q.nq, q.points.ptr(),
                        q.weights.ptr(), o, p, s);
    });
}

// coords, conn, u, a, qpts, qw, c, a_space, drift, out, prec, stream
PyObject *reaction(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_integrate_reaction_diffusion", n, 12, [&](PyObject *&result) {
        const MeshArgs m = mesh(a[0], a[1]);
        const fem_precision p = precision(a[10]);
        const at::ScalarType t = value_type(p);
        Rule q;
        need(a[4] != Py_None);
        rule(a[4], a[5], m.dim, q);
        const int64_t space = integer(a[7]);
        need(space == 0 || space == 1);
        need(PyFloat_CheckExact(a[8]) || PyLong_CheckExact(a[8]));
        const double drift = PyFloat_AsDouble(a[8]);
        need(!PyErr_Occurred());
        void *u = pointer(tensor(a[2]), t, {m.V}, m.dev);
        void *af = pointer(tensor(a[3]), t, {space == 1 ? m.V : m.C}, m.dev);
        void *c = a[6] == Py_None ? nullptr : pointer(tensor(a[6]), t, {q.nq, m.C}, m.dev);
        const fem_stream s = stream(a[11]);
        const at::Tensor out = made(a[9], t, {m.dim + 1, m.C}, m.dev);
        void *o = pointer(out, t, {m.dim + 1, m.C}, m.dev);
        result = a[9] != Py_None ? Py_NewRef(a[9]) : THPVariable_Wrap(out);
        return unlocked(fn.integrate_reaction_diffusion, m.dim, m.C, m.V, m.coords, m.conn, u, af,
                        static_cast<int>(space), c, drift, q.nq, q.points.ptr(), q.weights.ptr(), o, p, s);
    });
}

// coords, conn, u, coef, qpts, qw, f1, f0, out, prec, stream
PyObject *pointwise(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_integrate_pointwise", n, 11, [&](PyObject *&result) {
        const MeshArgs m = mesh(a[0], a[1]);
        const fem_precision p = precision(a[9]);
        const at::ScalarType t = value_type(p);
        Rule q;
        rule(a[4], a[5], m.dim, q);
        const char *src[2] = {nullptr, nullptr};  // f0, f1
        for (int i = 0; i < 2; ++i) {
            PyObject *f = a[7 - i];
            if (f == Py_None) continue;
            need(PyUnicode_Check(f));
            src[i] = PyUnicode_AsUTF8(f);
            need(src[i] != nullptr);
        }
        const at::Tensor &ut = tensor(a[2]);
        need(ut.dim() == 1 || (ut.dim() == 2 && ut.size(0) < (int64_t(1) << 31)));
        const int64_t nc = ut.dim() == 1 ? 1 : ut.size(0);
        void *u = ut.dim() == 1 ? pointer(ut, t, {m.V}, m.dev) : pointer(ut, t, {nc, m.V}, m.dev);
        int64_t ncoef = 0;
        void *coef = nullptr;
        if (a[3] != Py_None) {
            const at::Tensor &ct = tensor(a[3]);
            need(ct.dim() == 3 && ct.size(0) < (int64_t(1) << 31));
            ncoef = ct.size(0);
            coef = pointer(ct, t, {ncoef, q.nq, m.C}, m.dev);
        }
        const fem_stream s = stream(a[10]);
        const int64_t rows = (m.dim + 1) * nc;
        const at::Tensor out = made(a[8], t, {rows, m.C}, m.dev);
        void *o = pointer(out, t, {rows, m.C}, m.dev);
        result = a[8] != Py_None ? Py_NewRef(a[8]) : THPVariable_Wrap(out);
        return unlocked(fn.integrate_pointwise, src[0], src[1], m.dim, static_cast<int>(nc), static_cast<int>(ncoef),
                        m.C, m.V, m.coords, m.conn, u, coef, q.nq, q.points.ptr(), q.weights.ptr(), o, p, s);
    });
}

// conn, n_verts, u, K, qpts, qw, geom, out, prec, stream
PyObject *laplacian_geom(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_integrate_laplacian_geom", n, 10, [&](PyObject *&result) {
        const at::Tensor &c = tensor(a[0]);
        need(c.dim() == 2 && (c.size(0) == 3 || c.size(0) == 4));
        const int dim = static_cast<int>(c.size(0)) - 1;
        const int64_t C = c.size(1), V = integer(a[1]);
        need(V >= 0);
        const c10::Device dev = c.device();
        const fem_precision p = precision(a[8]);
        const at::ScalarType t = value_type(p);
        const int32_t *conn = static_cast<const int32_t *>(pointer(c, at::kInt, {dim + 1, C}, dev));
        Rule q;
        rule(a[4], a[5], dim, q);
        void *u = pointer(tensor(a[2]), t, {V}, dev), *K = pointer(tensor(a[3]), t, {q.nq, C}, dev);
        void *g = pointer(tensor(a[6]), t, {dim * dim + 1, C}, dev);
        const fem_stream s = stream(a[9]);
        const at::Tensor out = made(a[7], t, {dim + 1, C}, dev);
        void *o = pointer(out, t, {dim + 1, C}, dev);
        result = a[7] != Py_None ? Py_NewRef(a[7]) : THPVariable_Wrap(out);
        return unlocked(fn.integrate_laplacian_geom, dim, C, V, conn, u, K, q.nq, q.points.ptr(), q.weights.ptr(), g, o,
                        p, s);
    });
}

// coords, conn, u, K, qpts, qw, lam_adj, node_ptr, node_idx, dK, du, scratch, prec, stream
PyObject *adjoint(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_adjoint_laplacian", n, 14, [&](PyObject *&result) {
        const MeshArgs m = mesh(a[0], a[1]);
        const fem_precision p = precision(a[12]);
        const at::ScalarType t = value_type(p);
        Rule q;
        rule(a[4], a[5], m.dim, q);
        const int64_t nb = m.dim + 1;
        void *u = pointer(tensor(a[2]), t, {m.V}, m.dev), *K = pointer(tensor(a[3]), t, {q.nq, m.C}, m.dev);
        void *lam = pointer(tensor(a[6]), t, {nb, m.C}, m.dev);
        const int32_t *ptr = static_cast<const int32_t *>(pointer(tensor(a[7]), at::kInt, {m.V + 1}, m.dev));
        const int32_t *idx = static_cast<const int32_t *>(pointer(tensor(a[8]), at::kInt, {nb * m.C}, m.dev));
        const fem_stream s = stream(a[13]);
        const at::Tensor dK = made(a[9], t, {q.nq, m.C}, m.dev), du = made(a[10], t, {m.V}, m.dev);
        const at::Tensor scratch = made(a[11], t, {nb, m.C}, m.dev);
        void *pK = pointer(dK, t, {q.nq, m.C}, m.dev), *pu = pointer(du, t, {m.V}, m.dev);
        void *ps = pointer(scratch, t, {nb, m.C}, m.dev);
        PyObject *oK = a[9] != Py_None ? Py_NewRef(a[9]) : THPVariable_Wrap(dK);
        PyObject *ou = a[10] != Py_None ? Py_NewRef(a[10]) : THPVariable_Wrap(du);
        if (oK && ou) result = PyTuple_Pack(2, oK, ou);
        Py_XDECREF(oK);
        Py_XDECREF(ou);
        return unlocked(fn.adjoint_laplacian, m.dim, m.C, m.V, m.coords, m.conn, u, K, q.nq, q.points.ptr(),
                        q.weights.ptr(), lam, pK, pu, ptr, idx, ps, p, s);
    });
}

// conn, n_verts, node_ptr, node_idx, work, stream
PyObject *node2cell(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_build_node2cell", n, 6, [&](PyObject *&result) {
        const at::Tensor &c = tensor(a[0]);
        need(c.dim() == 2 && (c.size(0) == 3 || c.size(0) == 4));
        const int dim = static_cast<int>(c.size(0)) - 1;
        const int64_t C = c.size(1), V = integer(a[1]);
        need(V >= 0);
        const c10::Device dev = c.device();
        const int32_t *conn = static_cast<const int32_t *>(pointer(c, at::kInt, {dim + 1, C}, dev));
        const int64_t want = fn.node2cell_work_size(V);
        const fem_stream s = stream(a[5]);
        const at::Tensor ptr = made(a[2], at::kInt, {V + 1}, dev), idx = made(a[3], at::kInt, {(dim + 1) * C}, dev);
        const at::Tensor work = made(a[4], at::kInt, {want > 1 ? want : 1}, dev);
        need(work.dim() == 1 && work.numel() >= want);
        int32_t *pp = static_cast<int32_t *>(pointer(ptr, at::kInt, {V + 1}, dev));
        int32_t *pi = static_cast<int32_t *>(pointer(idx, at::kInt, {(dim + 1) * C}, dev));
        int32_t *pw = static_cast<int32_t *>(pointer(work, at::kInt, {work.size(0)}, dev));
        PyObject *op = a[2] != Py_None ? Py_NewRef(a[2]) : THPVariable_Wrap(ptr);
        PyObject *oi = a[3] != Py_None ? Py_NewRef(a[3]) : THPVariable_Wrap(idx);
        if (op && oi) result = PyTuple_Pack(2, op, oi);
        Py_XDECREF(op);
        Py_XDECREF(oi);
        return unlocked(fn.build_node2cell, dim, C, V, conn, pp, pi, pw, s);
    });
}

// elem, node_ptr, node_idx, n_verts, dim, out, prec, stream
PyObject *gather(PyObject *, PyObject *const *a, Py_ssize_t n) {
    return guarded("fem_gather_nodes", n, 8, [&](PyObject *&result) {
        const at::Tensor &e = tensor(a[0]);
        const int64_t V = integer(a[3]), dim = integer(a[4]);
        need(e.dim() == 2 && V >= 0 && (dim == 2 || dim == 3) && e.size(0) >= dim + 1 && e.size(0) % (dim + 1) == 0 &&
             e.size(0) <= 1024);
        const int64_t nc = e.size(0) / (dim + 1), C = e.size(1);
        const c10::Device dev = e.device();
        const fem_precision p = precision(a[6]);
        const at::ScalarType t = value_type(p);
        void *el = pointer(e, t, {e.size(0), C}, dev);
        const int32_t *ptr = static_cast<const int32_t *>(pointer(tensor(a[1]), at::kInt, {V + 1}, dev));
        const int32_t *idx = static_cast<const int32_t *>(pointer(tensor(a[2]), at::kInt, {(dim + 1) * C}, dev));
        const fem_stream s = stream(a[7]);
        const at::Tensor out = made(a[5], t, {nc, V}, dev);
        void *o = pointer(out, t, {nc, V}, dev);
        result = a[5] != Py_None ? Py_NewRef(a[5]) : THPVariable_Wrap(out);
        return unlocked(fn.gather_nodes, static_cast<int>(dim), static_cast<int>(nc), C, V, el, ptr, idx, o, p, s);
    });
}

// ------------------------------------------------------------------ module

template <class F>
bool address(PyObject *d, const char *name, F &f) {
    PyObject *o = PyDict_GetItemString(d, name);
    void *p = o ? PyLong_AsVoidPtr(o) : nullptr;
    if (!p) {
        if (!PyErr_Occurred()) PyErr_Format(PyExc_KeyError, "no address of %s", name);
        return false;
    }
    f = reinterpret_cast<F>(p);
    return true;
}

// init(check, torch.cuda.Stream, {name: address})
PyObject *init(PyObject *, PyObject *args) {
    PyObject *c, *t, *d;
    if (!PyArg_ParseTuple(args, "OO!O!", &c, &PyType_Type, &t, &PyDict_Type, &d)) return nullptr;
    if (!address(d, "fem_integrate_laplacian", fn.integrate_laplacian) ||
        !address(d, "fem_integrate_laplacian_fields", fn.integrate_laplacian_fields) ||
        !address(d, "fem_integrate_elasticity", fn.integrate_elasticity) ||
        !address(d, "fem_integrate_reaction_diffusion", fn.integrate_reaction_diffusion) ||
        !address(d, "fem_integrate_pointwise", fn.integrate_pointwise) ||
        !address(d, "fem_integrate_laplacian_geom", fn.integrate_laplacian_geom) ||
        !address(d, "fem_adjoint_laplacian", fn.adjoint_laplacian) ||
        !address(d, "fem_build_node2cell", fn.build_node2cell) || !address(d, "fem_gather_nodes", fn.gather_nodes) ||
        !address(d, "fem_node2cell_work_size", fn.node2cell_work_size))
        return nullptr;
    Py_XSETREF(check, Py_NewRef(c));
    Py_XSETREF(stream_type, Py_NewRef(t));
    Py_RETURN_NONE;
}

#define FAST(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {{"init", init, METH_VARARGS, nullptr},
                         FAST(laplacian),
                         FAST(laplacian_fields),
                         FAST(elasticity),
                         FAST(reaction),
                         FAST(pointwise),
                         FAST(laplacian_geom),
                         FAST(adjoint),
                         FAST(node2cell),
                         FAST(gather),
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", "native argument marshalling (fem_marshal.cpp)", -1, methods};

}  // namespace

// built_for: the torch and interpreter this was compiled against (build.marshal_stamp()); the
// binding uses the module only where they are the running ones
PyMODINIT_FUNC PyInit__marshal() {
    PyObject *m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", FEM_MARSHAL_BUILT_FOR) != 0) Py_CLEAR(m);
    return m;
}
