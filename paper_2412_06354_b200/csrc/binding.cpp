// CPython extension behind gnn.py: unpacks tensors, allocates outputs and workspaces and calls the C ABI.
//
// A call on a small graph is bound by the host: through ctypes and torch.empty a call of the library cost 12-17 us of
// Python (argument conversion, three allocations, the current stream) beside 2-3 us per kernel launch.  Here a call
// costs well under a microsecond beyond its allocations and launches.  Nothing is computed in this file.
//
// Allocation: outputs and workspaces come from torch's caching allocator, on the device of the inputs and the current
// stream, exactly as torch.empty would take them.  If the binding module's `torch` attribute has been replaced (an
// allocation checker standing in for it), every allocation goes through that object's empty() instead.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/DynamicTypes.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include "gnn.h"

namespace {

PyObject* g_module_dict = nullptr;  // of the Python module that offers the calls (holds its `torch` and GnnError)
PyObject* g_real_torch = nullptr;
PyObject* g_s_torch = nullptr;
PyObject* g_s_empty = nullptr;
PyObject* g_error = nullptr;

// the Python error that is set, as an exception
[[noreturn]] void rethrow() {
    python_error e;
    e.persist();
    throw e;
}

[[noreturn]] void raise(PyObject* type, const std::string& text) {
    PyErr_SetString(type, text.c_str());
    rethrow();
}

// int(o), float(o) and bool(o)
int64_t as_int(PyObject* o) {
    PyObject* n = PyNumber_Long(o);
    const int64_t v = n ? PyLong_AsLongLong(n) : -1;
    Py_XDECREF(n);
    if (v == -1 && PyErr_Occurred()) rethrow();
    return v;
}
double as_float(PyObject* o) {
    PyObject* n = PyNumber_Float(o);
    const double v = n ? PyFloat_AS_DOUBLE(n) : -1.0;
    Py_XDECREF(n);
    if (!n) rethrow();
    return v;
}
bool as_bool(PyObject* o) {
    const int v = PyObject_IsTrue(o);
    if (v < 0) rethrow();
    return v == 1;
}

// status of a C-ABI call -> GnnError(status, text)
void check(gnn_status rc) {
    if (rc == GNN_OK) return;
    PyObject* args = Py_BuildValue("(is)", (int)rc, gnn_last_error_string());
    if (args) {
        PyObject* exc = PyObject_CallObject(g_error, args);
        Py_DECREF(args);
        if (exc) {
            PyErr_SetObject(g_error, exc);
            Py_DECREF(exc);
        }
    }
    rethrow();
}

// a launch can block (a full queue, a synchronising call): other Python threads keep running meanwhile
#define CALL(expr)                      \
    do {                                \
        gnn_status rc_;                 \
        Py_BEGIN_ALLOW_THREADS          \
        rc_ = (expr);                   \
        Py_END_ALLOW_THREADS            \
        check(rc_);                     \
    } while (0)

gnn_stream stream() { return (gnn_stream)c10::cuda::getCurrentCUDAStream().stream(); }

// ---------------------------------------------------------------- arguments
struct Args {
    PyObject* const* a;
    Py_ssize_t n;
    PyObject* at(int i) const {
        if (i >= n) raise(PyExc_TypeError, "missing argument");
        return a[i];
    }
    bool none(int i) const { return at(i) == Py_None; }
    // a tensor, or an undefined one for None
    const at::Tensor& t(int i) const {
        static const at::Tensor undefined;
        PyObject* o = at(i);
        if (o == Py_None) return undefined;
        if (!THPVariable_Check(o)) raise(PyExc_TypeError, std::string("expected a tensor or None, got ") + Py_TYPE(o)->tp_name);
        return THPVariable_Unpack(o);
    }
    // a tensor that the call cannot do without
    const at::Tensor& must(int i) const {
        if (none(i)) raise(PyExc_AttributeError, "a tensor is needed, got None");
        return t(i);
    }
    // a contiguous tensor on the device
    const at::Tensor& dev(int i) const {
        const at::Tensor& x = t(i);
        if (!x.defined() || !x.is_cuda() || !x.is_contiguous()) raise(PyExc_AssertionError, "CUDA contiguous tensor expected");
        return x;
    }
    int64_t i(int k) const {
        const int64_t v = PyLong_AsLongLong(at(k));
        if (v == -1 && PyErr_Occurred()) rethrow();
        return v;
    }
    bool flag(int k) const { return as_bool(at(k)); }
    float f(int k) const { return (float)as_float(at(k)); }
    gnn_op op(int k) const {
        PyObject* o = at(k);
        if (PyUnicode_Check(o)) {
            static const char* const names[4] = {"sum", "mean", "max", "min"};
            for (int q = 0; q < 4; ++q)
                if (PyUnicode_CompareWithASCIIString(o, names[q]) == 0) return (gnn_op)q;
            PyErr_SetObject(PyExc_KeyError, o);
            rethrow();
        }
        return (gnn_op)as_int(o);
    }
    // heads of a row of F features: their number, and the features of one
    int heads(int k, int64_t F, int* C) const {
        const int64_t H = i(k);
        if (H == 0) raise(PyExc_ZeroDivisionError, "the number of heads is zero");
        const int64_t q = F / H;
        *C = (int)(F % H != 0 && (F < 0) != (H < 0) ? q - 1 : q);
        return (int)H;
    }
    const gnn_csr* g(int k) const { return reinterpret_cast<const gnn_csr*>((intptr_t)i(k)); }
};

void* ptr(const at::Tensor& t) { return t.defined() ? t.data_ptr() : nullptr; }

// pointer of a tensor whose element type the C ABI takes for granted
void* typed(const at::Tensor& t, at::ScalarType type, const char* name) {
    if (!t.defined()) return nullptr;
    if (t.scalar_type() != type) raise(PyExc_TypeError, std::string(name) + " must be torch." + (type == at::kFloat ? "float32" : type == at::kInt ? "int32" : "int64") + ", got " + c10::toString(t.scalar_type()));
    if (t.numel() && !t.is_contiguous()) raise(PyExc_TypeError, std::string(name) + " must be contiguous");
    return t.data_ptr();
}
float* f32(const at::Tensor& t, const char* name) { return (float*)typed(t, at::kFloat, name); }
int32_t* i32(const at::Tensor& t, const char* name) { return (int32_t*)typed(t, at::kInt, name); }
int64_t* i64(const at::Tensor& t, const char* name) { return (int64_t*)typed(t, at::kLong, name); }

gnn_dtype dtype_of(const at::Tensor& t) {
    if (t.scalar_type() == at::kFloat) return GNN_F32;
    if (t.scalar_type() == at::kBFloat16) return GNN_BF16;
    raise(PyExc_TypeError, std::string("unsupported feature dtype ") + c10::toString(t.scalar_type()));
}

// ---------------------------------------------------------------- allocation
at::Tensor empty(at::IntArrayRef shape, at::ScalarType type, c10::Device device) {
    PyObject* torch = PyDict_GetItem(g_module_dict, g_s_torch);
    if (torch == g_real_torch) return at::detail::empty_cuda(shape, type, device, std::nullopt);
    PyObject* fn = torch ? PyObject_GetAttr(torch, g_s_empty) : nullptr;
    PyObject* args = fn ? PyTuple_New(1) : nullptr;
    PyObject* kw = args ? PyDict_New() : nullptr;
    PyObject* r = nullptr;
    if (kw) {
        PyObject* sh = PyTuple_New((Py_ssize_t)shape.size());
        for (size_t k = 0; sh && k < shape.size(); ++k) PyTuple_SET_ITEM(sh, (Py_ssize_t)k, PyLong_FromLongLong(shape[k]));
        PyTuple_SET_ITEM(args, 0, sh);
        PyObject* dt = (PyObject*)torch::getTHPDtype(type);
        PyObject* dv = THPDevice_New(device);
        if (sh && dv && PyDict_SetItemString(kw, "dtype", dt) == 0 && PyDict_SetItemString(kw, "device", dv) == 0) r = PyObject_Call(fn, args, kw);
        Py_XDECREF(dv);
    }
    Py_XDECREF(kw);
    Py_XDECREF(args);
    Py_XDECREF(fn);
    if (!r || !THPVariable_Check(r)) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "empty() gave no tensor");
        Py_XDECREF(r);
        rethrow();
    }
    at::Tensor t = THPVariable_Unpack(r);
    Py_DECREF(r);
    return t;
}

at::Tensor empty_like(const at::Tensor& x) { return empty(x.sizes(), x.scalar_type(), x.device()); }

// scratch of one call: the caller's tensor, or memory of the caching allocator that goes back when the call has been
// enqueued (its next user on this stream comes after it in stream order)
struct Scratch {
    c10::DataPtr own;
    at::Tensor kept;
    void* p;
    size_t n;
    Scratch(const at::Tensor& given, size_t need, c10::Device device) {
        if (given.defined()) {
            p = given.data_ptr();
            n = (size_t)given.numel();
            return;
        }
        n = need;
        if (PyDict_GetItem(g_module_dict, g_s_torch) == g_real_torch) {
            c10::cuda::OptionalCUDAGuard guard;
            if (device.index() != c10::cuda::current_device()) guard.set_device(device);
            own = c10::cuda::CUDACachingAllocator::get()->allocate(need);
            p = own.get();
        } else {
            kept = empty({(int64_t)need}, at::kByte, device);
            p = kept.data_ptr();
        }
    }
};

// ---------------------------------------------------------------- results
PyObject* wrap(const at::Tensor& t) {
    if (!t.defined()) Py_RETURN_NONE;
    return THPVariable_Wrap(t);
}
template <class... Ts>
PyObject* wrap_all(const Ts&... ts) {
    PyObject* r = PyTuple_New((Py_ssize_t)sizeof...(ts));
    if (!r) return nullptr;
    Py_ssize_t k = 0;
    (PyTuple_SET_ITEM(r, k++, wrap(ts)), ...);
    return r;
}

// edge-aligned result: buffers hold at least one row, the result has E
at::Tensor first(const at::Tensor& t, int64_t E) { return t.defined() && t.size(0) != E ? t.narrow(0, 0, E) : t; }
int64_t at_least_one(int64_t n) { return n > 0 ? n : 1; }

#define FN(name)                                                                  \
    static PyObject* name##_impl(const Args& A);                                  \
    static PyObject* name(PyObject*, PyObject* const* args, Py_ssize_t nargs) {   \
        HANDLE_TH_ERRORS                                                          \
        return name##_impl(Args{args, nargs});                                    \
        END_HANDLE_TH_ERRORS                                                      \
    }                                                                             \
    static PyObject* name##_impl(const Args& A)

// ---------------------------------------------------------------- graph set-up
// (N, src, dst, ws) -> (rowptr, rowptrT, col, eid, colT, eidT, t2f)
FN(coo_to_csr) {
    const int64_t N = A.i(0);
    const at::Tensor &src = A.dev(1), &dst = A.dev(2);
    const int64_t E = src.numel(), n = at_least_one(E);
    const auto dev = src.device();
    at::Tensor rp = empty({N + 1}, at::kLong, dev), rpT = empty({N + 1}, at::kLong, dev);
    at::Tensor x[5];
    for (auto& t : x) t = empty({n}, at::kInt, dev);
    gnn_csr g;
    g.rowptr = (int64_t*)ptr(rp); g.rowptrT = (int64_t*)ptr(rpT);
    g.col = (int32_t*)ptr(x[0]); g.eid = (int32_t*)ptr(x[1]); g.colT = (int32_t*)ptr(x[2]); g.eidT = (int32_t*)ptr(x[3]); g.t2f = (int32_t*)ptr(x[4]);
    Scratch ws(A.t(3), gnn_coo_to_csr_workspace((int32_t)N, E), dev);
    const int32_t *s = i32(src, "src"), *d = i32(dst, "dst");
    const gnn_stream st = stream();
    CALL(gnn_coo_to_csr((int32_t)N, E, s, d, &g, ws.p, ws.n, st));
    return wrap_all(rp, rpT, x[0], x[1], x[2], x[3], x[4]);
}

// (g, transposed, w, rowptr)
FN(degree) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& w = A.t(2);
    at::Tensor out = empty({g->N}, w.defined() ? at::kFloat : at::kInt, A.t(3).device());
    const int tr = (int)as_int(A.at(1));
    const gnn_stream st = stream();
    CALL(gnn_degree(g, tr, (const float*)ptr(w), ptr(out), st));
    return wrap(out);
}

// (N, src, dst) -> (src, dst)
FN(add_self_loops) {
    const int64_t N = A.i(0);
    const at::Tensor &src = A.must(1), &dst = A.t(2);
    const int64_t E = src.numel();
    at::Tensor so = empty({E + N}, at::kInt, src.device()), d_o = empty({E + N}, at::kInt, src.device());
    const int32_t *s = i32(src, "src"), *d = i32(dst, "dst");
    const gnn_stream st = stream();
    CALL(gnn_add_self_loops((int32_t)N, E, s, d, (int32_t*)ptr(so), (int32_t*)ptr(d_o), st));
    return wrap_all(so, d_o);
}

// (g, w_csr, want_T, rowptr) -> (deg, coef, coefT or None)
FN(gcn_norm) {
    const gnn_csr* g = A.g(0);
    const auto dev = A.t(3).device();
    at::Tensor deg = empty({g->N}, at::kFloat, dev), coef = empty({at_least_one(g->E)}, at::kFloat, dev), coefT;
    if (A.flag(2)) coefT = empty({at_least_one(g->E)}, at::kFloat, dev);
    const float* w = f32(A.t(1), "w_csr");
    const gnn_stream st = stream();
    CALL(gnn_gcn_norm(g, w, (float*)ptr(deg), (float*)ptr(coef), (float*)ptr(coefT), st));
    return wrap_all(deg, first(coef, g->E), first(coefT, g->E));
}

// (perm, x, out)
FN(permute_edge_data) {
    const at::Tensor &perm = A.must(0), &x = A.dev(1);
    at::Tensor out = A.t(2);
    const int64_t E = perm.numel(), width = E ? x.numel() / E : 1;
    if (!out.defined()) out = empty_like(x);
    const int32_t* p = i32(perm, "perm");
    const gnn_stream st = stream();
    CALL(gnn_permute_edge_data(p, E, (int)at_least_one(width), (int)x.element_size(), ptr(x), ptr(out), st));
    return wrap(out);
}

// (g, seg_csr, seg_is_mean, w_csr, want_T, rowptr) -> (coef, coefT or None)
FN(segment_coef) {
    const gnn_csr* g = A.g(0);
    const auto dev = A.t(5).device();
    at::Tensor coef = empty({at_least_one(g->E)}, at::kFloat, dev), coefT;
    if (A.flag(4)) coefT = empty({at_least_one(g->E)}, at::kFloat, dev);
    const int32_t *seg = i32(A.t(1), "seg_csr"), *mean = i32(A.t(2), "seg_is_mean");
    const float* w = f32(A.t(3), "w_csr");
    const int S = (int)A.must(2).numel();
    const gnn_stream st = stream();
    CALL(gnn_segment_coef(g, seg, w, mean, S, (float*)ptr(coef), (float*)ptr(coefT), st));
    return wrap_all(first(coef, g->E), first(coefT, g->E));
}

// ([(src, dst, src_offset, dst_offset), ...]) -> (src, dst, seg)
FN(merge_edge_lists) {
    PyObject* seq = PySequence_Fast(A.at(0), "segments must be a sequence");
    if (!seq) rethrow();
    const Py_ssize_t S = PySequence_Fast_GET_SIZE(seq);
    std::vector<gnn_edge_segment> segs((size_t)S);
    int64_t total = 0;
    c10::Device dev(c10::kCUDA);
    try {
        for (Py_ssize_t k = 0; k < S; ++k) {
            PyObject* item = PySequence_Fast(PySequence_Fast_GET_ITEM(seq, k), "a segment is (src, dst, src_offset, dst_offset)");
            if (!item) rethrow();
            const Args B{PySequence_Fast_ITEMS(item), PySequence_Fast_GET_SIZE(item)};
            try {
                if (B.n != 4) raise(PyExc_ValueError, "a segment is (src, dst, src_offset, dst_offset)");
                const at::Tensor &src = B.must(0), &dst = B.must(1);
                segs[(size_t)k] = gnn_edge_segment{src.numel(), src.numel() ? i32(src, "src") : nullptr, dst.numel() ? i32(dst, "dst") : nullptr,
                                                   (int32_t)as_int(B.at(2)), (int32_t)as_int(B.at(3))};
                if (k == 0) dev = src.device();
                total += src.numel();
            } catch (...) { Py_DECREF(item); throw; }
            Py_DECREF(item);
        }
    } catch (...) { Py_DECREF(seq); throw; }
    Py_DECREF(seq);
    if (S == 0) raise(PyExc_IndexError, "list index out of range");
    at::Tensor x[3];
    for (auto& t : x) t = empty({at_least_one(total)}, at::kInt, dev);
    const gnn_stream st = stream();
    CALL(gnn_merge_edge_lists(segs.data(), (int)S, (int32_t*)ptr(x[0]), (int32_t*)ptr(x[1]), (int32_t*)ptr(x[2]), st));
    return wrap_all(first(x[0], total), first(x[1], total), first(x[2], total));
}

// (graph_id, G) -> graph_ptr
FN(graph_ptr_from_ids) {
    const at::Tensor& id = A.must(0);
    const int64_t G = A.i(1);
    at::Tensor out = empty({G + 1}, at::kLong, id.device());
    Scratch ws(at::Tensor(), 256, id.device());
    const int32_t* p = i32(id, "graph_id");
    const gnn_stream st = stream();
    CALL(gnn_graph_ptr_from_ids(p, (int32_t)id.numel(), (int32_t)G, (int64_t*)ptr(out), ws.p, ws.n, st));
    return wrap(out);
}

// ---------------------------------------------------------------- fused propagate
static bool has_winners(gnn_op op) { return op == GNN_MAX || op == GNN_MIN; }

// (g, X, w_csr, op, out, argmax, ws, built_in) -> out or (out, argmax); built_in: the call without a workspace argument
FN(propagate_fused) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& X = A.dev(1);
    const at::Tensor& w = A.t(2);
    const gnn_op op = A.op(3);
    at::Tensor out = A.t(4), arg = A.t(5);
    const int64_t F = X.size(1);
    if (!out.defined()) out = empty({g->N, F}, X.scalar_type(), X.device());
    if (has_winners(op) && !arg.defined()) arg = empty({g->N, F}, at::kInt, X.device());
    const gnn_msg msg = w.defined() ? GNN_MSG_E_MUL_XJ : GNN_MSG_COPY_XJ;
    const float* wp = f32(w, "w_csr");
    int32_t* ap = i32(arg, "argmax");
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    if (A.flag(7)) {
        CALL(gnn_propagate_fused_static(g, msg, op, ptr(X), wp, (int)F, dt, ptr(out), ap, st));
    } else {
        Scratch ws(A.t(6), gnn_propagate_fused_workspace(g->E, (int)F, op), X.device());
        CALL(gnn_propagate_fused(g, msg, op, ptr(X), wp, (int)F, dt, ptr(out), ap, ws.p, ws.n, st));
    }
    return has_winners(op) ? wrap_all(out, arg) : wrap(out);
}

// (g, dOut, op, X, w_csrT, argmax, want_dX, want_dW, dX, dW, ws) -> (dX, dW)
FN(propagate_fused_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& dO = A.dev(1);
    const gnn_op op = A.op(2);
    const at::Tensor &X = A.t(3), &w = A.t(4), &arg = A.t(5);
    const bool want_dX = A.flag(6), want_dW = A.flag(7);
    at::Tensor dX, dW;
    const int64_t F = dO.size(1);
    if (want_dX) {
        dX = A.t(8);
        if (!dX.defined()) dX = empty({g->N, F}, dO.scalar_type(), dO.device());
    }
    if (want_dW) {
        dW = A.t(9);
        if (!dW.defined()) dW = empty({at_least_one(g->E)}, at::kFloat, dO.device());
    }
    Scratch ws(A.t(10), gnn_propagate_fused_workspace(g->E, (int)F, op), dO.device());
    const float* wp = f32(w, "w_csrT");
    const int32_t* ap = i32(arg, "argmax");
    const gnn_dtype dt = dtype_of(dO);
    const gnn_stream st = stream();
    CALL(gnn_propagate_fused_backward(g, w.defined() ? GNN_MSG_E_MUL_XJ : GNN_MSG_COPY_XJ, op, ptr(dO), ptr(X), wp, ap, (int)F, dt, ptr(dX),
                                      (float*)ptr(dW), ws.p, ws.n, st));
    return wrap_all(dX, first(dW, g->E));
}

// gnn_row_epilogue from (Xself, self_coef, self_mode, bias, relu), or none for None
struct Epilogue {
    gnn_row_epilogue e{};
    const gnn_row_epilogue* p = nullptr;
    THPObjectPtr held[5];  // the values stay alive for the call, whatever becomes of the mapping meanwhile
    Epilogue(const Args& A, int k) {
        PyObject* o = A.at(k);
        if (o == Py_None) return;
        static const char* const names[5] = {"Xself", "self_coef", "self_mode", "bias", "relu"};
        for (int q = 0; q < 5; ++q) held[q] = value(o, names[q]);
        e.Xself = ptr(tensor(0, "Xself"));
        e.self_coef = held[1].get() ? (float)as_float(held[1].get()) : 0.f;
        e.self_mode = held[2].get() ? (int)as_int(held[2].get()) : GNN_SELF_ALWAYS;
        e.bias = f32(tensor(3, "bias"), "bias");
        e.relu = held[4].get() && as_bool(held[4].get());
        p = &e;
    }
    // a new reference, or null if the mapping (a dict, or anything with a get) has no such key
    static PyObject* value(PyObject* o, const char* name) {
        if (PyDict_Check(o)) {
            PyObject* v = PyDict_GetItemString(o, name);
            Py_XINCREF(v);
            return v;
        }
        static PyObject* const absent = PyList_New(0);
        PyObject* v = PyObject_CallMethod(o, "get", "sO", name, absent);
        if (!v) rethrow();
        if (v != absent) return v;
        Py_DECREF(v);
        return nullptr;
    }
    at::Tensor tensor(int q, const char* name) {
        PyObject* v = held[q].get();
        if (!v || v == Py_None) return at::Tensor();
        if (!THPVariable_Check(v)) raise(PyExc_TypeError, std::string(name) + " must be a tensor");
        return THPVariable_Unpack(v);
    }
};

static int factor_width(const at::Tensor& e) { return !e.defined() ? 0 : e.dim() == 1 ? 1 : (int)e.size(1); }

// (g, msg, Xj, Xi, e_csr, op, epi, out, argmax, ws) -> out or (out, argmax)
FN(propagate_msg) {
    const gnn_csr* g = A.g(0);
    const gnn_msg msg = (gnn_msg)A.i(1);
    const at::Tensor &Xj = A.dev(2), &Xi = A.t(3), &ef = A.t(4);
    const gnn_op op = A.op(5);
    const Epilogue epi(A, 6);
    at::Tensor out = A.t(7), arg = A.t(8);
    const int64_t F = Xj.size(1);
    if (!out.defined()) out = empty({g->N, F}, Xj.scalar_type(), Xj.device());
    if (has_winners(op) && !arg.defined()) arg = empty({g->N, F}, at::kInt, Xj.device());
    Scratch ws(A.t(9), gnn_propagate_fused_workspace(g->E, (int)F, op), Xj.device());
    const float* ep = f32(ef, "e_csr");
    int32_t* ap = i32(arg, "argmax");
    const gnn_dtype dt = dtype_of(Xj);
    const gnn_stream st = stream();
    CALL(gnn_propagate_msg(g, msg, op, ptr(Xj), ptr(Xi), ep, factor_width(ef), (int)F, dt, epi.p, ptr(out), ap, ws.p, ws.n, st));
    return has_winners(op) ? wrap_all(out, arg) : wrap(out);
}

// (g, msg, dOut, op, Xj, e_csrT, e_width, argmax, self_grad, want_dXj, want_dXi, want_de, ws) -> (dXj, dXi, de)
FN(propagate_msg_backward) {
    const gnn_csr* g = A.g(0);
    const gnn_msg msg = (gnn_msg)A.i(1);
    const at::Tensor& dO = A.dev(2);
    const gnn_op op = A.op(3);
    const at::Tensor &Xj = A.t(4), &ef = A.t(5), &arg = A.t(7);
    const int ew = A.flag(6) ? (int)A.i(6) : factor_width(ef);
    const Epilogue sg(A, 8);
    const int64_t F = dO.size(1);
    const auto dev = dO.device();
    at::Tensor dXj, dXi, de;
    if (A.flag(9)) dXj = empty({g->N, F}, dO.scalar_type(), dev);
    if (A.flag(10)) dXi = empty({g->N, F}, dO.scalar_type(), dev);
    if (A.flag(11)) de = empty({at_least_one(g->E), at_least_one(ew)}, at::kFloat, dev);
    Scratch ws(A.t(12), gnn_propagate_fused_workspace(g->E, (int)F, op), dev);
    const float* ep = f32(ef, "e_csrT");
    const int32_t* ap = i32(arg, "argmax");
    const gnn_dtype dt = dtype_of(dO);
    const gnn_stream st = stream();
    CALL(gnn_propagate_msg_backward(g, msg, op, ptr(dO), ptr(Xj), ep, ew, ap, (int)F, dt, sg.p, ptr(dXj), ptr(dXi), (float*)ptr(de), ws.p, ws.n, st));
    return wrap_all(dXj, dXi, first(de, g->E));
}

// (Y, dY, relu, want_dbias, dZ, ws) -> (dZ, dbias)
FN(row_epilogue_backward) {
    const at::Tensor &Y = A.t(0), &dY = A.dev(1);
    const int relu = A.flag(2);
    at::Tensor dZ = A.t(4), db;
    const int64_t N = dY.size(0), F = dY.size(1);
    if (!dZ.defined()) dZ = empty_like(dY);
    if (A.flag(3)) db = empty({F}, at::kFloat, dY.device());
    Scratch ws(A.t(5), gnn_row_epilogue_backward_workspace((int32_t)N, (int)F), dY.device());
    const gnn_dtype dt = dtype_of(dY);
    const gnn_stream st = stream();
    CALL(gnn_row_epilogue_backward(ptr(Y), ptr(dY), (int32_t)N, (int)F, dt, relu, ptr(dZ), (float*)ptr(db), ws.p, ws.n, st));
    return wrap_all(dZ, db);
}

// (g, X, eps, out, ws)
FN(gin) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& X = A.dev(1);
    const float eps = A.f(2);
    at::Tensor out = A.t(3);
    const int64_t F = X.size(1);
    if (!out.defined()) out = empty({g->N, F}, X.scalar_type(), X.device());
    Scratch ws(A.t(4), gnn_gin_workspace(g->E, (int)F), X.device());
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    CALL(gnn_gin(g, ptr(X), eps, (int)F, dt, ptr(out), ws.p, ws.n, st));
    return wrap(out);
}

// (g, dOut, eps, X, want_deps, ws) -> (dX, deps)
FN(gin_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& dO = A.dev(1);
    const float eps = A.f(2);
    const at::Tensor& X = A.t(3);
    const int64_t F = dO.size(1);
    at::Tensor dX = empty({g->N, F}, dO.scalar_type(), dO.device()), deps;
    if (A.flag(4)) deps = empty({1}, at::kFloat, dO.device());
    Scratch ws(A.t(5), gnn_gin_workspace(g->E, (int)F), dO.device());
    const gnn_dtype dt = dtype_of(dO);
    const gnn_stream st = stream();
    CALL(gnn_gin_backward(g, ptr(dO), ptr(X), eps, (int)F, dt, ptr(dX), (float*)ptr(deps), ws.p, ws.n, st));
    return wrap_all(dX, deps);
}

// (g, Xj, Xi, H) -> s [E,H]
FN(edge_dot) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &Xj = A.dev(1), &Xi = A.dev(2);
    int C;
    const int H = A.heads(3, Xj.size(1), &C);
    at::Tensor s = empty({at_least_one(g->E), H}, at::kFloat, Xj.device());
    const gnn_dtype dt = dtype_of(Xj);
    const gnn_stream st = stream();
    CALL(gnn_edge_dot(g, ptr(Xj), ptr(Xi), H, C, dt, (float*)ptr(s), st));
    return wrap(first(s, g->E));
}

// (g, Xj, Xi, ds_csr, H, want_dXj, want_dXi, ws) -> (dXj, dXi)
FN(edge_dot_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &Xj = A.dev(1), &Xi = A.dev(2);
    int C;
    const int H = A.heads(4, Xj.size(1), &C);
    at::Tensor dXj, dXi;
    if (A.flag(5)) dXj = empty_like(Xj);
    if (A.flag(6)) dXi = empty_like(Xi);
    Scratch ws(A.t(7), gnn_edge_dot_backward_workspace(g->E, H, C), Xj.device());
    const float* ds = f32(A.t(3), "ds_csr");
    const gnn_dtype dt = dtype_of(Xj);
    const gnn_stream st = stream();
    CALL(gnn_edge_dot_backward(g, ptr(Xj), ptr(Xi), ds, H, C, dt, ptr(dXj), ptr(dXi), ws.p, ws.n, st));
    return wrap_all(dXj, dXi);
}

// (g, Xl, Xr, a, H, slope) -> s [E,H]
FN(gatv2_logits) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &Xl = A.dev(1), &Xr = A.dev(2);
    const float* a = f32(A.t(3), "a");
    int C;
    const int H = A.heads(4, Xl.size(1), &C);
    const float slope = A.f(5);
    at::Tensor s = empty({at_least_one(g->E), H}, at::kFloat, Xl.device());
    const gnn_dtype dt = dtype_of(Xl);
    const gnn_stream st = stream();
    CALL(gnn_gatv2_logits(g, ptr(Xl), ptr(Xr), a, H, C, dt, slope, (float*)ptr(s), st));
    return wrap(first(s, g->E));
}

// (g, Xl, Xr, a, ds_csr, H, slope, ws) -> (dXl, dXr, da)
FN(gatv2_logits_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &Xl = A.dev(1), &Xr = A.dev(2);
    const float *a = f32(A.t(3), "a"), *ds = f32(A.t(4), "ds_csr");
    int C;
    const int H = A.heads(5, Xl.size(1), &C), N = (int)Xl.size(0);
    const float slope = A.f(6);
    at::Tensor dXl = empty_like(Xl), dXr = empty_like(Xr), da = empty({H, C}, at::kFloat, Xl.device());
    Scratch ws(A.t(7), gnn_gatv2_logits_backward_workspace(N, H, C), Xl.device());
    const gnn_dtype dt = dtype_of(Xl);
    const gnn_stream st = stream();
    CALL(gnn_gatv2_logits_backward(g, ptr(Xl), ptr(Xr), a, ds, H, C, dt, slope, ptr(dXl), ptr(dXr), (float*)ptr(da), ws.p, ws.n, st));
    return wrap_all(dXl, dXr, da);
}

// ---------------------------------------------------------------- unfused primitives
// (idx, X, out)
FN(gather) {
    const at::Tensor &idx = A.must(0), &X = A.dev(1);
    at::Tensor out = A.t(2);
    const int64_t E = idx.numel(), F = X.size(1);
    if (!out.defined()) out = empty({E, F}, X.scalar_type(), X.device());
    const int32_t* ip = i32(idx, "idx");
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    CALL(gnn_gather(ip, E, ptr(X), (int32_t)X.size(0), (int)F, dt, ptr(out), st));
    return wrap(out);
}

// (g, dOut_EF, by_src, ws) -> dX
FN(gather_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& dO = A.dev(1);
    const int by_src = (int)as_int(A.at(2));
    const int64_t F = dO.size(1);
    at::Tensor dX = empty({g->N, F}, dO.scalar_type(), dO.device());
    Scratch ws(A.t(3), gnn_propagate_fused_workspace(g->E, (int)F, GNN_SUM), dO.device());
    const gnn_dtype dt = dtype_of(dO);
    const gnn_stream st = stream();
    CALL(gnn_gather_backward(g, by_src, ptr(dO), (int)F, dt, ptr(dX), ws.p, ws.n, st));
    return wrap(dX);
}

// (g, msg, X, ar, e, slope) -> m [E,F]
FN(apply_edges) {
    const gnn_csr* g = A.g(0);
    const gnn_msg msg = (gnn_msg)A.i(1);
    const at::Tensor &X = A.dev(2), &ar = A.t(3), &ef = A.t(4);
    const float slope = A.f(5);
    const int64_t F = X.size(1);
    at::Tensor m = empty({at_least_one(g->E), F}, X.scalar_type(), X.device());
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    CALL(gnn_apply_edges(g, msg, ptr(X), ptr(ar), (const float*)ptr(ef), factor_width(ef), (int)F, dt, slope, ptr(m), st));
    return wrap(first(m, g->E));
}

// (g, m_EF, op, ws) -> out or (out, argmax)
FN(aggregate) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& m = A.dev(1);
    const gnn_op op = A.op(2);
    const int64_t F = m.size(1);
    at::Tensor out = empty({g->N, F}, m.scalar_type(), m.device()), arg;
    if (has_winners(op)) arg = empty({g->N, F}, at::kInt, m.device());
    Scratch ws(A.t(3), gnn_propagate_fused_workspace(g->E, (int)F, op), m.device());
    const gnn_dtype dt = dtype_of(m);
    const gnn_stream st = stream();
    CALL(gnn_aggregate(g, op, ptr(m), (int)F, dt, ptr(out), (int32_t*)ptr(arg), ws.p, ws.n, st));
    return has_winners(op) ? wrap_all(out, arg) : wrap(out);
}

// (g, dOut, op, argmax) -> dm [E,F]
FN(aggregate_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& dO = A.dev(1);
    const gnn_op op = A.op(2);
    const int32_t* ap = i32(A.t(3), "argmax");
    const int64_t F = dO.size(1);
    at::Tensor dm = empty({at_least_one(g->E), F}, dO.scalar_type(), dO.device());
    const gnn_dtype dt = dtype_of(dO);
    const gnn_stream st = stream();
    CALL(gnn_aggregate_backward(g, op, ptr(dO), ap, (int)F, dt, ptr(dm), st));
    return wrap(first(dm, g->E));
}

// (g, logits, want_stats) -> alpha or (alpha, rowmax, rowsum)
FN(edge_softmax) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& s = A.dev(1);
    const bool stats = A.flag(2);
    const int64_t H = s.size(1);
    at::Tensor alpha = empty_like(s), mx, sm;
    if (stats) {
        mx = empty({g->N, H}, at::kFloat, s.device());
        sm = empty({g->N, H}, at::kFloat, s.device());
    }
    const gnn_dtype dt = dtype_of(s);
    const gnn_stream st = stream();
    CALL(gnn_edge_softmax(g, ptr(s), (int)H, dt, ptr(alpha), (float*)ptr(mx), (float*)ptr(sm), st));
    return stats ? wrap_all(alpha, mx, sm) : wrap(alpha);
}

// (g, alpha, dalpha) -> ds
FN(edge_softmax_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &alpha = A.dev(1), &da = A.dev(2);
    at::Tensor ds = empty_like(alpha);
    const gnn_dtype dt = dtype_of(alpha);
    const gnn_stream st = stream();
    CALL(gnn_edge_softmax_backward(g, ptr(alpha), ptr(da), (int)alpha.size(1), dt, ptr(ds), st));
    return wrap(ds);
}

// (a, b, alpha, beta, out)
FN(axpby) {
    const at::Tensor &a = A.dev(0), &b = A.dev(1);
    const float al = A.f(2), be = A.f(3);
    at::Tensor out = A.t(4);
    if (!out.defined()) out = empty_like(a);
    const gnn_dtype dt = dtype_of(a);
    const gnn_stream st = stream();
    CALL(gnn_axpby(al, ptr(a), be, ptr(b), a.numel(), dt, ptr(out), st));
    return wrap(out);
}

// ---------------------------------------------------------------- pooling
// (graph_ptr, X, op, ws) -> out or (out, argmax)
FN(reduce_nodes) {
    const at::Tensor &gp = A.must(0), &X = A.dev(1);
    const gnn_op op = A.op(2);
    const int64_t G = gp.numel() - 1, N = X.size(0), F = X.size(1);
    at::Tensor out = empty({G, F}, X.scalar_type(), X.device()), arg;
    if (has_winners(op)) arg = empty({G, F}, at::kInt, X.device());
    Scratch ws(A.t(3), gnn_propagate_fused_workspace(N, (int)F, op), X.device());
    const int64_t* p = i64(gp, "graph_ptr");
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    CALL(gnn_reduce_nodes(p, (int32_t)G, (int32_t)N, op, ptr(X), (int)F, dt, ptr(out), (int32_t*)ptr(arg), ws.p, ws.n, st));
    return has_winners(op) ? wrap_all(out, arg) : wrap(out);
}

// (graph_ptr, dOut, N, op, argmax) -> dX
FN(reduce_nodes_backward) {
    const at::Tensor &gp = A.t(0), &dO = A.dev(1);
    const int64_t N = A.i(2), G = dO.size(0), F = dO.size(1);
    const gnn_op op = A.op(3);
    at::Tensor dX = empty({N, F}, dO.scalar_type(), dO.device());
    const int64_t* p = i64(gp, "graph_ptr");
    const int32_t* ap = i32(A.t(4), "argmax");
    const gnn_dtype dt = dtype_of(dO);
    const gnn_stream st = stream();
    CALL(gnn_reduce_nodes_backward(p, (int32_t)G, (int32_t)N, op, ptr(dO), ap, (int)F, dt, ptr(dX), st));
    return wrap(dX);
}

// ---------------------------------------------------------------- attention
// (g, Wx, a_src, a_dst, H, slope, ws) -> (out, alpha, al, ar)
FN(gat_fused) {
    const gnn_csr* g = A.g(0);
    const at::Tensor& Wx = A.dev(1);
    const int64_t N = Wx.size(0);
    int C;
    const int H = A.heads(4, Wx.size(1), &C);
    const float slope = A.f(5);
    const auto dev = Wx.device();
    at::Tensor out = empty_like(Wx), alpha = empty({at_least_one(g->E), H}, at::kFloat, dev), al = empty({N, H}, at::kFloat, dev),
               ar = empty({N, H}, at::kFloat, dev);
    Scratch ws(A.t(6), gnn_gat_fused_workspace((int32_t)N, g->E, H, C, 0), dev);
    const float *as = (const float*)ptr(A.t(2)), *ad = (const float*)ptr(A.t(3));
    const gnn_dtype dt = dtype_of(Wx);
    const gnn_stream st = stream();
    CALL(gnn_gat_fused(g, ptr(Wx), as, ad, H, C, dt, slope, ptr(out), (float*)ptr(alpha), (float*)ptr(al), (float*)ptr(ar), ws.p, ws.n, st));
    return wrap_all(out, first(alpha, g->E), al, ar);
}

// (g, Wx, a_src, a_dst, alpha, al, ar, dOut, H, slope, ws) -> (dWx, da_src, da_dst)
FN(gat_fused_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &Wx = A.dev(1), &dO = A.dev(7);
    const int64_t N = Wx.size(0);
    int C;
    const int H = A.heads(8, Wx.size(1), &C);
    const float slope = A.f(9);
    const auto dev = Wx.device();
    at::Tensor dWx = empty_like(Wx), das = empty({H, C}, at::kFloat, dev), dad = empty({H, C}, at::kFloat, dev);
    Scratch ws(A.t(10), gnn_gat_fused_workspace((int32_t)N, g->E, H, C, 1), dev);
    const float *as = (const float*)ptr(A.t(2)), *ad = (const float*)ptr(A.t(3)), *alpha = (const float*)ptr(A.t(4)), *al = (const float*)ptr(A.t(5)),
                *ar = (const float*)ptr(A.t(6));
    const gnn_dtype dt = dtype_of(Wx);
    const gnn_stream st = stream();
    CALL(gnn_gat_fused_backward(g, ptr(Wx), as, ad, alpha, al, ar, ptr(dO), H, C, dt, slope, ptr(dWx), (float*)ptr(das), (float*)ptr(dad), ws.p, ws.n, st));
    return wrap_all(dWx, das, dad);
}

// ---------------------------------------------------------------- dense transform
// the workspace of a dense call may be asked for (its first word is the status of the tensor-core kernels): a tensor then
static at::Tensor linear_scratch(const Args& A, int k, bool wanted, size_t need, c10::Device dev) {
    const at::Tensor& given = A.t(k);
    return given.defined() || !wanted ? given : empty({(int64_t)need}, at::kByte, dev);
}

// (X, W, bias, relu, ws, return_ws) -> Y or (Y, ws)
FN(linear) {
    const at::Tensor &X = A.dev(0), &W = A.dev(1);
    const int64_t N = X.size(0), K = X.size(1), M = W.size(1);
    const int relu = A.flag(3);
    const bool wanted = A.flag(5);
    at::Tensor Y = empty({N, M}, X.scalar_type(), X.device());
    const size_t need = gnn_linear_workspace((int32_t)N, (int)K, (int)M);
    const at::Tensor wt = linear_scratch(A, 4, wanted, need, X.device());
    Scratch ws(wt, K % 8 == 0 && M % 8 == 0 ? 256 : need, X.device());  // the status word only, unless rows may have to be padded
    const float* b = f32(A.t(2), "bias");
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    CALL(gnn_linear_bias_act(ptr(X), ptr(W), (int32_t)N, (int)K, (int)M, dt, b, relu, ptr(Y), ws.p, ws.n, st));
    return wanted ? wrap_all(Y, wt) : wrap(Y);
}

// (X, W, dY, want_dX, want_dW, ws, return_ws) -> (dX, dW) or (dX, dW, ws)
FN(linear_backward) {
    const at::Tensor &X = A.t(0), &W = A.t(1), &dY = A.dev(2);
    const int64_t N = dY.size(0), M = dY.size(1), K = W.defined() ? W.size(0) : A.must(0).size(1);
    const bool wanted = A.flag(6);
    at::Tensor dX, dW;
    if (A.flag(3)) dX = empty({N, K}, dY.scalar_type(), dY.device());
    if (A.flag(4)) dW = empty({K, M}, dY.scalar_type(), dY.device());
    const size_t need = gnn_linear_workspace((int32_t)N, (int)K, (int)M);
    const at::Tensor wt = linear_scratch(A, 5, wanted, need, dY.device());
    Scratch ws(wt, need, dY.device());
    const gnn_dtype dt = dtype_of(dY);
    const gnn_stream st = stream();
    CALL(gnn_linear_backward(ptr(X), ptr(W), ptr(dY), (int32_t)N, (int)K, (int)M, dt, ptr(dX), ptr(dW), ws.p, ws.n, st));
    return wanted ? wrap_all(dX, dW, wt) : wrap_all(dX, dW);
}

// (g, X, W, w_csr, op, bias, relu, ws, return_ws) -> Y or (Y, ws)
FN(propagate_linear) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &X = A.dev(1), &W = A.dev(2), &w = A.t(3);
    const gnn_op op = A.op(4);
    const int relu = A.flag(6);
    const bool wanted = A.flag(8);
    const int64_t K = W.size(0), M = W.size(1);
    at::Tensor Y = empty({g->N, M}, X.scalar_type(), X.device());
    const size_t need = gnn_propagate_linear_workspace(g->N, g->E, (int)K, (int)M);
    const at::Tensor wt = linear_scratch(A, 7, wanted, need, X.device());
    Scratch ws(wt, need, X.device());
    const float *wp = f32(w, "w_csr"), *b = f32(A.t(5), "bias");
    const gnn_dtype dt = dtype_of(X);
    const gnn_stream st = stream();
    CALL(gnn_propagate_linear(g, w.defined() ? GNN_MSG_E_MUL_XJ : GNN_MSG_COPY_XJ, op, ptr(X), wp, ptr(W), (int)K, (int)M, dt, b, relu, ptr(Y), ws.p, ws.n, st));
    return wanted ? wrap_all(Y, wt) : wrap(Y);
}

// (g, dY, X, W, w_csrT, op, want_dX, want_dW, ws) -> (dX, dW)
FN(propagate_linear_backward) {
    const gnn_csr* g = A.g(0);
    const at::Tensor &dY = A.dev(1), &X = A.t(2), &W = A.dev(3), &w = A.t(4);
    const gnn_op op = A.op(5);
    const int64_t K = W.size(0), M = W.size(1);
    at::Tensor dX, dW;
    if (A.flag(6)) dX = empty({g->N, K}, dY.scalar_type(), dY.device());
    if (A.flag(7)) dW = empty({K, M}, dY.scalar_type(), dY.device());
    Scratch ws(A.t(8), gnn_propagate_linear_workspace(g->N, g->E, (int)K, (int)M), dY.device());
    const float* wp = f32(w, "w_csrT");
    const gnn_dtype dt = dtype_of(dY);
    const gnn_stream st = stream();
    CALL(gnn_propagate_linear_backward(g, w.defined() ? GNN_MSG_E_MUL_XJ : GNN_MSG_COPY_XJ, op, ptr(dY), ptr(X), wp, ptr(W), (int)K, (int)M, dt, ptr(dX), ptr(dW),
                                       ws.p, ws.n, st));
    return wrap_all(dX, dW);
}

// (module dict, real torch, error class): what the calls take from the Python module
FN(attach) {
    g_module_dict = A.at(0);
    g_real_torch = A.at(1);
    g_error = A.at(2);
    for (PyObject* o : {g_module_dict, g_real_torch, g_error}) Py_INCREF(o);
    g_s_torch = PyUnicode_InternFromString("torch");
    g_s_empty = PyUnicode_InternFromString("empty");
    Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    ENTRY(attach), ENTRY(coo_to_csr), ENTRY(degree), ENTRY(add_self_loops), ENTRY(gcn_norm), ENTRY(permute_edge_data), ENTRY(segment_coef),
    ENTRY(merge_edge_lists), ENTRY(graph_ptr_from_ids), ENTRY(propagate_fused), ENTRY(propagate_fused_backward), ENTRY(propagate_msg),
    ENTRY(propagate_msg_backward), ENTRY(row_epilogue_backward), ENTRY(gin), ENTRY(gin_backward), ENTRY(edge_dot), ENTRY(edge_dot_backward),
    ENTRY(gatv2_logits), ENTRY(gatv2_logits_backward), ENTRY(gather), ENTRY(gather_backward), ENTRY(apply_edges), ENTRY(aggregate),
    ENTRY(aggregate_backward), ENTRY(edge_softmax), ENTRY(edge_softmax_backward), ENTRY(axpby), ENTRY(reduce_nodes), ENTRY(reduce_nodes_backward),
    ENTRY(gat_fused), ENTRY(gat_fused_backward), ENTRY(linear), ENTRY(linear_backward), ENTRY(propagate_linear), ENTRY(propagate_linear_backward),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", "calls of the C ABI on torch tensors", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) { return PyModule_Create(&module); }
