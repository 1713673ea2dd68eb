"""Binding of libgnn_b200.so: argument marshalling only.

The calls go through the compiled extension ``_binding`` (csrc/binding.cpp), which unpacks tensors and allocates
outputs and workspaces; the ctypes prototypes of the C ABI stay available through ``load()``.

Every function here has the name of the C entry point without the ``gnn_`` prefix, takes torch
CUDA tensors (torch is used for device memory and streams, nothing else), allocates outputs and
workspaces when they are not passed in, and raises ``GnnError`` on a non-zero status.  There is no
CPU path: loading fails if the CUDA library has not been built.
"""
from __future__ import annotations

import ctypes as C
import os
from ctypes import addressof as _addr

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libgnn_b200.so")
_lib = None


class _Unloaded:
    """Stands for the extension until the first call loads the library."""

    def __getattr__(self, name):
        load()
        return getattr(_b, name)


_b = _Unloaded()

SUM, MEAN, MAX, MIN = 0, 1, 2, 3
COPY_XJ, E_MUL_XJ, GAT_LOGIT, XI_SUB_XJ, XI_DOT_XJ = 0, 1, 2, 3, 4
SELF_ALWAYS, SELF_TIMES_DEGREE, SELF_IF_NONEMPTY = 0, 1, 2
F32, BF16 = 0, 1
OPS = {"sum": SUM, "mean": MEAN, "max": MAX, "min": MIN}
STATUS_NAMES = ["OK", "INVALID_ARG", "INDEX_OUT_OF_RANGE", "NOT_SORTED", "WORKSPACE_TOO_SMALL", "UNSUPPORTED", "CUDA", "TIMEOUT"]


class GnnError(RuntimeError):
    def __init__(self, status, msg):
        super().__init__(f"gnn status {status} ({STATUS_NAMES[status] if 0 <= status < len(STATUS_NAMES) else '?'}): {msg}")
        self.status = status


class CsrStruct(C.Structure):
    _fields_ = [("N", C.c_int32), ("E", C.c_int64), ("rowptr", C.c_void_p), ("col", C.c_void_p), ("eid", C.c_void_p),
                ("rowptrT", C.c_void_p), ("colT", C.c_void_p), ("eidT", C.c_void_p), ("t2f", C.c_void_p)]


class RowEpilogueStruct(C.Structure):
    _fields_ = [("Xself", C.c_void_p), ("self_coef", C.c_float), ("self_mode", C.c_int), ("bias", C.c_void_p), ("relu", C.c_int)]


class EdgeSegmentStruct(C.Structure):
    _fields_ = [("E", C.c_int64), ("src", C.c_void_p), ("dst", C.c_void_p), ("src_offset", C.c_int32), ("dst_offset", C.c_int32)]


_VP, _I32, _I64, _INT, _SZ, _F = C.c_void_p, C.c_int32, C.c_int64, C.c_int, C.c_size_t, C.c_float
_CSR = C.POINTER(CsrStruct)
_EPI = C.POINTER(RowEpilogueStruct)
_SEG = C.POINTER(EdgeSegmentStruct)

# name -> (restype, argtypes); mirrors include/gnn.h
SIGNATURES = {
    "gnn_status_string": (C.c_char_p, [_INT]),
    "gnn_last_error_string": (C.c_char_p, []),
    "gnn_version": (_INT, []),
    "gnn_coo_to_csr_workspace": (_SZ, [_I32, _I64]),
    "gnn_coo_to_csr": (_INT, [_I32, _I64, _VP, _VP, _CSR, _VP, _SZ, _VP]),
    "gnn_probe_gather_sink_floats": (_SZ, [_I64]),
    "gnn_probe_gather": (_INT, [_VP, _I64, _VP, _I32, _INT, _VP, _VP]),
    "gnn_csr_validate_workspace": (_SZ, [_I64]),
    "gnn_csr_validate": (_INT, [_CSR, _VP, _SZ, _VP]),
    "gnn_degree": (_INT, [_CSR, _INT, _VP, _VP, _VP]),
    "gnn_add_self_loops": (_INT, [_I32, _I64, _VP, _VP, _VP, _VP, _VP]),
    "gnn_gcn_norm": (_INT, [_CSR, _VP, _VP, _VP, _VP, _VP]),
    "gnn_permute_edge_data": (_INT, [_VP, _I64, _INT, _INT, _VP, _VP, _VP]),
    "gnn_propagate_fused_workspace": (_SZ, [_I64, _INT, _INT]),
    "gnn_propagate_fused": (_INT, [_CSR, _INT, _INT, _VP, _VP, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_fused_backward": (_INT, [_CSR, _INT, _INT, _VP, _VP, _VP, _VP, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_fused_static_max_bytes": (_SZ, []),
    "gnn_propagate_fused_static": (_INT, [_CSR, _INT, _INT, _VP, _VP, _INT, _INT, _VP, _VP, _VP]),
    "gnn_propagate_msg": (_INT, [_CSR, _INT, _INT, _VP, _VP, _VP, _INT, _INT, _INT, _EPI, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_msg_backward": (_INT, [_CSR, _INT, _INT, _VP, _VP, _VP, _INT, _VP, _INT, _INT, _EPI, _VP, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_row_epilogue_backward_workspace": (_SZ, [_I32, _INT]),
    "gnn_row_epilogue_backward": (_INT, [_VP, _VP, _I32, _INT, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_gin_workspace": (_SZ, [_I64, _INT]),
    "gnn_gin": (_INT, [_CSR, _VP, _F, _INT, _INT, _VP, _VP, _SZ, _VP]),
    "gnn_gin_backward": (_INT, [_CSR, _VP, _VP, _F, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_edge_dot": (_INT, [_CSR, _VP, _VP, _INT, _INT, _INT, _VP, _VP]),
    "gnn_edge_dot_backward_workspace": (_SZ, [_I64, _INT, _INT]),
    "gnn_edge_dot_backward": (_INT, [_CSR, _VP, _VP, _VP, _INT, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_gatv2_logits": (_INT, [_CSR, _VP, _VP, _VP, _INT, _INT, _INT, _F, _VP, _VP]),
    "gnn_gatv2_logits_backward_workspace": (_SZ, [_I32, _INT, _INT]),
    "gnn_gatv2_logits_backward": (_INT, [_CSR, _VP, _VP, _VP, _VP, _INT, _INT, _INT, _F, _VP, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_merge_edge_lists": (_INT, [_SEG, _INT, _VP, _VP, _VP, _VP]),
    "gnn_segment_coef": (_INT, [_CSR, _VP, _VP, _VP, _INT, _VP, _VP, _VP]),
    "gnn_gather": (_INT, [_VP, _I64, _VP, _I32, _INT, _INT, _VP, _VP]),
    "gnn_gather_backward": (_INT, [_CSR, _INT, _VP, _INT, _INT, _VP, _VP, _SZ, _VP]),
    "gnn_apply_edges": (_INT, [_CSR, _INT, _VP, _VP, _VP, _INT, _INT, _INT, _F, _VP, _VP]),
    "gnn_aggregate": (_INT, [_CSR, _INT, _VP, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_aggregate_backward": (_INT, [_CSR, _INT, _VP, _VP, _INT, _INT, _VP, _VP]),
    "gnn_axpby": (_INT, [_F, _VP, _F, _VP, _I64, _INT, _VP, _VP]),
    "gnn_edge_softmax": (_INT, [_CSR, _VP, _INT, _INT, _VP, _VP, _VP, _VP]),
    "gnn_edge_softmax_backward": (_INT, [_CSR, _VP, _VP, _INT, _INT, _VP, _VP]),
    "gnn_gat_fused_workspace": (_SZ, [_I32, _I64, _INT, _INT, _INT]),
    "gnn_gat_fused": (_INT, [_CSR, _VP, _VP, _VP, _INT, _INT, _INT, _F, _VP, _VP, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_gat_fused_backward": (_INT, [_CSR, _VP, _VP, _VP, _VP, _VP, _VP, _VP, _INT, _INT, _INT, _F, _VP, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_graph_ptr_from_ids": (_INT, [_VP, _I32, _I32, _VP, _VP, _SZ, _VP]),
    "gnn_reduce_nodes": (_INT, [_VP, _I32, _I32, _INT, _VP, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_reduce_nodes_backward": (_INT, [_VP, _I32, _I32, _INT, _VP, _VP, _INT, _INT, _VP, _VP]),
    "gnn_linear_workspace": (_SZ, [_I32, _INT, _INT]),
    "gnn_linear": (_INT, [_VP, _VP, _I32, _INT, _INT, _INT, _VP, _VP, _SZ, _VP]),
    "gnn_linear_bias_act": (_INT, [_VP, _VP, _I32, _INT, _INT, _INT, _VP, _INT, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_linear_workspace": (_SZ, [_I32, _I64, _INT, _INT]),
    "gnn_propagate_linear": (_INT, [_CSR, _INT, _INT, _VP, _VP, _VP, _INT, _INT, _INT, _VP, _INT, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_linear_backward": (_INT, [_CSR, _INT, _INT, _VP, _VP, _VP, _VP, _INT, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_linear_backward": (_INT, [_VP, _VP, _VP, _I32, _INT, _INT, _INT, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_fused_host": (_INT, [_CSR, _INT, _INT, _VP, _VP, _INT, _INT, _VP, _VP, _VP, _VP, _VP, _SZ, _VP]),
    "gnn_propagate_fused_backward_host": (_INT, [_CSR, _INT, _INT, _VP, _VP, _VP, _INT, _INT, _VP, _VP, _VP, _VP, _SZ, _VP]),
}


def load(path: str = LIB_PATH):
    """Load the CUDA library (no GPU needed to load it) and set the prototypes."""
    global _lib
    if _lib is None:
        if not os.path.exists(path):
            raise ImportError(f"{path} is missing: build it with `python -m paper_2412_06354_b200.build` "
                              "(there is no CPU fallback)")
        lib = C.CDLL(path)
        for name, (res, args) in SIGNATURES.items():
            fn = getattr(lib, name)
            fn.restype = res
            fn.argtypes = args
        from . import _binding
        _binding.attach(globals(), torch, GnnError)
        globals()["_b"] = _binding
        _lib = lib
    return _lib


def _check(rc):
    if rc != 0:
        raise GnnError(rc, load().gnn_last_error_string().decode())


def _stream():
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


def _p(t):
    return None if t is None else C.c_void_p(t.data_ptr())


def _pi(t, dtype, name):
    """Pointer of an index tensor, after checking its element type (the C ABI cannot)."""
    if t is None:
        return None
    if t.dtype != dtype:
        raise TypeError(f"{name} must be {dtype}, got {t.dtype}")
    if t.numel() and not t.is_contiguous():
        raise TypeError(f"{name} must be contiguous")
    return C.c_void_p(t.data_ptr())


def _pf32(t, name):
    return _pi(t, torch.float32, name)


def _dtype(t):
    if t.dtype == torch.float32:
        return F32
    if t.dtype == torch.bfloat16:
        return BF16
    raise TypeError(f"unsupported feature dtype {t.dtype}")


def _op(op):
    return OPS[op] if isinstance(op, str) else int(op)


def _dev(t):
    assert t.is_cuda and t.is_contiguous(), "CUDA contiguous tensor expected"
    return t


class Graph:
    """Both sparse forms of a graph on the device (see gnn_csr in gnn.h)."""

    def __init__(self, N, E, device):
        i64 = dict(dtype=torch.int64, device=device)
        i32 = dict(dtype=torch.int32, device=device)
        self.N, self.E = int(N), int(E)
        self.rowptr = torch.empty(N + 1, **i64)
        self.rowptrT = torch.empty(N + 1, **i64)
        n = max(self.E, 1)
        self.col, self.eid, self.colT, self.eidT, self.t2f = (torch.empty(n, **i32) for _ in range(5))
        self._describe()

    def _describe(self):
        self.c = CsrStruct(self.N, self.E, *(t.data_ptr() for t in (self.rowptr, self.col, self.eid, self.rowptrT, self.colT, self.eidT, self.t2f)))

    @property
    def ref(self):
        return C.byref(self.c)

    def nbytes(self):
        return sum(t.numel() * t.element_size() for t in (self.rowptr, self.col, self.eid, self.rowptrT, self.colT, self.eidT, self.t2f))


# ------------------------------------------------------------------ graph set-up
def coo_to_csr(N, src, dst, ws=None) -> Graph:
    g = Graph.__new__(Graph)
    g.rowptr, g.rowptrT, g.col, g.eid, g.colT, g.eidT, g.t2f = _b.coo_to_csr(N, src, dst, ws)
    g.N, g.E = int(N), src.numel()
    g._describe()
    return g


def probe_gather(col, X, row_bytes, sink=None):
    """The bare gathers of one pass over col (see gnn_probe_gather): returns the sink buffer."""
    E = col.numel()
    if sink is None:
        sink = torch.empty(load().gnn_probe_gather_sink_floats(E), dtype=torch.float32, device=col.device)
    _check(load().gnn_probe_gather(_pi(col, torch.int32, "col"), E, _p(X), X.shape[0], int(row_bytes), _p(sink), _stream()))
    return sink


def csr_validate(g: Graph, ws=None):
    """Raises GnnError (INVALID_ARG, the failed checks in its text) unless g is a sound sparse form."""
    if ws is None:
        ws = torch.empty(load().gnn_csr_validate_workspace(g.E), dtype=torch.uint8, device=g.rowptr.device)
    _check(load().gnn_csr_validate(g.ref, _p(ws), ws.numel(), _stream()))


def degree(g: Graph, transposed=False, w=None):
    return _b.degree(_addr(g.c), transposed, w, g.rowptr)


def add_self_loops(N, src, dst):
    return _b.add_self_loops(N, src, dst)


def gcn_norm(g: Graph, w_csr=None, want_T=True):
    """-> (degrees, coefficients in CSR order, coefficients in transposed-CSR order or None)"""
    return _b.gcn_norm(_addr(g.c), w_csr, want_T, g.rowptr)


def permute_edge_data(perm, x, out=None):
    return _b.permute_edge_data(perm, x, out)


# ------------------------------------------------------------------ fused propagate
def propagate_fused_workspace(E, F, op="sum"):
    return load().gnn_propagate_fused_workspace(E, F, _op(op))


def propagate_fused(g: Graph, X, w_csr=None, op="sum", out=None, argmax=None, ws=None):
    """-> out, or (out, argmax) for max/min."""
    return _b.propagate_fused(_addr(g.c), X, w_csr, op, out, argmax, ws, False)


def propagate_fused_backward(g: Graph, dOut, op="sum", X=None, w_csrT=None, argmax=None, want_dX=True, want_dW=False,
                             dX=None, dW=None, ws=None):
    """-> (dX or None, dW or None)."""
    return _b.propagate_fused_backward(_addr(g.c), dOut, op, X, w_csrT, argmax, want_dX, want_dW, dX, dW, ws)


def propagate_fused_host(g: Graph, h_X, w_csr, op, h_out, d_in, d_out, ws, argmax=None):
    """Host-buffer forward: h_X, h_out are (pinned) host tensors; d_in, d_out device staging."""
    F = h_X.shape[1]
    msg = COPY_XJ if w_csr is None else E_MUL_XJ
    _check(load().gnn_propagate_fused_host(g.ref, msg, _op(op), _p(h_X), _pf32(w_csr, "w_csr"), F, _dtype(h_X), _p(h_out), _pi(argmax, torch.int32, "argmax"),
                                           _p(d_in), _p(d_out), _p(ws), ws.numel(), _stream()))
    return h_out


def propagate_fused_backward_host(g: Graph, h_dOut, op, w_csrT, h_dX, d_in, d_out, ws, argmax=None):
    F = h_dOut.shape[1]
    msg = COPY_XJ if w_csrT is None else E_MUL_XJ
    _check(load().gnn_propagate_fused_backward_host(g.ref, msg, _op(op), _p(h_dOut), _pf32(w_csrT, "w_csrT"), _pi(argmax, torch.int32, "argmax"), F, _dtype(h_dOut),
                                                    _p(h_dX), _p(d_in), _p(d_out), _p(ws), ws.numel(), _stream()))
    return h_dX


# ------------------------------------------------------------------ more (message, op) pairs, GIN, XI_DOT_XJ
def propagate_msg(g: Graph, msg, Xj, Xi=None, e_csr=None, op="sum", epi=None, out=None, argmax=None, ws=None):
    """gnn_propagate_msg -> out, or (out, argmax) for max/min.  e_csr: float32 [E] or [E,width] in CSR order.
    epi: dict(Xself=, self_coef=, self_mode=, bias=, relu=) or None."""
    return _b.propagate_msg(_addr(g.c), msg, Xj, Xi, e_csr, op, epi, out, argmax, ws)


def propagate_msg_backward(g: Graph, msg, dOut, op="sum", Xj=None, e_csrT=None, e_width=0, argmax=None, self_grad=None,
                           want_dXj=True, want_dXi=False, want_de=False, ws=None):
    """gnn_propagate_msg_backward -> dict(dXj, dXi, de) with None for the outputs not asked for."""
    dXj, dXi, de = _b.propagate_msg_backward(_addr(g.c), msg, dOut, op, Xj, e_csrT, e_width, argmax, self_grad, want_dXj, want_dXi, want_de, ws)
    return dict(dXj=dXj, dXi=dXi, de=de)


def row_epilogue_backward(Y, dY, relu=True, want_dbias=True, dZ=None, ws=None):
    """-> (dZ, dbias or None)"""
    return _b.row_epilogue_backward(Y, dY, relu, want_dbias, dZ, ws)


def gin(g: Graph, X, eps, out=None, ws=None):
    return _b.gin(_addr(g.c), X, eps, out, ws)


def gin_backward(g: Graph, dOut, eps, X=None, want_deps=False, ws=None):
    """-> (dX, deps as a float32 device tensor of one element, or None)"""
    return _b.gin_backward(_addr(g.c), dOut, eps, X, want_deps, ws)


def edge_dot(g: Graph, Xj, Xi, H=1):
    """s[p,h] = <Xi[row(p),h,:], Xj[col[p],h,:]> -> float32 [E,H], CSR order."""
    return _b.edge_dot(_addr(g.c), Xj, Xi, H)


def edge_dot_backward(g: Graph, Xj, Xi, ds_csr, H=1, want_dXj=True, want_dXi=True, ws=None):
    return _b.edge_dot_backward(_addr(g.c), Xj, Xi, ds_csr, H, want_dXj, want_dXi, ws)


def gatv2_logits(g: Graph, Xl, Xr, a, H, slope=0.2):
    """s[p,h] = sum_c a[h,c] * LeakyReLU(Xl[col[p],h,c] + Xr[row(p),h,c]) -> float32 [E,H], CSR order."""
    return _b.gatv2_logits(_addr(g.c), Xl, Xr, a, H, slope)


def gatv2_logits_backward(g: Graph, Xl, Xr, a, ds_csr, H, slope=0.2, ws=None):
    """-> (dXl, dXr, da)"""
    return _b.gatv2_logits_backward(_addr(g.c), Xl, Xr, a, ds_csr, H, slope, ws)


# ------------------------------------------------------------------ heterogeneous / temporal graphs
def merge_edge_lists(segments):
    """segments: list of (src, dst, src_offset, dst_offset) with int32 device tensors -> (src, dst, seg) of the merged list."""
    return _b.merge_edge_lists(segments)


def segment_coef(g: Graph, seg_csr, seg_is_mean, w_csr=None, want_T=True):
    """-> (coef_csr, coef_csrT or None): per-position multipliers of a merged multi-relation / multi-snapshot form."""
    return _b.segment_coef(_addr(g.c), seg_csr, seg_is_mean, w_csr, want_T, g.rowptr)


# ------------------------------------------------------------------ unfused primitives
def gather(idx, X, out=None):
    return _b.gather(idx, X, out)


def gather_backward(g: Graph, dOut_EF, by_src=False, ws=None):
    return _b.gather_backward(_addr(g.c), dOut_EF, by_src, ws)


def apply_edges(g: Graph, msg, X, ar=None, e=None, slope=0.2):
    """COPY_XJ / E_MUL_XJ: X [N,F], e float32 [E] or [E,w] (CSR order) -> m [E,F] of X.dtype.
    GAT_LOGIT: X = al, ar float32 [N,H] -> float32 [E,H]."""
    return _b.apply_edges(_addr(g.c), msg, X, ar, e, slope)


def aggregate(g: Graph, m_EF, op="sum", ws=None):
    return _b.aggregate(_addr(g.c), m_EF, op, ws)


def aggregate_backward(g: Graph, dOut, op="sum", argmax=None):
    return _b.aggregate_backward(_addr(g.c), dOut, op, argmax)


def edge_softmax(g: Graph, logits, want_stats=False):
    return _b.edge_softmax(_addr(g.c), logits, want_stats)


def edge_softmax_backward(g: Graph, alpha, dalpha):
    return _b.edge_softmax_backward(_addr(g.c), alpha, dalpha)


# ------------------------------------------------------------------ pooling
def graph_ptr_from_ids(graph_id, G):
    return _b.graph_ptr_from_ids(graph_id, G)


def reduce_nodes(graph_ptr, X, op="mean", ws=None):
    return _b.reduce_nodes(graph_ptr, X, op, ws)


def reduce_nodes_backward(graph_ptr, dOut, N, op="mean", argmax=None):
    return _b.reduce_nodes_backward(graph_ptr, dOut, N, op, argmax)


# ------------------------------------------------------------------ GAT
def gat_fused(g: Graph, Wx, a_src, a_dst, H, slope=0.2, ws=None):
    """Wx [N, H*C] -> dict(out, alpha (float32 [E,H], CSR order), al, ar (float32 [N,H]))."""
    out, alpha, al, ar = _b.gat_fused(_addr(g.c), Wx, a_src, a_dst, H, slope, ws)
    return dict(out=out, alpha=alpha, al=al, ar=ar)


def gat_fused_backward(g: Graph, Wx, a_src, a_dst, fwd, dOut, H, slope=0.2, ws=None):
    dWx, da_src, da_dst = _b.gat_fused_backward(_addr(g.c), Wx, a_src, a_dst, fwd["alpha"], fwd["al"], fwd["ar"], dOut, H, slope, ws)
    return dict(dWx=dWx, da_src=da_src, da_dst=da_dst)


def propagate_fused_static(g: Graph, X, w_csr=None, op="sum", out=None, argmax=None):
    """gnn_propagate_fused_static: the fused propagate with the library's built-in 8 MiB scratch, for
    embedders that may not allocate device memory.  The caller passes `out` (and `argmax` for max/min);
    nothing is allocated here when they are given."""
    return _b.propagate_fused(_addr(g.c), X, w_csr, op, out, argmax, None, True)


# ------------------------------------------------------------------ dense transform
def linear(X, W, ws=None, return_ws=False):
    return _b.linear(X, W, None, False, ws, return_ws)


def linear_bias_act(X, W, bias=None, relu=False, ws=None):
    """Y = act(X W + bias) with the tail inside the product kernel's epilogue."""
    return _b.linear(X, W, bias, relu, ws, False)


def propagate_linear(g: Graph, X, W, w_csr=None, op="sum", bias=None, relu=False, ws=None, return_ws=False):
    """Y = act((op over incoming edges of w * X[source]) W + bias) in one kernel."""
    return _b.propagate_linear(_addr(g.c), X, W, w_csr, op, bias, relu, ws, return_ws)


def propagate_linear_backward(g: Graph, dY, X, W, w_csrT=None, op="sum", want_dX=True, want_dW=True, ws=None):
    """-> (dX or None, dW or None)"""
    return _b.propagate_linear_backward(_addr(g.c), dY, X, W, w_csrT, op, want_dX, want_dW, ws)


def linear_backward(X, W, dY, want_dX=True, want_dW=True, ws=None, return_ws=False):
    return _b.linear_backward(X, W, dY, want_dX, want_dW, ws, return_ws)


def axpby(alpha, a, beta, b, out=None):
    return _b.axpby(a, b, alpha, beta, out)
