"""GPU parity: the unfused primitives (gather, apply_edges, aggregate), edge softmax and batched
pooling against the CPU checker, through the C ABI."""
import numpy as np
import pytest

import oracle
from paper_2412_06354_b200 import synth
from util import assert_close, bits, f64_to_dtype_bits, host_bits, to_dev, to_host64
from test_gpu_propagate import build_graph, feats, host_csr, ragged_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gnn():
    from paper_2412_06354_b200 import gnn as g
    g.load()
    return g


@pytest.mark.parametrize("dtype,F", [("f32", 4), ("f32", 100), ("bf16", 8), ("bf16", 128)])
def test_gather_and_its_backward(gnn, dtype, F):
    n, src, dst = ragged_graph(50 + F)
    g = build_graph(gnn, n, src, dst)
    X = feats((n, F), dtype, 500 + F)
    for idx in (src, dst):
        out = gnn.gather(to_dev(idx), to_dev(X))
        assert np.array_equal(bits(out), host_bits(X[idx])), "gather is a bit-exact copy"
    R = feats((len(src), F), dtype, 501 + F)  # one row per edge, original edge order
    for by_src, idx in ((False, dst), (True, src)):
        dX = gnn.gather_backward(g, to_dev(R), by_src=by_src)
        ref, S = oracle.gather_backward(n, idx, R)
        assert_close(to_host64(dX), ref, S, dtype, f"gather_backward by_src={by_src}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_apply_edges_messages(gnn, dtype):
    H, C = 4, 16
    F = H * C
    n, src, dst = ragged_graph(60)
    g = build_graph(gnn, n, src, dst)
    ref = host_csr(n, src, dst)
    eid = ref["eid"]
    X = feats((n, F), dtype, 600)
    Xd = to_dev(X)
    m = gnn.apply_edges(g, gnn.COPY_XJ, Xd)
    assert np.array_equal(bits(m), host_bits(X[src[eid]]))
    for ew in (1, H, F):
        e = synth.uniform_f32((len(src), ew), -1.0, 1.0, 601 + ew)
        m = gnn.apply_edges(g, gnn.E_MUL_XJ, Xd, e=to_dev(e[eid]))
        mo = oracle.apply_edges(oracle.E_MUL_XJ, src, dst, X, e=e)[eid]
        assert_close(to_host64(m), mo, np.abs(mo), dtype, f"e_mul_xj width {ew}")
    if dtype == "f32":
        al = synth.normal_f32((n, H), 610)
        ar = synth.normal_f32((n, H), 611)
        s = gnn.apply_edges(g, gnn.GAT_LOGIT, to_dev(al), ar=to_dev(ar), slope=0.2)
        so = oracle.apply_edges(oracle.GAT_LOGIT, src, dst, al, Y=ar, slope=0.2)[eid]
        # a two-term sum: the scale is |al| + |ar| (times the slope on the negative side)
        scale = np.abs(al[src[eid]].astype(np.float64)) + np.abs(ar[dst[eid]].astype(np.float64))
        assert_close(to_host64(s), so, scale, "f32", "gat logit")


@pytest.mark.parametrize("dtype,F", [("f32", 64), ("bf16", 128), ("bf16", 40)])
def test_aggregate_matches_checker_and_fused_path(gnn, dtype, F):
    n, src, dst = ragged_graph(70 + F)
    g = build_graph(gnn, n, src, dst)
    eid = host_csr(n, src, dst)["eid"]
    X = feats((n, F), dtype, 700 + F)
    w = synth.uniform_f32((len(src),), 0.0, 1.0, 701)
    m = gnn.apply_edges(g, gnn.E_MUL_XJ, to_dev(X), e=to_dev(w[eid]))  # CSR order, stored dtype
    m_host = np.empty((len(src), F), np.float64)
    m_host[eid] = to_host64(m)  # the device's own messages, back in original edge order
    for op in ("sum", "mean", "max", "min"):
        got = gnn.aggregate(g, m, op)
        o, S, a = oracle.aggregate(op, n, dst, m_host)
        if op in ("max", "min"):
            out, arg = got
            assert np.array_equal(bits(out), f64_to_dtype_bits(o, dtype))
            ga = arg.cpu().numpy()
            assert np.array_equal(np.where(ga >= 0, eid[np.maximum(ga, 0)], -1), a)
            R = feats((n, F), dtype, 702)
            dm = gnn.aggregate_backward(g, to_dev(R), op, argmax=arg)
            dmo = oracle.aggregate_backward(op, n, dst, R, a)[eid]
            assert np.array_equal(bits(dm), f64_to_dtype_bits(dmo, dtype))
        else:
            assert_close(to_host64(got), o, S, dtype, f"aggregate {op}")
            R = feats((n, F), dtype, 703)
            dm = gnn.aggregate_backward(g, to_dev(R), op)
            dmo = oracle.aggregate_backward(op, n, dst, R)[eid]
            assert_close(to_host64(dm), dmo, np.abs(dmo), dtype, f"aggregate_backward {op}")
    # propagate == aggregate(apply_edges): fused and unfused agree (the unfused path rounds each
    # message to the storage dtype first, so agreement is within tolerance, not bitwise)
    fused = gnn.propagate_fused(g, to_dev(X), to_dev(w[eid]), "sum")
    o, S, _ = oracle.propagate("sum", n, src, dst, X, w)
    if dtype == "f32":  # bf16 messages carry a 2^-9 rounding each, which the fused path does not have
        assert_close(to_host64(gnn.aggregate(g, m, "sum")), o, S, dtype, "unfused vs checker")
    assert_close(to_host64(fused), o, S, dtype, "fused vs checker")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("H", [1, 3, 4, 8, 16, 32])
def test_edge_softmax_forward_backward(gnn, dtype, H):
    n, src, dst = ragged_graph(80 + H)  # hub row of 6000 edges takes the block-per-row path
    g = build_graph(gnn, n, src, dst)
    eid = host_csr(n, src, dst)["eid"]
    E = len(src)
    s = feats((E, H), dtype, 800 + H)
    if dtype == "f32":
        s = (s * 3).astype(np.float32)
    alpha, rmax, rsum = gnn.edge_softmax(g, to_dev(s[eid]), want_stats=True)
    ao = oracle.edge_softmax(n, dst, s)
    assert_close(to_host64(alpha), ao[eid], ao[eid], dtype, "alpha")
    tot = np.zeros((n, H))
    np.add.at(tot, dst, to_host64(alpha)[np.argsort(eid)])
    deg = np.bincount(dst, minlength=n)
    assert np.allclose(tot[deg > 0], 1.0, atol=2e-2 if dtype == "bf16" else 1e-5)
    smax = np.full((n, H), -np.inf)
    np.maximum.at(smax, dst, synth.to_f64(s))
    assert np.array_equal(to_host64(rmax)[deg > 0], smax[deg > 0])
    assert np.all(to_host64(rmax)[deg == 0] == 0) and np.all(to_host64(rsum)[deg == 0] == 0)
    # backward, from the device's own (rounded) alpha
    a_host = np.empty((E, H), np.float64)
    a_host[eid] = to_host64(alpha)
    R = feats((E, H), dtype, 801 + H)
    ds = gnn.edge_softmax_backward(g, alpha, to_dev(R[eid]))
    dso, S = oracle.edge_softmax_backward(n, dst, a_host, R)
    assert_close(to_host64(ds), dso[eid], S[eid], dtype, "dlogits")
    again = gnn.edge_softmax(g, to_dev(s[eid]))
    assert np.array_equal(bits(again), bits(alpha))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("H", [1, 4, 8, 32])
def test_edge_softmax_rows_of_tens_of_thousands_of_positions(gnn, dtype, H):
    """Three rows above 8192 positions (a cluster of blocks each when H is 4, 8 or 32; with 4 and 8 found at multiples of 4096 and 2048 positions,
    else two of them in one scan window and one a single position above the threshold); a band of rows of 513 ... 3000 positions (a block each, 4 and 8
    heads in chunks up to 4096 and 2048).  Over its own input the softmax goes by row length with every head count."""
    rng = np.random.default_rng(31 + H)
    n, e = 3000, 120000
    src = rng.integers(0, n, e).astype(np.int32)
    dst = rng.integers(0, n, e).astype(np.int32)
    dst[:20000] = 7
    dst[20000:29000] = 9
    dst[29000:37193] = 2990
    at = 40000
    for k in range(12):
        dst[at:at + 513 + 220 * k] = 300 + 5 * k
        at += 513 + 220 * k
    perm = rng.permutation(e)
    src, dst = src[perm].copy(), dst[perm].copy()
    g = build_graph(gnn, n, src, dst)
    eid = host_csr(n, src, dst)["eid"]
    s = feats((e, H), dtype, 900 + H)
    if dtype == "f32":
        s = (s * 3).astype(np.float32)
    alpha, rmax, rsum = gnn.edge_softmax(g, to_dev(s[eid]), want_stats=True)
    ao = oracle.edge_softmax(n, dst, s)
    assert_close(to_host64(alpha), ao[eid], ao[eid], dtype, "alpha")
    deg = np.bincount(dst, minlength=n)
    smax = np.full((n, H), -np.inf)
    np.maximum.at(smax, dst, synth.to_f64(s))
    assert np.array_equal(to_host64(rmax)[deg > 0], smax[deg > 0])
    ssum = np.zeros((n, H))
    np.add.at(ssum, dst, np.exp(synth.to_f64(s) - smax[dst]))
    assert np.allclose(to_host64(rsum)[deg > 0], ssum[deg > 0], rtol=1e-4)
    a_host = np.empty((e, H), np.float64)
    a_host[eid] = to_host64(alpha)
    R = feats((e, H), dtype, 901 + H)
    ds = gnn.edge_softmax_backward(g, alpha, to_dev(R[eid]))
    dso, S = oracle.edge_softmax_backward(n, dst, a_host, R)
    assert_close(to_host64(ds), dso[eid], S[eid], dtype, "dlogits")
    again = gnn.edge_softmax(g, to_dev(s[eid]))
    assert np.array_equal(bits(again), bits(alpha))
    assert np.array_equal(bits(gnn.edge_softmax_backward(g, alpha, to_dev(R[eid]))), bits(ds))
    own, upstream = to_dev(s[eid]), to_dev(R[eid])
    gnn._check(gnn.load().gnn_edge_softmax(gnn.C.byref(g.c), gnn._p(own), H, gnn._dtype(own), gnn._p(own), None, None, gnn._stream()))
    assert_close(to_host64(own), ao[eid], ao[eid], dtype, "alpha over the logits")
    gnn._check(gnn.load().gnn_edge_softmax_backward(gnn.C.byref(g.c), gnn._p(alpha), gnn._p(upstream), H, gnn._dtype(own), gnn._p(upstream), gnn._stream()))
    assert_close(to_host64(upstream), dso[eid], S[eid], dtype, "dlogits over dalpha")


# One row beside short ones: as long as the chunk kernels take, one position more, and over many blocks' chunks.  Up to 8192 edges they take any row.
@pytest.mark.parametrize("H,longest,e", [(8, 2048, 20_000), (8, 2049, 20_000), (4, 4096, 30_000), (4, 4097, 30_000), (8, 8000, 8192), (4, 8193, 8193), (8, 8192, 430_000), (8, 8193, 430_000), (4, 120_000, 900_000)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_edge_softmax_one_long_row(gnn, dtype, H, longest, e):
    rng = np.random.default_rng(longest + H)
    n = e // 7
    dst = np.sort(np.concatenate([np.full(longest, n // 2), rng.integers(0, n, e - longest)])).astype(np.int32)
    src = rng.integers(0, n, e).astype(np.int32)
    keep = (dst == n // 2).nonzero()[0][longest:]  # (exactly `longest` positions)
    dst[keep] = n // 2 + 1
    g = build_graph(gnn, n, src, dst)  # sorted by target: positions are in the order of the list
    s, R = feats((e, H), dtype, 940 + H), feats((e, H), dtype, 941 + H)
    alpha, top, total = gnn.edge_softmax(g, to_dev(s), want_stats=True)
    ao = oracle.edge_softmax(n, dst, s)
    assert_close(to_host64(alpha), ao, ao, dtype, "alpha")
    x = synth.to_f64(s)
    most, sums = np.full((n, H), -np.inf), np.zeros((n, H))
    np.maximum.at(most, dst, x)
    np.add.at(sums, dst, np.exp(x - most[dst]))
    most[np.isinf(most)] = 0.0
    assert np.array_equal(to_host64(top), most)
    assert_close(to_host64(total), sums, sums, "f32", "sums of the rows")
    dso, S = oracle.edge_softmax_backward(n, dst, to_host64(alpha), R)
    assert_close(to_host64(gnn.edge_softmax_backward(g, alpha, to_dev(R))), dso, S, dtype, "dlogits")


def test_edge_softmax_time_of_a_very_long_row(gnn):
    """A row of 2.4 M positions (a readout node) is read a fixed number of times: 21 times as long as rows of 8 when measured, 240 times with every
    block that it reaches reading all of it."""
    import torch
    e, H = 2_400_000, 8
    times = []
    for dst in (torch.arange(e, device="cuda") // 8, torch.zeros(e, device="cuda")):
        g = gnn.coo_to_csr(e // 8, torch.randint(e // 8, (e,), device="cuda", dtype=torch.int32), dst.to(torch.int32))
        s, R = torch.randn(e, H, device="cuda"), torch.randn(e, H, device="cuda")
        for f in (lambda: gnn.edge_softmax(g, s), lambda: gnn.edge_softmax_backward(g, s, R)):
            f()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                f()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
    assert times[2] < 80 * times[0] and times[3] < 80 * times[1], times


@pytest.mark.parametrize("H,n,dtype", [(8, 50_000, "f32"), (8, 50_000, "bf16"), (4, 14_000, "f32")])
def test_edge_softmax_of_many_long_rows(gnn, H, n, dtype):
    """Rows that are long on average take a warp, a block or a cluster each, and no more time than over their own input, which always does."""
    import torch
    e = 2_100_000
    rng = np.random.default_rng(n)
    dst = np.sort(rng.integers(0, n, e)).astype(np.int32)
    dst[400_000:409_000], dst[500_000:500_700] = dst[400_000], dst[500_000]
    g = build_graph(gnn, n, rng.integers(0, n, e).astype(np.int32), dst)
    s, R = feats((e, H), dtype, 950 + H), feats((e, H), dtype, 951 + H)
    S, up = to_dev(s), to_dev(R)
    alpha = gnn.edge_softmax(g, S)
    ao = oracle.edge_softmax(n, dst, s)
    assert_close(to_host64(alpha), ao, ao, dtype, "alpha")
    dso, terms = oracle.edge_softmax_backward(n, dst, to_host64(alpha), R)
    assert_close(to_host64(gnn.edge_softmax_backward(g, alpha, up)), dso, terms, dtype, "dlogits")
    own, times = S.clone(), []
    for f in (lambda: gnn.edge_softmax(g, S), lambda: gnn._check(gnn.load().gnn_edge_softmax(gnn.C.byref(g.c), gnn._p(own), H, gnn._dtype(own), gnn._p(own), None, None, gnn._stream()))):
        f()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            f()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert times[0] < 1.2 * times[1], times  # (by chunks: 1.4 to 1.7 times as long)


def test_edge_softmax_degenerate(gnn):
    import torch
    # one edge -> 1; equal logits -> 1/deg; huge logits do not overflow
    src = np.array([0, 1, 2, 3, 1], np.int32)
    dst = np.array([4, 4, 4, 0, 0], np.int32)
    g = build_graph(gnn, 5, src, dst)
    eid = g.eid[:5].cpu().numpy()
    s = np.array([[1000.0], [1000.0], [1000.0], [-50.0], [30.0]], np.float32)
    a = to_host64(gnn.edge_softmax(g, to_dev(s[eid])))
    back = np.empty_like(a)
    back[eid] = a
    assert np.allclose(back[:3, 0], 1 / 3, rtol=1e-6) and abs(back[3, 0] - np.exp(-80.0)) < 1e-40 and abs(back[4, 0] - 1) < 1e-6
    g0 = build_graph(gnn, 3, np.zeros(0, np.int32), np.zeros(0, np.int32))
    gnn.edge_softmax(g0, torch.empty((0, 4), device="cuda"))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_batched_pooling(gnn, dtype):
    """512 graphs of 10-40 nodes, F=128: mean-aggregation layer on the batch, then pooling."""
    wl = synth.workload_batched()
    n, G, F, gp = wl["N"], wl["G"], wl["F"], wl["graph_ptr"]
    X = wl["X"] if dtype == "f32" else synth.normal_bf16((n, F), synth.BASE_SEED + 2, 10)
    gid = np.repeat(np.arange(G), np.diff(gp)).astype(np.int32)
    gptr = gnn.graph_ptr_from_ids(to_dev(gid), G)
    assert np.array_equal(gptr.cpu().numpy(), gp.astype(np.int64))
    g = build_graph(gnn, n, wl["src"], wl["dst"])
    h = gnn.propagate_fused(g, to_dev(X), None, "mean")
    ho, S, _ = oracle.propagate("mean", n, wl["src"], wl["dst"], X)
    assert_close(to_host64(h), ho, S, dtype, "mean layer on the batch")
    R = feats((G, F), dtype, 900)
    for op in ("sum", "mean", "max", "min"):
        got = gnn.reduce_nodes(gptr, to_dev(X), op)
        o, S, a = oracle.reduce_nodes(op, gp, X)
        if op in ("max", "min"):
            out, arg = got
            assert np.array_equal(bits(out), f64_to_dtype_bits(o, dtype))
            assert np.array_equal(arg.cpu().numpy(), a)
            dX = gnn.reduce_nodes_backward(gptr, to_dev(R), n, op, argmax=arg)
            assert np.array_equal(bits(dX), f64_to_dtype_bits(oracle.reduce_nodes_backward(op, gp, R, a), dtype))
        else:
            assert_close(to_host64(got), o, S, dtype, f"reduce_nodes {op}")
            dX = gnn.reduce_nodes_backward(gptr, to_dev(R), n, op)
            ref = oracle.reduce_nodes_backward(op, gp, R)
            assert_close(to_host64(dX), ref, np.abs(ref), dtype, f"reduce_nodes_backward {op}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_pooling_over_graphs_of_a_million_nodes(gnn, dtype):
    """Two graphs of 700000 and 499980 nodes around one of 20: a graph spans thousands of chunks of the reduction,
    so its partial results are combined by the block-per-row pass, for max / min with the winning positions."""
    import torch
    sizes = [700_000, 20, 499_980]
    gp = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, F = int(gp[-1]), 32
    X = feats((n, F), dtype, 1234)
    p0 = int(oracle.reduce_nodes("max", gp, X)[2][0, 0])  # the winner of column 0 in the first graph ...
    X[(p0 + 350_000) % 700_000] = X[p0]                   # ... now has a twin far away: the smaller position wins
    gptr = to_dev(gp)
    R = feats((3, F), dtype, 1235)
    for op in ("mean", "max", "min"):
        got = gnn.reduce_nodes(gptr, to_dev(X), op)
        o, S, a = oracle.reduce_nodes(op, gp, X)
        if op in ("max", "min"):
            out, arg = got
            assert np.array_equal(bits(out), f64_to_dtype_bits(o, dtype))
            assert np.array_equal(arg.cpu().numpy(), a)
            again = gnn.reduce_nodes(gptr, to_dev(X), op)
            assert torch.equal(again[1], arg)
        else:
            assert_close(to_host64(got), o, S, dtype, f"reduce_nodes {op}")


def test_pooling_edge_cases(gnn):
    import torch
    # an empty graph in the middle of the batch, and unsorted ids
    gid = to_dev(np.array([0, 0, 2, 2, 2], np.int32))
    gptr = gnn.graph_ptr_from_ids(gid, 4)
    assert gptr.cpu().tolist() == [0, 2, 2, 5, 5]
    X = to_dev(feats((5, 8), "f32", 1))
    out, arg = gnn.reduce_nodes(gptr, X, "max")
    assert torch.count_nonzero(out[1]) == 0 and bool((arg[1] == -1).all()) and bool((arg[3] == -1).all())
    assert torch.equal(out[0], torch.maximum(X[0], X[1]))
    with pytest.raises(gnn.GnnError) as e:
        gnn.graph_ptr_from_ids(to_dev(np.array([0, 2, 1], np.int32)), 3)
    assert e.value.status == 3
    with pytest.raises(gnn.GnnError) as e:
        gnn.graph_ptr_from_ids(to_dev(np.array([0, 1, 5], np.int32)), 3)
    assert e.value.status == 3


# Nodes before graph_ptr[0] and from graph_ptr[G] on (a padded X) belong to no graph: inside a warp's share, whole shares and whole
# blocks of them, for every number of lane groups, positions first and (last two) a row per lane group.
@pytest.mark.parametrize("gp,n,dtype,F", [
    ([0, 10, 20], 64, "f32", 128), ([0, 10, 20], 64, "f32", 4), ([37, 45], 400, "bf16", 8), ([300, 300, 301, 333], 5000, "f32", 32),
    ([5, 9, 64], 64, "f32", 64), ([0, 64, 128], 1000, "bf16", 64), ([9000, 150_000, 290_000], 300_000, "f32", 16),
    ([0, 1, 270_001], 600_000, "bf16", 256), ([3, 3, 5, 9, 9, 12, 13, 14, 15, 16, 17, 20], 40, "f32", 12), ([40] * 8, 40, "f32", 4)])
def test_pooling_leaves_nodes_of_no_graph_out(gnn, gp, n, dtype, F):
    import torch
    gp = np.array(gp, np.int64)
    G, lo, hi = len(gp) - 1, int(gp[0]), int(gp[-1])
    X, R = feats((n, F), dtype, 40), feats((G, F), dtype, 41)
    inner = gp - lo
    for op in ("sum", "mean", "max", "min"):
        got = gnn.reduce_nodes(to_dev(gp), to_dev(X), op)
        o, S, a = oracle.reduce_nodes(op, inner, X[lo:hi])
        arg = None
        if op in ("max", "min"):
            got, arg = got
            a = np.where(a >= 0, a + lo, a)
            assert np.array_equal(bits(got), f64_to_dtype_bits(o, dtype)) and np.array_equal(arg.cpu().numpy(), a)
        else:
            assert_close(to_host64(got), o, S, dtype, op)
        dX = gnn.reduce_nodes_backward(to_dev(gp), to_dev(R), n, op, argmax=arg)
        assert torch.count_nonzero(dX[:lo]) == 0 and torch.count_nonzero(dX[hi:]) == 0
        ref = oracle.reduce_nodes_backward(op, inner, R, None if arg is None else np.where(a >= 0, a - lo, a))
        assert_close(to_host64(dX[lo:hi]), ref, np.abs(ref), dtype, f"backward {op}")


# Four 256-thread tiles of (edge, 16-byte chunk) pairs per block; the backward pass takes 8 to 128 positions per warp: rows of
# one chunk, of a number of chunks that divides nothing, and of more than 4096 chunks (64 KB), which divide instead of multiplying
@pytest.mark.parametrize("e,dtype,F", [(1, "f32", 4), (65, "bf16", 8), (1025, "f32", 4), (700, "bf16", 56), (70_001, "f32", 12), (131_200, "bf16", 24), (525_000, "f32", 4), (67, "f32", 16_420)])
def test_edge_tensor_tiles(gnn, e, dtype, F):
    import torch
    rng = np.random.default_rng(e)
    n = 50
    src, dst = rng.integers(0, n, e).astype(np.int32), np.sort(rng.integers(0, n - 3, e)).astype(np.int32)  # edge order = CSR order
    g = build_graph(gnn, n, src, dst)
    X, R = feats((n, F), dtype, 900 + F), feats((n, F), dtype, 901 + F)
    assert np.array_equal(bits(gnn.gather(to_dev(src), to_dev(X))), host_bits(X[src]))
    f = np.float32(2.0) ** rng.integers(-3, 4, (e, 1)).astype(np.float32)  # powers of two: products are exact
    m = gnn.apply_edges(g, gnn.E_MUL_XJ, to_dev(X), e=to_dev(f))
    assert np.array_equal(to_host64(m), to_host64(to_dev(X))[src] * f)
    assert np.array_equal(bits(gnn.aggregate_backward(g, to_dev(R), "sum")), host_bits(R[dst]))
    mean = gnn.aggregate_backward(g, to_dev(R), "mean")
    ref = to_host64(to_dev(R))[dst] / np.bincount(dst, minlength=n)[dst][:, None]
    assert_close(to_host64(mean), ref, np.abs(ref), dtype, "mean")
    first = np.searchsorted(dst, np.arange(n))
    count = np.bincount(dst, minlength=n)
    win = np.where(count > 0, first + rng.integers(0, 1 << 30, n) % np.maximum(count, 1), -1)
    arg = np.repeat(win[:, None], F, 1).astype(np.int32)
    arg[:, ::3] = np.where(count > 0, first, -1)[:, None]
    want = np.where(arg[dst] == np.arange(e)[:, None], to_host64(to_dev(R))[dst], 0.0)
    off = torch.empty(n * F + 1, dtype=torch.int32, device="cuda")[1:].view(n, F)  # winners that start off 16 bytes
    off.copy_(to_dev(arg))
    for a in (to_dev(arg), off):
        assert np.array_equal(to_host64(gnn.aggregate_backward(g, to_dev(R), "max", argmax=a)), want)


# Rows of whole 16-byte chunks, single elements (four to a thread) and other widths; perm of one block less, exactly and more
@pytest.mark.parametrize("e", [1, 1023, 1024, 1025, 70_001])
@pytest.mark.parametrize("width,dtype", [(1, "int32"), (1, "uint8"), (3, "float32"), (4, "float32"), (8, "float32"), (8, "bfloat16"), (2, "float64"), (16, "uint8")])
def test_permuted_edge_data(gnn, e, width, dtype):
    import torch
    perm = torch.randperm(e, device="cuda").to(torch.int32)
    data = torch.randint(0, 200, (e + 1, width) if width > 1 else (e + 1,), device="cuda").to(getattr(torch, dtype))[1:]  # (off 16 bytes where a row is less)
    out = gnn.permute_edge_data(perm, data)
    assert torch.equal(out, data[perm.long()])


# fp32 rows over 256 bytes take 32 bytes per lane where matrices lie on 32 bytes, 16 otherwise: one warp's share of positions less, exactly and more
@pytest.mark.parametrize("e", [1, 63, 64, 65, 513, 6001])
@pytest.mark.parametrize("H,C", [(1, 128), (4, 32), (2, 64), (1, 72), (8, 16)])
def test_gatv2_logits_lane_widths(gnn, e, H, C):
    import torch
    rng = np.random.default_rng(e)
    n, F = 97, H * C
    src, dst = rng.integers(0, n, e).astype(np.int32), np.sort(rng.integers(0, n, e).astype(np.int32))
    g = build_graph(gnn, n, src, dst)
    eid = host_csr(n, src, dst)["eid"]
    Xl, Xr, a = feats((n, F), "f32", 70), feats((n, F), "f32", 71), feats((H, C), "f32", 72)
    z = synth.to_f64(Xl)[src] + synth.to_f64(Xr)[dst]
    terms = (np.where(z > 0, z, 0.2 * z) * synth.to_f64(a).reshape(1, F)).reshape(e, H, C)
    for off in (0, 4):  # elements before the matrix
        room = torch.zeros(n * F + off, device="cuda")
        room[off:] = to_dev(Xl).reshape(-1)
        got = gnn.gatv2_logits(g, room[off:].view(n, F), to_dev(Xr), to_dev(a), H, 0.2)
        assert_close(to_host64(got).reshape(e, H), terms.sum(-1)[eid], np.abs(terms).sum(-1)[eid], "f32", f"logits, offset {off}")
