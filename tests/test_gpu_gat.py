"""GPU parity: fused GAT core, forward and backward, against the CPU checker."""
import numpy as np
import pytest

import oracle
from paper_2412_06354_b200 import synth
from util import assert_close, to_dev, to_host64
from test_gpu_propagate import build_graph, ragged_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gnn():
    from paper_2412_06354_b200 import gnn as g
    g.load()
    return g


def run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, dtype, what, masked=()):
    """masked: nodes whose scores al are below the range of fp32"""
    F = H * C
    g = build_graph(gnn, n, src, dst)
    eid = g.eid[:g.E].cpu().numpy() if g.E else np.zeros(0, np.int64)
    fwd = gnn.gat_fused(g, to_dev(Wx), to_dev(a_s), to_dev(a_d), H)
    ref = oracle.gat(n, src, dst, Wx, a_s, a_d, H, C)
    x64 = synth.to_f64(Wx).reshape(n, H, C)
    Sal = np.einsum("nhc,hc->nh", np.abs(x64), np.abs(a_s.astype(np.float64)))
    Sar = np.einsum("nhc,hc->nh", np.abs(x64), np.abs(a_d.astype(np.float64)))
    seen = np.setdiff1d(np.arange(n), masked)
    assert_close(to_host64(fwd["al"])[seen], ref["al"][seen], Sal[seen], "f32", what + " al")
    assert np.all(to_host64(fwd["al"])[np.asarray(masked, int)] == -np.inf)
    assert_close(to_host64(fwd["ar"]), ref["ar"], Sar, "f32", what + " ar")
    if g.E:
        # a coefficient moves by about (error of its logit) * alpha; the logit is a two-dot-product sum
        scale = ref["alpha"][eid] * np.maximum(1.0, Sal[src[eid]] + Sar[dst[eid]])
        assert_close(to_host64(fwd["alpha"]), ref["alpha"][eid], scale, "f32", what + " alpha")
    assert_close(to_host64(fwd["out"]), ref["out"], ref["S"], dtype, what + " out")

    R = synth.normal((n, F), dtype, 4242, 3)
    bw = gnn.gat_fused_backward(g, to_dev(Wx), to_dev(a_s), to_dev(a_d), fwd, to_dev(R), H)
    rb = oracle.gat_backward(n, src, dst, Wx, a_s, a_d, H, C, ref, R)
    # LeakyReLU'(z) is decided by the sign of z.  Where |z| is below the fp32 resolution of its terms the
    # two precisions may decide differently: such an edge moves dz[k,h] by at most |ds[k,h]|*(1-slope), which
    # reaches dal[src], dar[dst] and, through them, three outputs.  The allowance is accumulated from the
    # checker's own intermediates and added to the bound of exactly the elements it can reach.
    slope = 0.2
    z = ref["al"][src] + ref["ar"][dst]
    risky = np.abs(z) < 2e-6 * (Sal[src] + Sar[dst])
    assert risky.mean() < 0.01, risky.mean()
    r64 = synth.to_f64(R).reshape(n, H, C)
    dalpha = np.empty((len(src), H))
    for h in range(H):
        dalpha[:, h] = (r64[dst, h, :] * x64[src, h, :]).sum(axis=1)
    ds, _ = oracle.edge_softmax_backward(n, dst, ref["alpha"], dalpha) if len(src) else (np.zeros((0, H)), None)
    slack = np.where(risky, np.abs(ds) * (1.0 - slope), 0.0)
    sl_al, sl_ar = np.zeros((n, H)), np.zeros((n, H))
    for h in range(H):
        sl_al[:, h] = np.bincount(src, weights=slack[:, h], minlength=n)
        sl_ar[:, h] = np.bincount(dst, weights=slack[:, h], minlength=n)
    as64, ad64 = np.abs(a_s.astype(np.float64)), np.abs(a_d.astype(np.float64))
    extra_dWx = (sl_al[:, :, None] * as64[None] + sl_ar[:, :, None] * ad64[None]).reshape(n, F)
    extra_src = np.einsum("nh,nhc->hc", sl_al, np.abs(x64))
    extra_dst = np.einsum("nh,nhc->hc", sl_ar, np.abs(x64))
    assert_close(to_host64(bw["dWx"]), rb["dWx"], rb["SdWx"], dtype, what + " dWx", extra=extra_dWx)
    assert_close(to_host64(bw["da_src"]), rb["da_src"], rb["Sda_src"], "f32", what + " da_src", extra=extra_src)
    assert_close(to_host64(bw["da_dst"]), rb["da_dst"], rb["Sda_dst"], "f32", what + " da_dst", extra=extra_dst)
    return g, fwd


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("H,C", [(4, 16), (8, 32), (1, 64), (2, 8), (16, 8), (32, 8), (8, 64)])
def test_gat_ragged(gnn, dtype, H, C):
    n, src, dst = ragged_graph(90 + H)
    Wx = synth.normal((n, H * C), dtype, 900 + H, 1)
    a = (6.0 / (C + 1)) ** 0.5
    a_s = synth.uniform_f32((H, C), -a, a, 901, 1)
    a_d = synth.uniform_f32((H, C), -a, a, 902, 1)
    run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, dtype, f"gat H={H} C={C} {dtype}")


@pytest.mark.parametrize("H,C", [(1, 64), (2, 16)])
def test_gat_one_and_two_heads_with_source_hubs(gnn, H, C):
    """Sources with 5000 and 1025 outgoing edges: the per-source sum of the logit gradients takes the
    block-per-row path (one and two heads do not go through the chunked reduction)."""
    n, src, dst = ragged_graph(97 + H)
    src = src.copy()
    src[100:5100] = 11
    src[6000:7025] = 1499
    Wx = synth.normal((n, H * C), "f32", 960 + H, 1)
    a = (6.0 / (C + 1)) ** 0.5
    a_s = synth.uniform_f32((H, C), -a, a, 961, 1)
    a_d = synth.uniform_f32((H, C), -a, a, 962, 1)
    run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", f"gat source hubs H={H}")


# The row kernels of four and eight heads take chunks of positions: 512 and 256 on small graphs, 2048 and 1024 from 800 and 400 Ki edges on.
# The gradient takes rows by length below 48 Ki and 24 Ki edges.  Rows that fill a chunk, end one before or one past its end, lie over several chunks, empty rows at the seams, a last chunk of a few.
@pytest.mark.parametrize("H,chunk,edges", [(4, 512, 9_001), (8, 256, 4_611), (8, 256, 256), (4, 512, 49_151), (4, 512, 49_152), (8, 256, 24_576), (8, 1024, 420_003), (4, 2048, 830_011)])
def test_gat_and_softmax_rows_at_chunk_ends(gnn, H, chunk, edges):
    rng = np.random.default_rng(edges)
    degree = [chunk, 0, chunk - 1, 1, chunk + 1, chunk - 2, 1, 3 * chunk, 0, 0, 5, 2 * chunk - 5] if edges > chunk else []
    while sum(degree) < edges:
        degree += [min(int(d), edges - sum(degree)) for d in rng.integers(0, 40, 1 if edges - sum(degree) < 4000 else 100)]
    n = len(degree)
    order = rng.permutation(edges)
    dst = np.repeat(np.arange(n, dtype=np.int32), degree)[order]
    src = rng.integers(0, n, edges).astype(np.int32)
    C = 8
    Wx = synth.normal((n, H * C), "f32", 910 + H, 1)
    a_s = synth.uniform_f32((H, C), -0.8, 0.8, 911, 1)
    a_d = synth.uniform_f32((H, C), -0.8, 0.8, 912, 1)
    g, _ = run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", f"gat H={H}, chunks of {chunk}")
    eid = g.eid[:g.E].cpu().numpy()
    for dtype in ("f32", "bf16"):
        logits, R = synth.normal((edges, H), dtype, 913, 1), synth.normal((edges, H), dtype, 914, 1)
        alpha, top, total = gnn.edge_softmax(g, to_dev(logits[eid]), want_stats=True)
        ao = oracle.edge_softmax(n, dst, logits)
        assert_close(to_host64(alpha), ao[eid], ao[eid], dtype, "alpha")
        x = synth.to_f64(logits)
        most = np.full((n, H), -np.inf)
        np.maximum.at(most, dst, x)
        sums = np.zeros((n, H))
        np.add.at(sums, dst, np.exp(x - most[dst]))
        most[np.array(degree) == 0] = 0.0  # what a row without edges has
        assert np.array_equal(to_host64(top), most)
        assert_close(to_host64(total), sums, sums, "f32", "sums of the rows")
        a_host = np.empty((edges, H))
        a_host[eid] = to_host64(alpha)
        ds = gnn.edge_softmax_backward(g, alpha, to_dev(R[eid]))
        dso, S = oracle.edge_softmax_backward(n, dst, a_host, R)
        assert_close(to_host64(ds), dso[eid], S[eid], dtype, "dlogits")
        # written over their own input (no chunks then): within the same bounds
        own, upstream = to_dev(logits[eid]).clone(), to_dev(R[eid]).clone()
        gnn._check(gnn.load().gnn_edge_softmax(gnn.C.byref(g.c), gnn._p(own), H, gnn._dtype(own), gnn._p(own), None, None, gnn._stream()))
        assert_close(to_host64(own), ao[eid], ao[eid], dtype, "alpha over the logits")
        gnn._check(gnn.load().gnn_edge_softmax_backward(gnn.C.byref(g.c), gnn._p(alpha), gnn._p(upstream), H, gnn._dtype(own), gnn._p(upstream), gnn._stream()))
        assert_close(to_host64(upstream), dso[eid], S[eid], dtype, "dlogits over dalpha")


# Logits of -inf (scores that overflow) take no part in their rows, wherever the chunks cut them: a single position past a chunk's end, a
# chunk's whole share in the middle or at the beginning of a row, scattered ones.
@pytest.mark.parametrize("H,chunk,edges", [(4, 512, 9_001), (8, 256, 6_611), (4, 512, 50_003), (8, 256, 25_001), (8, 1024, 420_003), (4, 2048, 830_011)])
def test_gat_scores_of_minus_infinity(gnn, H, chunk, edges):
    rng = np.random.default_rng(edges)
    degree = [chunk + 1, 3 * chunk, 2 * chunk]
    while sum(degree) < edges:
        degree.append(min(int(rng.integers(1, 3000)), edges - sum(degree)))
    n, C = max(len(degree), 500), 8
    dst = np.repeat(np.arange(len(degree), dtype=np.int32), degree)  # positions in the order of the edge list
    hidden = np.arange(n - 5, n)
    src = rng.integers(0, n - 5, edges).astype(np.int32)
    away = rng.random(edges) < 0.05
    away[np.cumsum(degree) - 1] = False  # no row of nothing else
    away[chunk] = True
    away[2 * chunk:3 * chunk] = True
    away[4 * chunk + 1:5 * chunk] = True
    src[away] = rng.choice(hidden, away.sum())
    Wx = synth.normal((n, H * C), "f32", 920 + H, 1).reshape(n, H, C)
    Wx[:, :, 0] = 0.0
    Wx[hidden, :, 0] = -1e37
    a_s = synth.uniform_f32((H, C), -0.8, 0.8, 921, 1)
    a_d = synth.uniform_f32((H, C), -0.8, 0.8, 922, 1)
    a_s[:, 0], a_d[:, 0] = 100.0, 0.0
    Wx = Wx.reshape(n, H * C)
    _, fwd = run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", f"gat H={H}, chunks of {chunk}, scores of -inf", masked=hidden)
    # rows of nothing but -inf, cut and whole, are NaN; the others are what they were
    rows = np.array([1, 3, 5])
    src[np.isin(dst, rows)] = hidden[0]
    alpha = to_host64(gnn.gat_fused(build_graph(gnn, n, src, dst), to_dev(Wx), to_dev(a_s), to_dev(a_d), H)["alpha"])
    assert np.isnan(alpha[np.isin(dst, rows)]).all()
    others = ~np.isin(dst, rows)
    assert np.array_equal(alpha[others], to_host64(fwd["alpha"])[others])


# Few edges on many nodes: rows one by one below 150 k / heads edges on more nodes than edges, chunks from there on
@pytest.mark.parametrize("H,n,edges", [(4, 9_000, 8_999), (4, 9_000, 9_000), (8, 60_000, 1_000), (8, 18_760, 18_750), (8, 18_760, 18_749), (4, 40_000, 37_500), (4, 40_000, 37_499)])
def test_gat_mostly_empty_rows(gnn, H, n, edges):
    rng = np.random.default_rng(n + edges)
    src, dst = rng.integers(0, n, edges).astype(np.int32), rng.integers(0, n, edges).astype(np.int32)
    C = 8
    Wx = synth.normal((n, H * C), "f32", 930 + H, 1)
    a_s, a_d = synth.uniform_f32((H, C), -0.8, 0.8, 931, 1), synth.uniform_f32((H, C), -0.8, 0.8, 932, 1)
    g, _ = run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", f"gat H={H}, {edges} edges on {n} nodes")
    eid = g.eid[:g.E].cpu().numpy()
    logits = synth.normal((edges, H), "f32", 933, 1)
    alpha, top, total = gnn.edge_softmax(g, to_dev(logits[eid]), want_stats=True)
    ao = oracle.edge_softmax(n, dst, logits)
    assert_close(to_host64(alpha), ao[eid], ao[eid], "f32", "alpha")
    most, sums = np.full((n, H), -np.inf), np.zeros((n, H))
    np.maximum.at(most, dst, synth.to_f64(logits))
    np.add.at(sums, dst, np.exp(synth.to_f64(logits) - most[dst]))
    most[np.isinf(most)] = 0.0
    assert np.array_equal(to_host64(top), most)
    assert_close(to_host64(total), sums, sums, "f32", "sums of the rows")


# A row over so many chunks that its shares are combined by a kernel of their own: in one chunk less (2048 of them), exactly and more
@pytest.mark.parametrize("H,positions", [(8, 2047 * 1024 + 5), (8, 2048 * 1024 + 5), (8, 2_300_000), (4, 2048 * 2048 + 5)])
def test_gat_row_of_millions(gnn, H, positions):
    n, C, before = 250_000, 8 if H == 4 else 4, 1_000
    rng = np.random.default_rng(positions)
    others = rng.integers(0, n, 400_000)
    dst = np.sort(np.concatenate([np.full(before, 0), np.full(positions, 1), others[others > 1]])).astype(np.int32)  # the row begins inside the first chunk
    src = rng.integers(0, n, len(dst)).astype(np.int32)
    Wx = synth.normal((n, H * C), "f32", 937, 1)
    a_s, a_d = synth.uniform_f32((H, C), -0.8, 0.8, 938, 1), synth.uniform_f32((H, C), -0.8, 0.8, 939, 1)
    oracle.set_threads(8)
    try:
        run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", f"gat H={H}, a row of {positions}")
    finally:
        oracle.set_threads(1)


def test_gat_gradient_of_many_long_rows(gnn):
    """3.1 M edges, rows of 70 on average: by length"""
    n, e, H, C = 43_000, 3_100_000, 8, 8
    rng = np.random.default_rng(n)
    src, dst = rng.integers(0, n, e).astype(np.int32), rng.integers(0, n, e).astype(np.int32)
    Wx = synth.normal((n, H * C), "f32", 934, 1)
    a_s, a_d = synth.uniform_f32((H, C), -0.8, 0.8, 935, 1), synth.uniform_f32((H, C), -0.8, 0.8, 936, 1)
    oracle.set_threads(8)
    try:
        run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", "gat, long rows")
    finally:
        oracle.set_threads(1)


def test_softmax_time_of_a_thousand_edges_on_two_million_nodes(gnn):
    """No longer than three times what 16 heads, twice the values, take (by chunks: 15 times as long as these)."""
    import torch
    n, e, C = 2_000_000, 1_000, 4
    src, dst = (torch.randint(n, (e,), device="cuda", dtype=torch.int32) for _ in range(2))
    g = gnn.coo_to_csr(n, src, dst)
    times = []
    for H in (4, 8, 16):
        s = torch.randn(e, H, device="cuda")
        gnn.edge_softmax(g, s, want_stats=True)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            gnn.edge_softmax(g, s, want_stats=True)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    assert max(times[:2]) < 3 * times[2], times


def test_gat_zero_attention_is_mean_aggregation(gnn):
    n, src, dst = ragged_graph(95)
    H, C = 4, 16
    Wx = synth.normal_f32((n, H * C), 950)
    zero = np.zeros((H, C), np.float32)
    g = build_graph(gnn, n, src, dst)
    fwd = gnn.gat_fused(g, to_dev(Wx), to_dev(zero), to_dev(zero), H)
    o, S, _ = oracle.propagate("mean", n, src, dst, Wx)
    assert_close(to_host64(fwd["out"]), o, S, "f32", "alpha = 1/deg")


def test_gat_degenerate(gnn):
    import torch
    H, C = 2, 8
    a_s = to_dev(synth.normal_f32((H, C), 1))
    g = build_graph(gnn, 4, np.zeros(0, np.int32), np.zeros(0, np.int32))
    Wx = to_dev(synth.normal_f32((4, H * C), 2))
    fwd = gnn.gat_fused(g, Wx, a_s, a_s, H)
    assert torch.count_nonzero(fwd["out"]) == 0
    bw = gnn.gat_fused_backward(g, Wx, a_s, a_s, fwd, Wx, H)
    assert torch.count_nonzero(bw["dWx"]) == 0 and torch.count_nonzero(bw["da_src"]) == 0
    with pytest.raises(gnn.GnnError) as e:  # three heads
        gnn.gat_fused(g, to_dev(synth.normal_f32((4, 24), 3)), a_s, a_s, 3)
    assert e.value.status == 5
    # a head of 24 bf16 values (three 16-byte chunks) is refused by the forward and the backward call alike
    Wx3 = to_dev(synth.normal_bf16((4, 48), 4))
    a3 = to_dev(synth.normal_f32((2, 24), 5))
    with pytest.raises(gnn.GnnError) as e:
        gnn.gat_fused(g, Wx3, a3, a3, 2)
    assert e.value.status == 5


def test_gat_attention_workload_full_size(gnn):
    """R-MAT N=100000, 1.6M directed edges, 8 heads x 32 features bf16."""
    wl = synth.workload_attention()
    oracle.set_threads(8)
    try:
        run_case(gnn, wl["N"], wl["src"], wl["dst"], wl["Wx"], wl["a_src"], wl["a_dst"], wl["H"], wl["C"], "bf16", "attention workload")
    finally:
        oracle.set_threads(1)


@pytest.mark.parametrize("E", [8_400_000, 17_000_000])
def test_gat_more_than_8mi_edges_uses_the_row_walking_kernels(gnn, E):
    """8.4 M edges: the per-head gather, its transposed form and the per-head dot products with the most positions
    per warp.  17 M edges: hub rows are cut into more than 64 pieces and finished by the block-per-row fix-up, here with the per-head multipliers and the rank-1 row epilogue of the backward pass."""
    n, H, C = 200_000, 4, 8
    src, dst = synth.rmat(18, n, E, 4321, symmetric=False)
    Wx = synth.normal_f32((n, H * C), 4322)
    a = (6.0 / (C + 1)) ** 0.5
    a_s = synth.uniform_f32((H, C), -a, a, 4323)
    a_d = synth.uniform_f32((H, C), -a, a, 4324)
    oracle.set_threads(8)
    try:
        g, _ = run_case(gnn, n, src, dst, Wx, a_s, a_d, H, C, "f32", "gat %.1fM edges" % (E / 1e6))
        if E > 16_000_000:
            assert int(np.diff(g.rowptr.cpu().numpy()).max()) > 65 * 1024 and int(np.diff(g.rowptrT.cpu().numpy()).max()) > 65 * 1024
    finally:
        oracle.set_threads(1)


def test_attention_calls_under_capture_after_a_first_call_that_forks_nothing():
    """The first call of a process, a forward pass by chunks, needs no helper streams; the calls captured after it fork onto them."""
    import subprocess
    import sys
    code = """
import torch
from paper_2412_06354_b200 import gnn
n, e, H, C = 5000, 60000, 8, 8
dst = torch.randint(n, (e,), device="cuda", dtype=torch.int32)
dst[:9000] = 7
g = gnn.coo_to_csr(n, torch.randint(n, (e,), device="cuda", dtype=torch.int32), dst)
Wx, a1, a2, R = torch.randn(n, H * C, device="cuda"), torch.randn(H, C, device="cuda"), torch.randn(H, C, device="cuda"), torch.randn(n, H * C, device="cuda")
s, up = torch.randn(e, H, device="cuda"), torch.randn(e, H, device="cuda")
fwd = gnn.gat_fused(g, Wx, a1, a2, H)
def calls():
    alpha = gnn.edge_softmax(g, s)
    b = gnn.gat_fused_backward(g, Wx, a1, a2, fwd, R, H)
    f = gnn.gat_fused(g, Wx, a1, a2, H)
    return [alpha, gnn.edge_softmax_backward(g, alpha, up), b["dWx"], b["da_src"], b["da_dst"], f["out"], f["alpha"]]
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    got = calls()
graph.replay()
want = calls()
torch.cuda.synchronize()
assert all(torch.equal(x, y) for x, y in zip(got, want))
print("same")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stderr[-2000:]
