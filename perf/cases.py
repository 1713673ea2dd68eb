"""The work that users of this library have it do, as cases that can be timed.

A case is one training step (forward and backward) or one inference pass of a layer, one graph set-up, or one run of the
unfused primitives, made of calls of ``paper_2412_06354_b200.gnn`` as a program makes them: outputs and workspaces are left
to the binding, nothing is synchronised.  What a program keeps between steps (the sparse forms of a graph, its
normalisation coefficients, weights) is made by ``prepare``.

Every kind has a range of sizes; ``listed`` names fixed points of it and ``draw`` gives others.
"""
import math

import torch

from paper_2412_06354_b200 import gnn, synth

SLOPE = 0.2  # of LeakyReLU in the attention layers


def listed():
    return [
        # A mini-batch of 32 graphs of 10..40 nodes through a GIN layer (a two-layer perceptron) and sum pooling, the
        # batch size of the usual graph-classification training loop: some 800 nodes, so latency and launches are all of it.
        dict(name="gin, batch of 32 graphs", kind="gin", graphs=32, F=64, hidden=64, dtype="f32", pool="sum", train=True),
        # One GCN layer with bias and relu on a graph of the size of the classic citation sets; every epoch is this step.
        dict(name="gcn, 2000 nodes", kind="gcn", nodes=2000, degree=5, F=64, out=64, dtype="f32", train=True),
        # GraphConv with mean aggregation and mean pooling on a large mini-batch of small graphs.
        dict(name="graphconv, 512 graphs", kind="graphconv", graphs=512, F=128, dtype="f32", pool="mean", train=True),
        # SAGE with mean aggregation on a power-law graph of citation scale, in mixed precision.
        dict(name="sage mean, 170k bf16", kind="sage", nodes=170_000, m=4, F=128, out=128, dtype="bf16", op="mean", train=True),
        # The same graph with max aggregation (winners saved for the backward pass), in single precision.
        dict(name="sage max, 170k f32", kind="sage", nodes=170_000, m=4, F=128, out=128, dtype="f32", op="max", train=True),
        # A GAT layer of 8 heads x 32 features on a skewed graph: transform, attention, weighted sum, and back.
        dict(name="gat, 100k bf16", kind="gat", nodes=100_000, edges=1_600_000, heads=8, channels=32, dtype="bf16", train=True),
        # The GATv2 kind of attention, whose calls are separate (logits, edge softmax, weighted sum), in single precision.
        dict(name="gatv2, 100k f32", kind="gatv2", nodes=100_000, edges=1_600_000, heads=4, channels=32, dtype="f32", train=True),
        # A weighted sum over a graph of co-purchase scale with narrow rows, the edge weights being learnt.
        dict(name="weighted sum, 123M x 64", kind="sum", nodes=2_400_000, edges=123_000_000, F=64, dtype="bf16", op="sum",
             weighted=True, dW=True),
        # The same scale with the widest rows: the largest case.
        dict(name="sum, 123M x 512", kind="sum", nodes=2_400_000, edges=123_000_000, F=512, dtype="f32", op="sum",
             weighted=False, dW=False),
        # Set-up of a new graph (self-loops, both sparse forms, degrees, GCN coefficients): every sampled or newly loaded graph.
        dict(name="set-up, 1.36M edges", kind="setup", nodes=170_000, edges=1_360_000, relations=1, weighted=True),
        # A message that is not one of the fused pairs: edge-wise messages and their reduction as calls of their own.
        dict(name="messages, 1.36M bf16", kind="messages", nodes=170_000, m=4, F=128, dtype="bf16", op="max"),
        # The dense transform of a classifier: input features and classes that are no multiple of anything.
        dict(name="dense, 170k x 100 x 47", kind="dense", rows=170_000, K=100, M=47, dtype="f32", act=False, train=True),
    ]


# ---------------------------------------------------------------------------------------------------- drawn cases
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, dtype, lo, hi):
    """A feature width: a usual one, or any that fills whole 16-byte chunks."""
    step = 8 if dtype == "bf16" else 4
    usual = [w for w in (16, 32, 64, 96, 128, 192, 256, 384, 512) if lo <= w <= hi]
    return rng.choice(usual) if rng.random() < 0.6 else step * rng.randint(-(-lo // step), hi // step)


def draw(rng):
    kind = rng.choice(["gin", "gcn", "graphconv", "sage", "sage", "gat", "gatv2", "sum", "sum", "setup", "messages", "dense"])
    dtype = rng.choice(["f32", "bf16"])
    train = rng.random() < 0.75
    if kind in ("gin", "graphconv"):
        # Max pooling in inference only: which of two nodes that round to nearly the same value takes the gradient is chance.
        pool = rng.choice(["sum", "mean"] if train else ["sum", "mean", "max"])
    if kind == "gin":
        return dict(kind=kind, graphs=_log(rng, 8, 2048), F=_width(rng, dtype, 16, 128), hidden=_width(rng, dtype, 16, 128),
                    dtype=dtype, pool=pool, train=train)
    if kind == "gcn":
        return dict(kind=kind, nodes=_log(rng, 500, 200_000), degree=rng.randint(2, 16), F=_width(rng, dtype, 16, 256),
                    out=_width(rng, dtype, 8, 256), dtype=dtype, train=train)
    if kind == "graphconv":
        return dict(kind=kind, graphs=_log(rng, 8, 4096), F=_width(rng, dtype, 16, 256), dtype=dtype, pool=pool, train=train)
    if kind == "sage":
        return dict(kind=kind, nodes=_log(rng, 5_000, 400_000), m=rng.randint(2, 8), F=_width(rng, dtype, 16, 256),
                    out=_width(rng, dtype, 16, 256), dtype=dtype, op=rng.choice(["mean", "max"]), train=train)
    if kind in ("gat", "gatv2"):
        nodes = _log(rng, 2_000, 200_000)
        heads = rng.choice([1, 2, 4, 8])
        channels = rng.choice([8, 16, 32, 64])
        while heads * channels * (2 if dtype == "bf16" else 4) > 512:
            channels //= 2
        return dict(kind=kind, nodes=nodes, edges=nodes * rng.randint(4, 32) + rng.randint(0, 999), heads=heads, channels=channels,
                    dtype=dtype, train=train)
    if kind == "sum":
        edges = _log(rng, 1_000_000, 123_000_000)
        F = _width(rng, dtype, 32, 512)
        dW = rng.random() < 0.4 and edges * F * (2 if dtype == "bf16" else 4) <= 1e11
        return dict(kind=kind, nodes=int(edges / math.exp(rng.uniform(math.log(4), math.log(64)))), edges=edges, F=F, dtype=dtype,
                    op=rng.choice(["sum", "mean"]), weighted=dW or rng.random() < 0.5, dW=dW)
    if kind == "setup":
        edges = _log(rng, 2_000, 30_000_000)
        return dict(kind=kind, nodes=max(16, int(edges / rng.uniform(2, 40))), edges=edges, relations=rng.choice([1, 1, 3, 5]),
                    weighted=rng.random() < 0.5)
    if kind == "messages":
        return dict(kind=kind, nodes=_log(rng, 5_000, 300_000), m=rng.randint(2, 6), F=_width(rng, dtype, 16, 256), dtype=dtype,
                    op=rng.choice(["sum", "mean", "max", "min"]))
    rows = _log(rng, 1_000, 500_000)
    if rng.random() < 0.5:
        K, M = rng.choice([32, 64, 128, 256]), rng.choice([16, 32, 64, 128, 256])
    else:
        K, M = rng.randint(16, 512), rng.randint(2, 256)
    act = M % 8 == 0 and rng.random() < 0.7  # the backward call of bias and relu takes rows of whole 16-byte chunks
    return dict(kind="dense", rows=rows, K=K, M=M, dtype=dtype, act=act, train=train)


# ---------------------------------------------------------------------------------------------------- inputs
class _Inputs:
    """Random tensors and graphs on the GPU, from one seed."""

    def __init__(self, seed, dtype="f32"):
        self.seed = seed
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        self.dtype = torch.bfloat16 if dtype == "bf16" else torch.float32

    def normal(self, *shape):
        """Features or gradients, N(0,1)."""
        return torch.randn(shape, device="cuda", generator=self.gen).to(self.dtype)

    def weight(self, k, m):
        """A weight matrix, Glorot uniform."""
        a = math.sqrt(6.0 / (k + m))
        return ((torch.rand((k, m), device="cuda", generator=self.gen) * 2 - 1) * a).to(self.dtype)

    def uniform(self, *shape, lo=0.0, hi=1.0):
        return torch.rand(shape, device="cuda", generator=self.gen) * (hi - lo) + lo

    def ids(self, count, n):
        return torch.randint(n, (count,), device="cuda", dtype=torch.int32, generator=self.gen)

    def random_graph(self, n, edges):
        """Uniform random pairs without loops, both directions."""
        a = self.ids(edges // 2, n)
        b = (a + 1 + self.ids(edges // 2, n - 1)) % n
        return torch.cat([a, b]), torch.cat([b, a])

    def batch(self, graphs):
        """Block-diagonal batch of graphs of 10..40 nodes, as many of each size, every pair linked with probability 0.2, and its graph_ptr."""
        size = 10 + torch.randperm(graphs, device="cuda", generator=self.gen) % 31
        ptr = torch.zeros(graphs + 1, dtype=torch.int64, device="cuda")
        ptr[1:] = torch.cumsum(size, 0)
        k = torch.arange(40, device="cuda")
        link = torch.rand((graphs, 40, 40), device="cuda", generator=self.gen) < 0.2
        link &= (k[:, None] < k[None, :]) & (k[None, None, :] < size[:, None, None])
        which, i, j = link.nonzero(as_tuple=True)
        i, j = ((ptr[which] + v).to(torch.int32) for v in (i, j))
        return torch.cat([i, j]), torch.cat([j, i]), ptr

    def power_law(self, n, m):
        """Preferential attachment, m links per new node, both directions, nodes in random order."""
        src, dst = synth.barabasi_albert(n, m, self.seed)
        return torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()

    def rmat(self, n, edges, symmetric):
        """R-MAT (0.57, 0.19, 0.19) without loops, nodes in random order."""
        want = edges // 2 if symmetric else edges
        order = torch.randperm(n, device="cuda", dtype=torch.int32, generator=self.gen)
        got, have = [], 0
        while have < want:
            count = int((want - have) * 1.3) + 1024
            src = torch.zeros(count, dtype=torch.int32, device="cuda")
            dst = torch.zeros(count, dtype=torch.int32, device="cuda")
            for _ in range(max(1, (n - 1).bit_length())):
                r = torch.rand(count, device="cuda", generator=self.gen)
                src = src * 2 + (r >= 0.76)
                dst = dst * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
            keep = (src < n) & (dst < n) & (src != dst)
            got.append(torch.stack([order[src[keep]], order[dst[keep]]]))
            have += got[-1].shape[1]
        src, dst = torch.cat(got, 1)[:, :want].contiguous()
        return (torch.cat([src, dst]), torch.cat([dst, src])) if symmetric else (src, dst)


def prepare(case, seed):
    kind = case["kind"]
    r = _Inputs(seed, case.get("dtype", "f32"))
    s = dict(case)
    if kind in ("gin", "graphconv"):
        src, dst, ptr = r.batch(case["graphs"])
        n = int(ptr[-1])
        F, out = case["F"], case.get("hidden", case["F"])
        s.update(g=gnn.coo_to_csr(n, src, dst), ptr=ptr, X=r.normal(n, F), W1=r.weight(F, out), W2=r.weight(out if kind == "gin" else F, out),
                 b1=r.uniform(out, lo=-0.1, hi=0.1), b2=r.uniform(out, lo=-0.1, hi=0.1), eps=0.1, dP=r.normal(case["graphs"], out))
    elif kind == "gcn":
        n, F, out = case["nodes"], case["F"], case["out"]
        src, dst = gnn.add_self_loops(n, *r.random_graph(n, n * case["degree"]))
        g = gnn.coo_to_csr(n, src, dst)
        _, coef, coefT = gnn.gcn_norm(g)
        s.update(g=g, coef=coef, coefT=coefT, X=r.normal(n, F), W=r.weight(F, out), b=r.uniform(out, lo=-0.1, hi=0.1), dY=r.normal(n, out))
    elif kind == "sage":
        n, F, out = case["nodes"], case["F"], case["out"]
        s.update(g=gnn.coo_to_csr(n, *r.power_law(n, case["m"])), X=r.normal(n, F), Ws=r.weight(F, out), Wn=r.weight(F, out),
                 dY=r.normal(n, out))
    elif kind in ("gat", "gatv2"):
        n, H, C = case["nodes"], case["heads"], case["channels"]
        F, a = H * C, math.sqrt(6.0 / (C + 1))
        s.update(g=gnn.coo_to_csr(n, *r.rmat(n, case["edges"], False)), X=r.normal(n, F), W=r.weight(F, F), W2=r.weight(F, F),
                 a1=r.uniform(H, C, lo=-a, hi=a), a2=r.uniform(H, C, lo=-a, hi=a), dY=r.normal(n, F))
    elif kind == "sum":
        n, F = case["nodes"], case["F"]
        g = gnn.coo_to_csr(n, *r.rmat(n, case["edges"], True))
        w = r.uniform(g.E) if case["weighted"] else None
        s.update(g=g, w=w, wT=None if w is None else gnn.permute_edge_data(g.t2f, w), X=r.normal(n, F), dY=r.normal(n, F))
    elif kind == "setup":
        n, rel = case["nodes"], case["relations"]
        per = [r.rmat(max(4, n // rel), case["edges"] // rel, True) for _ in range(rel)]
        s.update(coo=per, w=r.uniform(sum(p[0].numel() for p in per) + n) if case["weighted"] else None,
                 is_mean=torch.arange(rel, dtype=torch.int32, device="cuda") % 2)
    elif kind == "messages":
        n, F = case["nodes"], case["F"]
        src, dst = r.power_law(n, case["m"])
        order = torch.argsort(dst, stable=True)  # edges kept by target, so that edge data need no reordering
        src, dst = src[order], dst[order]
        s.update(g=gnn.coo_to_csr(n, src, dst), src=src, dst=dst, X=r.normal(n, F), dY=r.normal(n, F))
    else:
        n, K, M = case["rows"], case["K"], case["M"]
        s.update(X=r.normal(n, K), W=r.weight(K, M), b=r.uniform(M, lo=-0.1, hi=0.1), dY=r.normal(n, M))
    return s


# ---------------------------------------------------------------------------------------------------- one pass
def run(s):
    return _RUN[s["kind"]](s)


def _gin(s):
    g, X, W1, W2, pool = s["g"], s["X"], s["W1"], s["W2"], s["pool"]
    A = gnn.gin(g, X, s["eps"])
    H = gnn.linear_bias_act(A, W1, s["b1"], relu=True)
    Z = gnn.linear_bias_act(H, W2, s["b2"])
    P, arg = _pooled(s, Z, pool)
    if not s["train"]:
        return P
    dZ = gnn.reduce_nodes_backward(s["ptr"], s["dP"], X.shape[0], pool, argmax=arg)
    dZ, db2 = gnn.row_epilogue_backward(Z, dZ, relu=False)
    dH, dW2 = gnn.linear_backward(H, W2, dZ)
    dH, db1 = gnn.row_epilogue_backward(H, dH, relu=True)
    dA, dW1 = gnn.linear_backward(A, W1, dH)
    dX, _ = gnn.gin_backward(g, dA, s["eps"])
    return P, dX, dW1, dW2, db1, db2


def _pooled(s, Z, pool):
    P = gnn.reduce_nodes(s["ptr"], Z, pool)
    return P if pool in ("max", "min") else (P, None)


def _gcn(s):
    g, X, W = s["g"], s["X"], s["W"]
    H = gnn.linear(X, W)
    Y = gnn.propagate_msg(g, gnn.E_MUL_XJ, H, e_csr=s["coef"], epi=dict(bias=s["b"], relu=True))
    if not s["train"]:
        return Y
    dZ, db = gnn.row_epilogue_backward(Y, s["dY"], relu=True)
    dH, _ = gnn.propagate_fused_backward(g, dZ, "sum", w_csrT=s["coefT"])
    dX, dW = gnn.linear_backward(X, W, dH)
    return Y, dX, dW, db


def _graphconv(s):
    g, X, W1, W2, pool = s["g"], s["X"], s["W1"], s["W2"], s["pool"]
    A = gnn.propagate_fused(g, X, None, "mean")
    H = gnn.axpby(1.0, gnn.linear(X, W1), 1.0, gnn.linear(A, W2))
    P, arg = _pooled(s, H, pool)
    if not s["train"]:
        return P
    dH = gnn.reduce_nodes_backward(s["ptr"], s["dP"], X.shape[0], pool, argmax=arg)
    dX1, dW1 = gnn.linear_backward(X, W1, dH)
    dA, dW2 = gnn.linear_backward(A, W2, dH)
    dX2, _ = gnn.propagate_fused_backward(g, dA, "mean")
    return P, gnn.axpby(1.0, dX1, 1.0, dX2), dW1, dW2


def _sage(s):
    g, X, Ws, Wn, op = s["g"], s["X"], s["Ws"], s["Wn"], s["op"]
    A, arg = gnn.propagate_fused(g, X, None, op) if op == "max" else (gnn.propagate_fused(g, X, None, op), None)
    Y = gnn.axpby(1.0, gnn.linear(X, Ws), 1.0, gnn.linear(A, Wn))
    if not s["train"]:
        return Y
    dX1, dWs = gnn.linear_backward(X, Ws, s["dY"])
    dA, dWn = gnn.linear_backward(A, Wn, s["dY"])
    dX2, _ = gnn.propagate_fused_backward(g, dA, op, argmax=arg)
    return Y, gnn.axpby(1.0, dX1, 1.0, dX2), dWs, dWn


def _gat(s):
    g, X, W, a1, a2, H = s["g"], s["X"], s["W"], s["a1"], s["a2"], s["heads"]
    Wx = gnn.linear(X, W)
    f = gnn.gat_fused(g, Wx, a1, a2, H, SLOPE)
    if not s["train"]:
        return f["out"]
    b = gnn.gat_fused_backward(g, Wx, a1, a2, f, s["dY"], H, SLOPE)
    dX, dW = gnn.linear_backward(X, W, b["dWx"])
    return f["out"], f["alpha"], dX, dW, b["da_src"], b["da_dst"]


def _gatv2(s):
    g, X, W, W2, a, H = s["g"], s["X"], s["W"], s["W2"], s["a1"], s["heads"]
    Xl, Xr = gnn.linear(X, W), gnn.linear(X, W2)
    alpha = gnn.edge_softmax(g, gnn.gatv2_logits(g, Xl, Xr, a, H, SLOPE))
    Y = gnn.propagate_msg(g, gnn.E_MUL_XJ, Xl, e_csr=alpha)
    if not s["train"]:
        return Y
    alphaT = gnn.permute_edge_data(g.t2f, alpha)
    b = gnn.propagate_msg_backward(g, gnn.E_MUL_XJ, s["dY"], Xj=Xl, e_csrT=alphaT, want_de=True)
    ds = gnn.edge_softmax_backward(g, alpha, b["de"])
    dXl, dXr, da = gnn.gatv2_logits_backward(g, Xl, Xr, a, ds, H, SLOPE)
    dX1, dW = gnn.linear_backward(X, W, gnn.axpby(1.0, b["dXj"], 1.0, dXl))
    dX2, dW2 = gnn.linear_backward(X, W2, dXr)
    return Y, alpha, gnn.axpby(1.0, dX1, 1.0, dX2), dW, dW2, da


def _sum(s):
    g, X = s["g"], s["X"]
    Y = gnn.propagate_fused(g, X, s["w"], s["op"])
    dX, dw = gnn.propagate_fused_backward(g, s["dY"], s["op"], X=X, w_csrT=s["wT"], want_dW=s["dW"])
    return Y, dX, dw


def _setup(s):
    if s["relations"] == 1:
        n = s["nodes"]
        src, dst = gnn.add_self_loops(n, *s["coo"][0])
        g = gnn.coo_to_csr(n, src, dst)
        w = None if s["w"] is None else gnn.permute_edge_data(g.eid, s["w"])
        more = gnn.gcn_norm(g, w)
    else:
        rel, per = s["relations"], max(4, s["nodes"] // s["relations"])
        src, dst, seg = gnn.merge_edge_lists([(a, b, k * per, 0) for k, (a, b) in enumerate(s["coo"])])
        g = gnn.coo_to_csr(rel * per, src, dst)
        w = None if s["w"] is None else gnn.permute_edge_data(g.eid, s["w"][: g.E])
        more = gnn.segment_coef(g, gnn.permute_edge_data(g.eid, seg), s["is_mean"], w)
    return g.rowptr, g.col, g.eid, g.rowptrT, g.colT, g.eidT, g.t2f, more


def _messages(s):
    g, X, src, dst, op = s["g"], s["X"], s["src"], s["dst"], s["op"]
    m = gnn.axpby(1.0, gnn.gather(dst, X), -1.0, gnn.gather(src, X))
    out, arg = gnn.aggregate(g, m, op) if op in ("max", "min") else (gnn.aggregate(g, m, op), None)
    dm = gnn.aggregate_backward(g, s["dY"], op, argmax=arg)
    return out, gnn.axpby(1.0, gnn.gather_backward(g, dm), -1.0, gnn.gather_backward(g, dm, by_src=True))


def _dense(s):
    X, W, dY = s["X"], s["W"], s["dY"]
    Y = gnn.linear_bias_act(X, W, s["b"], relu=True) if s["act"] else gnn.linear(X, W)
    if not s["train"]:
        return Y
    if not s["act"]:
        return (Y, *gnn.linear_backward(X, W, dY))
    dZ, db = gnn.row_epilogue_backward(Y, dY, relu=True)
    return (Y, *gnn.linear_backward(X, W, dZ), db)


_RUN = dict(gin=_gin, gcn=_gcn, graphconv=_graphconv, sage=_sage, gat=_gat, gatv2=_gatv2, sum=_sum, setup=_setup, messages=_messages, dense=_dense)


# ---------------------------------------------------------------------------------------------------- what a pass needs
def work(case):
    """Inputs read once and outputs written once; nothing for what lies between two calls of a pass."""
    kind, train = case["kind"], case.get("train", True)
    size = 2 if case.get("dtype") == "bf16" else 4
    both = 2 if train else 1  # forms of the graph read, sides of a layer

    def graph(n, e, weights=0):
        return 8 * n + (4 + 4 * weights) * e

    if kind in ("gin", "graphconv"):
        n, e, F, out = 25 * case["graphs"], 136 * case["graphs"], case["F"], case.get("hidden", case["F"])
        k = F if kind == "graphconv" else out
        values = both * (n * F + case["graphs"] * out + F * out + k * out)
        return dict(bytes=size * values + both * graph(n, e), flops=(3 if train else 1) * 2 * n * (F + k) * out + both * 2 * e * F)
    if kind == "gcn":
        n, F, out = case["nodes"], case["F"], case["out"]
        e = n * (case["degree"] + 1)
        values = both * (n * F + n * out + F * out)
        return dict(bytes=size * values + both * graph(n, e, 1), flops=(3 if train else 1) * 2 * n * F * out + both * 2 * e * out)
    if kind == "sage":
        n, F, out = case["nodes"], case["F"], case["out"]
        e = 2 * n * case["m"]
        values = both * (n * F + n * out + 2 * F * out)
        return dict(bytes=size * values + both * graph(n, e), flops=(3 if train else 1) * 4 * n * F * out + both * 2 * e * F)
    if kind in ("gat", "gatv2"):
        n, e, H = case["nodes"], case["edges"], case["heads"]
        F, products = H * case["channels"], 1 if kind == "gat" else 2
        values = both * (2 * n * F + products * F * F)
        return dict(bytes=size * values + both * graph(n, e) + (4 * e * H if train else 0),
                    flops=(3 if train else 1) * (products * 2 * n * F * F + 4 * e * F))
    if kind == "sum":
        n, e, F = case["nodes"], case["edges"], case["F"]
        return dict(bytes=size * 4 * n * F + 2 * graph(n, e, int(case["weighted"])) + 4 * e * case["dW"],
                    flops=2 * e * F * (2 + case["dW"]))
    if kind == "setup":
        n, e = case["nodes"], case["edges"]
        return dict(bytes=8 * e + 16 * n + 28 * e + 4 * e * case["weighted"], flops=0)
    if kind == "messages":
        n, e, F = case["nodes"], 2 * case["nodes"] * case["m"], case["F"]
        return dict(bytes=size * 4 * n * F + 2 * graph(n, e), flops=5 * e * F)
    n, K, M = case["rows"], case["K"], case["M"]
    values = both * (n * K + n * M + K * M)
    return dict(bytes=size * values, flops=(3 if train else 1) * 2 * n * K * M)


def tolerance(case):
    if case["kind"] == "setup":
        return dict(rel=1e-5)  # degrees and coefficients; whole numbers are exact
    if case.get("dtype") == "bf16":
        return dict(rel=1e-2)  # two or three roundings of 2^-9 each, one after the other
    if case["kind"] in ("gat", "gatv2") and case["train"]:
        # An argument of LeakyReLU within rounding of zero (one in about 10^7) may take the other slope.
        return dict(rel=1e-4, max=5e-2)
    mask = {"gin": lambda c: 25 * c["graphs"] * c["hidden"], "gcn": lambda c: c["nodes"] * c["out"],
            "dense": lambda c: c["rows"] * c["M"] if c["act"] else 0}.get(case["kind"], lambda c: 0)(case)
    if mask > 10**6 and case["train"]:
        # Of this many values before a relu some lie within rounding of zero, and each takes its gradient with it.
        return dict(rel=1e-3, max=0.5)
    return dict(rel=1e-5)
