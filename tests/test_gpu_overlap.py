"""Chains of small calls whose launches overlap, through buffers that are written again and again: every result has the bits that
it has when the device is waited for between the calls."""
import numpy as np
import pytest

from util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gnn():
    from paper_2412_06354_b200 import gnn as g
    g.load()
    return g


@pytest.mark.parametrize("n,e,dtype", [(800, 6000, "f32"), (800, 6000, "bf16"), (3000, 200_000, "f32"), (20_000, 150_000, "bf16")])
def test_producers_and_consumers_over_reused_buffers(gnn, n, e, dtype):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(n)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    src, dst = (torch.randint(n, (e,), dtype=torch.int32, device="cuda", generator=gen) for _ in range(2))
    g = gnn.coo_to_csr(n, src, dst)
    F = 64
    U, V = (torch.randn((n, F), device="cuda", generator=gen).to(dt) for _ in range(2))
    W = (torch.randn((F, F), device="cuda", generator=gen) / 8).to(dt)
    a = torch.randn((8, 8), device="cuda", generator=gen)
    ptr = torch.linspace(0, n, 33, device="cuda").to(torch.int64)
    X, A, Y = (torch.empty((n, F), dtype=dt, device="cuda") for _ in range(3))
    arg = torch.empty((n, F), dtype=torch.int32, device="cuda")
    de, ws = torch.empty(g.E, device="cuda"), torch.empty(64 << 20, dtype=torch.uint8, device="cuda")

    def step(i, wait):
        """Every buffer above is overwritten; what comes back is memory of its own."""
        def call(r):
            if wait:
                torch.cuda.synchronize()
            return r
        call(gnn.axpby(1.0 + i, U, 0.5 * i - 3.0, V, out=X))
        call(gnn.propagate_fused(g, X, None, "mean", out=A, ws=ws))
        call(gnn.propagate_fused(g, A, None, "max", out=Y, argmax=arg, ws=ws))
        dX, _ = call(gnn.propagate_fused_backward(g, Y, "max", argmax=arg, ws=ws))
        call(gnn.propagate_fused_backward(g, A, "sum", X=dX, want_dX=False, want_dW=True, dW=de, ws=ws))
        s = call(gnn.gatv2_logits(g, X, A, a, 8))
        _, _, da = call(gnn.gatv2_logits_backward(g, X, Y, a, s, 8, ws=ws))
        Z = call(gnn.linear(Y, W, ws=ws))
        dZ, db = call(gnn.row_epilogue_backward(Z, A, ws=ws))
        _, dW = call(gnn.linear_backward(Y, W, dZ, ws=ws))
        P = call(gnn.reduce_nodes(ptr, Z, "mean", ws=ws))
        dP = call(gnn.reduce_nodes_backward(ptr, P, n, "mean"))
        _, eps = call(gnn.gin_backward(g, dP, 0.1, X=Z, want_deps=True, ws=ws))
        m = call(gnn.gather(dst, dP))
        out, win = call(gnn.aggregate(g, m, "min", ws=ws))
        return da, db, dW, P, eps, out, win, call(gnn.permute_edge_data(g.t2f, de))

    want = [step(i, True) for i in range(12)]
    got = [step(i % 12, False) for i in range(240)]
    torch.cuda.synchronize()
    for i, r in enumerate(got):
        for k, (x, y) in enumerate(zip(r, want[i % 12])):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), (i, k)
