"""GPU parity: dense node-wise transform Y = X*W, dX = dY*W^T, dW = X^T*dY against the CPU checker's
triple loop.  bf16 shapes with K, M multiples of 16 take the tensor-core path."""
import numpy as np
import pytest

import oracle
from paper_2412_06354_b200 import synth
from util import assert_close, bits, to_dev, to_host64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gnn():
    from paper_2412_06354_b200 import gnn as g
    g.load()
    return g


def status_word(ws):
    import torch
    torch.cuda.synchronize()
    return int(ws[:4].view(torch.int32).item())


CASES = [("f32", 2000, 64, 64), ("f32", 1000, 100, 36), ("f32", 333, 128, 128), ("f32", 1000, 256, 64), ("f32", 700, 128, 48), ("f32", 5000, 16, 256), ("bf16", 2000, 64, 64),
         ("bf16", 1000, 128, 128), ("bf16", 777, 256, 256), ("bf16", 129, 16, 32), ("bf16", 5, 256, 16),
         ("bf16", 300, 48, 112), ("bf16", 257, 40, 24),
         # one row; exactly one tile with K and M off the 64-element boxes; several tiles and slots per CTA
         ("bf16", 1, 64, 64), ("bf16", 128, 208, 240), ("bf16", 40000, 128, 64), ("bf16", 20001, 256, 144),
         # fp32 dW on the pipelined kernel (K and M multiples of 32 up to 128): one row, a ragged last slot of 32 rows, many slots per CTA
         ("f32", 1, 128, 32), ("f32", 31, 128, 96), ("f32", 33, 128, 64), ("f32", 30017, 128, 128),
         # ... and with fewer than the 128 feature rows of the MMA
         ("f32", 500, 32, 128), ("f32", 77, 96, 32), ("f32", 6001, 64, 96),
         # ... and up to 256 wide: 16-row slots, two accumulator halves, feature rows past K zero in the second half
         ("f32", 2049, 256, 256), ("f32", 900, 160, 224), ("f32", 300, 128, 256),
         # bf16 dW with K off the 128-row blocks of the MMA (boxes past column K arrive as zeros)
         ("bf16", 5000, 192, 192), ("bf16", 1234, 96, 80), ("bf16", 777, 224, 256), ("bf16", 40, 32, 16),
         # fp32 beyond 256: long contraction (16 slices per tile), many column blocks, four accumulator blocks in dW
         ("f32", 3000, 512, 64), ("f32", 3000, 64, 512), ("f32", 700, 384, 128), ("f32", 900, 512, 512),
         # bf16 dW with up to 512 features (four accumulator blocks)
         ("bf16", 3000, 512, 64), ("bf16", 2000, 384, 128), ("bf16", 1000, 320, 48),
         # bf16 forward / dX beyond 256: weight blocks of two boxes, several column blocks
         ("bf16", 3000, 64, 512), ("bf16", 900, 512, 512), ("bf16", 500, 288, 1024)]


@pytest.mark.parametrize("dtype,n,K,M", CASES)
def test_linear_forward_backward(gnn, dtype, n, K, M):
    oracle.set_threads(8)
    try:
        X = synth.normal((n, K), dtype, 1000 + K)
        a = (6.0 / (K + M)) ** 0.5
        W32 = synth.uniform_f32((K, M), -a, a, 1001 + M)
        W = W32
        if dtype == "bf16":
            import torch
            W = torch.from_numpy(W32).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
        dY = synth.normal((n, M), dtype, 1002 + M, 1)
        Y, ws = gnn.linear(to_dev(X), to_dev(W), return_ws=True)
        assert status_word(ws) == 0
        Yo, S = oracle.matmul(X, W)
        assert_close(to_host64(Y), Yo, S, dtype, f"Y {dtype} {n}x{K}x{M}")
        dX, dW, ws = gnn.linear_backward(to_dev(X), to_dev(W), to_dev(dY), return_ws=True)
        assert status_word(ws) == 0
        dXo, S = oracle.matmul(dY, W, tb=True)
        assert_close(to_host64(dX), dXo, S, dtype, "dX")
        dWo, S = oracle.matmul(X, dY, ta=True)
        assert_close(to_host64(dW), dWo, S, dtype, "dW")
        Y2 = gnn.linear(to_dev(X), to_dev(W))
        assert np.array_equal(bits(Y), bits(Y2)), "not bit-reproducible"
    finally:
        oracle.set_threads(1)


# Sizes that divide nothing: rows that start off 16 bytes (padded copies of X, dY and W, directly written Y and dX), rows on 16
# bytes but off the 16- and 32-element steps of the MMA, one column, one row, the 512-wide contraction, column blocks of dW
RAGGED = [("f32", 700, 100, 47), ("f32", 1, 33, 2), ("f32", 129, 511, 255), ("f32", 300, 20, 36), ("f32", 4097, 37, 130), ("f32", 260, 500, 250),
          ("bf16", 700, 100, 47), ("bf16", 1, 17, 3), ("bf16", 129, 511, 255), ("bf16", 300, 24, 40), ("bf16", 4097, 37, 130), ("bf16", 515, 272, 8),
          ("bf16", 64, 1, 1), ("f32", 64, 1, 1)]


@pytest.mark.parametrize("dtype,n,K,M", RAGGED)
def test_linear_ragged_sizes(gnn, dtype, n, K, M):
    import torch
    oracle.set_threads(8)
    try:
        X, dY = synth.normal((n, K), dtype, 1300 + K), synth.normal((n, M), dtype, 1301 + M)
        W = synth.normal((K, M), dtype, 1302)
        b = synth.uniform_f32((M,), -1.0, 1.0, 1303)
        Xd, Wd, dYd = to_dev(X), to_dev(W), to_dev(dY)
        Yo, S = oracle.matmul(X, W)
        Y, ws = gnn.linear(Xd, Wd, return_ws=True)
        assert status_word(ws) == 0
        assert_close(to_host64(Y), Yo, S, dtype, "Y")
        # bias and relu in the epilogue: |b| joins the terms, relu is 1-Lipschitz
        Z = gnn.linear_bias_act(Xd, Wd, to_dev(b), relu=True)
        assert_close(to_host64(Z), np.maximum(Yo + b, 0.0), S + np.abs(b), dtype, "relu(Y + b)")
        # the bytes of the status word alone are enough workspace for the forward call, whatever the shape
        small = gnn.linear(Xd, Wd, ws=torch.empty(256, dtype=torch.uint8, device="cuda"))
        assert_close(to_host64(small), Yo, S, dtype, "Y with 256 bytes of workspace")
        dX, dW, ws = gnn.linear_backward(Xd, Wd, dYd, return_ws=True)
        assert status_word(ws) == 0
        dXo, S = oracle.matmul(dY, W, tb=True)
        assert_close(to_host64(dX), dXo, S, dtype, "dX")
        dWo, S = oracle.matmul(X, dY, ta=True)
        assert_close(to_host64(dW), dWo, S, dtype, "dW")
    finally:
        oracle.set_threads(1)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K,M", [(100, 47), (104, 40), (48, 16), (96, 20), (128, 128), (36, 128)])
def test_linear_backward_workspace_of_a_wider_layer(gnn, dtype, K, M):
    """A workspace sized for 128 x 128 serves every layer up to that, with rows to be padded or partials to be rounded up or not."""
    import torch
    n = 3000
    lib = gnn.load()
    wide = lib.gnn_linear_workspace(n, 128, 128)
    X, W, dY = synth.normal((n, K), dtype, 1500 + K), synth.normal((K, M), dtype, 1501), synth.normal((n, M), dtype, 1502 + M)
    dXo, Sx = oracle.matmul(dY, W, tb=True)
    dWo, Sw = oracle.matmul(X, dY, ta=True)
    least = 512 + 4 * K * M * 148
    for size in (wide, least):
        room = torch.full((max(size, 256) + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        ws = room[:size]
        dX, dW = gnn.linear_backward(to_dev(X), to_dev(W), to_dev(dY), ws=ws)
        assert status_word(ws) == 0 and bool((room[size:] == 0xA5).all())
        assert_close(to_host64(dX), dXo, Sx, dtype, "dX")
        assert_close(to_host64(dW), dWo, Sw, dtype, "dW")
    with pytest.raises(gnn.GnnError) as e:
        gnn.linear_backward(to_dev(X), to_dev(W), to_dev(dY), ws=room[:4 * K * M * 148])
    assert e.value.status == 4


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K,M", [(100, 48), (20, 40), (47, 33), (64, 64), (64, 24)])
def test_linear_matrices_off_16_bytes(gnn, dtype, K, M):
    """Sizes that are no multiples of 16 take matrices that begin at any element, multiples of 16 refuse them."""
    import torch
    n, s = 700, 4 if dtype == "f32" else 2
    lib, st = gnn.load(), torch.cuda.current_stream().cuda_stream
    X, W, dY = synth.normal((n, K), dtype, 1600 + K), synth.normal((K, M), dtype, 1601), synth.normal((n, M), dtype, 1602 + M)
    want = [oracle.matmul(X, W), oracle.matmul(dY, W, tb=True), oracle.matmul(X, dY, ta=True)]

    def at(a, off):  # the matrix, one element past a 16-byte boundary if off
        room = torch.zeros(a.numel() + 8, dtype=a.dtype, device="cuda")
        v = room[off:off + a.numel()].view(a.shape)
        v.copy_(a)
        return v

    ws = torch.empty(lib.gnn_linear_workspace(n, K, M), dtype=torch.uint8, device="cuda")
    d = [to_dev(a) for a in (X, W, dY)]
    outs = [torch.zeros(sh, dtype=d[0].dtype, device="cuda") for sh in ((n, M), (n, K), (K, M))]
    code = {"f32": gnn.F32, "bf16": gnn.BF16}[dtype]
    for odd in range(5):  # X, W, dY, Y, dX
        x, w, dy, y, dx = (at(a, k == odd) for k, a in enumerate((*d, outs[0], outs[1])))
        dw = outs[2]
        rc = [lib.gnn_linear(x.data_ptr(), w.data_ptr(), n, K, M, code, y.data_ptr(), ws.data_ptr(), ws.numel(), st),
              lib.gnn_linear_backward(None, w.data_ptr(), dy.data_ptr(), n, K, M, code, dx.data_ptr(), None, ws.data_ptr(), ws.numel(), st),
              lib.gnn_linear_backward(x.data_ptr(), None, dy.data_ptr(), n, K, M, code, None, dw.data_ptr(), ws.data_ptr(), ws.numel(), st)]
        touches = [odd in (0, 1, 3), odd in (1, 2, 4), odd in (0, 2)]
        for k, (got, what) in enumerate(((y, "Y"), (dx, "dX"), (dw, "dW"))):
            if (K, M) == (64, 64) and touches[k]:
                assert rc[k] == 1, (odd, what)
            else:
                assert rc[k] == 0, (odd, what)
                assert_close(to_host64(got), *want[k], dtype, f"{what}, matrix {odd} off 16 bytes")


# fp32 sums of sizes that divide nothing: no further from 64 bits than plain fp32 FMAs.  The tensor core truncates its accumulator at
# every MMA of 16 terms, half a unit in the last place (2^-23 of the running sum) on average and one way; at most 10 main MMAs of
# a forward sum follow one another (16 in each of two sums above that), 32 in dW, and the sums are then added with rounding:
# norm-wise n * 2^-24 + 2^-23 for n in a row.  One sum for all products of all levels was 7.3e-7 / 3.4e-6 for contractions of 100
# / 511 and 7.8e-6 / 2.3e-5 for dW over 170k / 500k rows.
@pytest.mark.parametrize("n,K,M", [(170_000, 100, 47), (500_000, 33, 9), (20_000, 511, 255), (30_000, 161, 40), (9_000, 47, 100), (2_000, 300, 1)])
def test_linear_ragged_fp32_is_as_exact_as_plain_fp32(gnn, n, K, M):
    oracle.set_threads(8)
    try:
        X, W, dY = synth.normal((n, K), "f32", 1400 + K), synth.normal((K, M), "f32", 1401), synth.normal((n, M), "f32", 1402 + M)
        Xd, Wd, dYd = to_dev(X), to_dev(W), to_dev(dY)

        def check(got, ref, in_a_row, what):
            err = np.linalg.norm(to_host64(got) - ref) / np.linalg.norm(ref)
            assert err <= in_a_row * 2.0**-24 + 2.0**-23, f"{what}: {err:.2e}"

        def steps(k):
            s = -(-k // 16)
            return s if s <= 10 else -(-s // 2)

        check(gnn.linear(Xd, Wd), oracle.matmul(X, W)[0], steps(K), "Y")
        dX, dW = gnn.linear_backward(Xd, Wd, dYd)
        check(dX, oracle.matmul(dY, W, tb=True)[0], steps(M), "dX")
        check(dW, oracle.matmul(X, dY, ta=True)[0], min(32, -(-n // (148 * 16)) + 1), "dW")
    finally:
        oracle.set_threads(1)


# dW of fp32 has X's levels in tensor memory up to 128 x 128, for some wider products too, in shared memory for the others: both sides of each line
@pytest.mark.parametrize("K,M", [(128, 128), (129, 128), (128, 129), (160, 128), (160, 96), (160, 160), (160, 192), (256, 160), (256, 128), (256, 127), (96, 256), (64, 256), (128, 224)])
def test_linear_dw_operand_places(gnn, K, M):
    import torch
    n = 9_700
    X, W, D = (torch.randn(s, device="cuda") for s in ((n, K), (K, M), (n, M)))
    dW = gnn.linear_backward(X, W, D, want_dX=False)[1]
    want, terms = X.double().T @ D.double(), X.double().abs().T @ D.double().abs()
    assert bool(((dW.double() - want).abs() <= 1e-5 * terms).all())
    assert float((dW.double() - want).norm() / want.norm()) < 4e-6  # as plain fp32 sums of 9700 terms
    assert torch.equal(dW, gnn.linear_backward(X, W, D, want_dX=False)[1])


def test_linear_large_rows_tensor_core(gnn):
    """N = 100000 rows, 256 -> 256 bf16 (the attention workload's transform): many tiles per CTA."""
    import torch
    n, K, M = 100_000, 256, 256
    X = synth.normal_bf16((n, K), 1100)
    W = torch.from_numpy(synth.glorot_f32(K, M, 1101)).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    Y, ws = gnn.linear(to_dev(X), to_dev(W), return_ws=True)
    assert status_word(ws) == 0
    rows = np.random.default_rng(3).choice(n, 3000, replace=False)
    rows = np.union1d(rows, [0, 127, 128, n - 1])
    Yo, S = oracle.matmul(X[rows], W)
    assert_close(to_host64(Y)[rows], Yo, S, "bf16", "sampled rows of Y")
    # linearity in exact arithmetic: rows of zeros give zeros
    Xz = X.copy()
    Xz[::2] = 0
    Yz = gnn.linear(to_dev(Xz), to_dev(W))
    assert torch.count_nonzero(Yz[::2]) == 0 and torch.equal(Yz[1::2], Y[1::2])


def test_linear_degenerate(gnn):
    import torch
    W = torch.zeros((64, 64), device="cuda")
    Y = gnn.linear(torch.zeros((0, 64), device="cuda"), W)
    assert Y.shape == (0, 64)
    dX, dW = gnn.linear_backward(torch.zeros((0, 64), device="cuda"), W, torch.zeros((0, 64), device="cuda"))
    assert torch.count_nonzero(dW) == 0
    with pytest.raises(gnn.GnnError) as e:
        gnn.linear(torch.zeros((8, 64), device="cuda"), W, ws=torch.empty(8, dtype=torch.uint8, device="cuda"))
    assert e.value.status == 4


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_linear_back_to_back_launches_are_bitwise_identical(gnn, dtype):
    """Forty launches in a row with nothing in between (the pipelines' barrier phases and ring slots are
    reused at full speed): every result must equal the first one bit for bit, and no wait may expire."""
    import torch
    n, K, M = 170_000, 128, 128
    X = to_dev(synth.normal((n, K), dtype, 1200))
    W32 = synth.glorot_f32(K, M, 1201)
    W = to_dev(W32) if dtype == "f32" else torch.from_numpy(W32).to(torch.bfloat16).cuda()
    dY = to_dev(synth.normal((n, M), dtype, 1202))
    ws = torch.empty(gnn.load().gnn_linear_workspace(n, K, M), dtype=torch.uint8, device="cuda")
    Y0 = gnn.linear(X, W, ws=ws).clone()
    dX0, dW0 = (t.clone() for t in gnn.linear_backward(X, W, dY, ws=ws))
    for _ in range(40):
        Y = gnn.linear(X, W, ws=ws)
        dX, dW = gnn.linear_backward(X, W, dY, ws=ws)
    torch.cuda.synchronize()
    assert status_word(ws) == 0
    assert torch.equal(Y.view(torch.int16 if dtype == "bf16" else torch.int32), Y0.view(torch.int16 if dtype == "bf16" else torch.int32))
    assert torch.equal(dX.float(), dX0.float()) and torch.equal(dW.float(), dW0.float())


# Blocks of output columns side by side (width a multiple of 16 that is not one of 32, a last block that is narrower), blocks of
# 32 columns for few rows, four and two converter groups, dW in slots of 16 and 32 rows with four and two groups
@pytest.mark.parametrize("dtype,n,K,M", [("f32", 9700, 256, 256), ("f32", 19100, 64, 224), ("f32", 9601, 480, 140), ("f32", 2000, 128, 128),
                                         ("f32", 5000, 160, 160), ("f32", 257, 128, 192), ("f32", 700, 512, 128), ("bf16", 515, 64, 64)])
def test_linear_column_blocks(gnn, dtype, n, K, M):
    test_linear_ragged_sizes(gnn, dtype, n, K, M)
