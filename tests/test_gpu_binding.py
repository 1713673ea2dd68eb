"""What the compiled binding does with arguments before the library sees them: errors are Python errors."""
import numpy as np
import pytest

from util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gnn():
    from paper_2412_06354_b200 import gnn as g
    g.load()
    return g


@pytest.fixture(scope="module")
def small(gnn):
    """A graph of 6 nodes and 7 edges and features of 16 fp32 columns."""
    import torch
    src, dst = (to_dev(np.array(a, np.int32)) for a in ([0, 1, 2, 3, 4, 5, 0], [1, 2, 3, 4, 5, 0, 3]))
    return gnn.coo_to_csr(6, src, dst), torch.randn((6, 16), device="cuda")


def test_zero_heads_are_an_error_and_not_the_end_of_the_process(gnn, small):
    import torch
    g, X = small
    a, s = torch.zeros((4, 4), device="cuda"), torch.zeros((g.E, 4), device="cuda")
    fwd = gnn.gat_fused(g, X, a, a, 4)
    for call in (lambda H: gnn.edge_dot(g, X, X, H), lambda H: gnn.edge_dot_backward(g, X, X, s, H), lambda H: gnn.gatv2_logits(g, X, X, a, H),
                 lambda H: gnn.gatv2_logits_backward(g, X, X, a, s, H), lambda H: gnn.gat_fused(g, X, a, a, H),
                 lambda H: gnn.gat_fused_backward(g, X, a, a, fwd, X, H)):
        with pytest.raises(ZeroDivisionError):
            call(0)
        with pytest.raises((RuntimeError, ValueError)):  # (GnnError is a RuntimeError)
            call(-1)
        call(4)


def test_none_is_not_an_empty_index(gnn, small):
    import torch
    g, X = small
    i = torch.zeros(3, dtype=torch.int32, device="cuda")
    for call in (lambda: gnn.gather(None, X), lambda: gnn.permute_edge_data(None, X), lambda: gnn.add_self_loops(3, None, i),
                 lambda: gnn.merge_edge_lists([(i, None, 0, 0)]), lambda: gnn.merge_edge_lists([(None, i, 0, 0)]),
                 lambda: gnn.graph_ptr_from_ids(None, 2), lambda: gnn.reduce_nodes(None, X), lambda: gnn.segment_coef(g, i, None),
                 lambda: gnn.linear_backward(None, None, X)):
        with pytest.raises(AttributeError):
            call()


def test_arguments_convert_as_python_would(gnn, small):
    import types
    import torch
    g, X = small
    i = torch.zeros(3, dtype=torch.int32, device="cuda")
    assert torch.equal(gnn.degree(g, transposed=np.bool_(True)), gnn.degree(g, transposed=True))
    assert torch.equal(gnn.propagate_fused(g, X, None, np.float64(gnn.MEAN)), gnn.propagate_fused(g, X, None, "mean"))
    b = torch.ones(16, device="cuda")
    want = gnn.propagate_msg(g, gnn.COPY_XJ, X, epi=dict(Xself=X, self_coef=0.5, bias=b, relu=True))
    for epi in (types.MappingProxyType(dict(Xself=X, self_coef="0.5", bias=b, relu=1)), dict(Xself=X, self_coef=torch.tensor(0.5), self_mode=np.float32(0), bias=b, relu=np.True_)):
        assert torch.equal(gnn.propagate_msg(g, gnn.COPY_XJ, X, epi=epi), want)
    assert torch.equal(gnn.propagate_msg(g, gnn.COPY_XJ, X, epi={}), gnn.propagate_fused(g, X))
    w = torch.ones(g.E, device="cuda")
    assert gnn.propagate_msg_backward(g, gnn.E_MUL_XJ, X, Xj=X, e_csrT=w, e_width=None, want_de=True)["de"].shape == (g.E, 1)
    assert len(gnn.merge_edge_lists([[i, i, np.float64(0), 0]])) == 3


def test_arguments_that_python_would_refuse(gnn, small):
    import torch
    g, X = small
    i = torch.zeros(3, dtype=torch.int32, device="cuda")
    two = torch.zeros(2, device="cuda")
    for error, call in ((ValueError, lambda: gnn.merge_edge_lists([(i, i, 0, 0, 0)])), ((TypeError, ValueError), lambda: gnn.merge_edge_lists([(i, i, 0)])),
                        (RuntimeError, lambda: gnn.linear_bias_act(X, torch.ones((16, 8), device="cuda"), relu=two)),
                        (TypeError, lambda: gnn.propagate_msg(g, gnn.COPY_XJ, X, epi=dict(self_coef=None))),
                        ((AttributeError, TypeError), lambda: gnn.propagate_fused(g, X, ws=False)), (KeyError, lambda: gnn.propagate_fused(g, X, None, "sums")),
                        (TypeError, lambda: gnn.degree(g, transposed=None)), (TypeError, lambda: gnn.gather(i.long(), X)),
                        (TypeError, lambda: gnn.propagate_fused(g, X, torch.ones(g.E, dtype=torch.float64, device="cuda"))),
                        (AssertionError, lambda: gnn.propagate_fused(g, X.t()))):
        with pytest.raises(error):
            call()
