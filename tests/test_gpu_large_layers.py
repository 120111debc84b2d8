"""Layers whose products the library computes (graphsage._large), as a model runs them."""
from types import SimpleNamespace

import pytest
import torch

from paper_2104_06700_b200 import binding, graphsage, synth
from parity_util import make_graph

pytestmark = pytest.mark.gpu
DEV = "cuda"


def random_graph(n, seed=0):
    """Rows of 0 to 8 entries."""
    gen = torch.Generator().manual_seed(seed)
    rowptr = torch.cat([torch.zeros(1, dtype=torch.int64), torch.randint(0, 9, (n,), generator=gen).cumsum(0)])
    nnz = int(rowptr[-1])
    colidx = torch.randint(0, n, (nnz,), generator=gen, dtype=torch.int32)
    return SimpleNamespace(n=n, nnz=nnz, rowptr=rowptr, colidx=colidx, edge_w=None)


@pytest.mark.parametrize("n", [2000, 32768])
@pytest.mark.parametrize("dims,project_first", [([100, 256], False), ([300, 64], True)])
def test_features_of_another_width_are_refused(dims, project_first, n):
    """On a large graph as on a small one, with gradients and without."""
    g = make_graph(random_graph(n))
    model = graphsage.GraphSAGE(g, dims, project_first=project_first).to(DEV)
    for width in (dims[0] + 28, dims[0] - 4):
        X = synth.features(n, width, 1, DEV)
        with pytest.raises((RuntimeError, ValueError)):
            model(X)
        with torch.no_grad(), pytest.raises((RuntimeError, ValueError)):
            model(X)


@pytest.fixture
def tf32():
    torch.set_float32_matmul_precision("high")
    yield
    torch.set_float32_matmul_precision("highest")


def test_a_caller_who_asked_for_tf32_keeps_it(tf32):
    n, dims = 8192 + 5, [256, 256]
    g = make_graph(random_graph(n))
    g.dg_graph_transpose()
    model = graphsage.GraphSAGE(g, dims).to(DEV)
    X, dOut = synth.features(n, 256, 1, DEV).requires_grad_(True), synth.features(n, 256, 2, DEV)
    W, b = (p.detach() for p in model.parameters())
    out = model(X)
    out.backward(dOut)
    Z = g.dg_aggregate_fwd_self(X.detach(), binding.DG_OP_SUM)
    assert torch.equal(out, g.dg_layer_fwd(Z @ W.t(), model.inv_deg1, b, False))
    G, _ = g.dg_layer_bwd(dOut, None, model.inv_deg1)
    assert torch.equal(X.grad, g.dg_aggregate_bwd_self(G @ W, binding.DG_OP_SUM))
    torch.set_float32_matmul_precision("highest")
    assert not torch.equal(out, model(X))
