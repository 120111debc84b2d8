"""Layers whose products the library computes (graphsage._by_library), as a model runs them."""
from types import SimpleNamespace

import pytest
import torch

from paper_2104_06700_b200 import binding, graphsage, synth
from parity_util import make_graph
from test_gpu_epoch import reference_forward

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


def run(g, sg, dims, project_first=False, fused=False, bf16=False, relayout=False):
    """Output and gradients of a model on g, and those of the fp64 reference."""
    torch.manual_seed(0)
    model = graphsage.GraphSAGE(g, dims, project_first=project_first, fused_aggregator=fused, bf16_aggregate=bf16).to(DEV)
    if relayout:  # columns of the weights side by side
        for lin in model.lin:
            lin.weight.data = lin.weight.data.t().contiguous().t()
    X = synth.features(sg.n, dims[0], 3, DEV).requires_grad_(True)
    dOut = synth.features(sg.n, dims[-1], 4, DEV)
    out = model(X)
    out.backward(dOut)
    got = [out.detach(), X.grad] + [p.grad for p in model.parameters()]
    Xr = X.detach().double().requires_grad_(True)
    Ws = [lin.weight.detach().clone().requires_grad_(True) for lin in model.lin]
    bs = [lin.bias.detach().clone().requires_grad_(True) for lin in model.lin]
    ref = reference_forward(sg, Xr, Ws, bs)
    ref.backward(dOut.double())
    return got, [ref.detach(), Xr.grad] + [t.grad for pair in zip(Ws, bs) for t in pair]


def close(got, want, rel):
    for x, y in zip(got, want):
        assert float((x.double() - y.double()).norm()) <= rel * float(y.double().norm())


@pytest.fixture
def calls(monkeypatch):
    """Counts the calls of the library's products."""
    count = {}
    for name in ("dg_linear_fwd", "dg_linear_bwd_input", "dg_linear_bwd_weight"):
        def counted(self, *args, _name=name, _call=getattr(binding.Graph, name), **kwargs):
            count[_name] = count.get(_name, 0) + 1
            return _call(self, *args, **kwargs)
        monkeypatch.setattr(binding.Graph, name, counted)
    return lambda: tuple(count.get(f"dg_linear_{name}", 0) for name in ("fwd", "bwd_input", "bwd_weight"))


# 2^29 multiplications from 8192 rows of 256 x 256 on, and from 44 621 of 256 x 47
@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("n,dims,project_first,expected", [
    (8192, [256, 256], False, (1, 1, 1)), (8191, [256, 256], False, (0, 0, 0)), (8192, [300, 256], True, (1, 1, 1)),
    (44621, [100, 256, 47], False, (2, 2, 1)), (44620, [256, 47], True, (0, 0, 0)), (44621, [256, 47], True, (1, 1, 0)),
    (44621, [256, 47], False, (1, 1, 0)), (40000, [128, 47, 300], False, (1, 0, 0)),
    (36000, [100, 150], False, (1, 1, 1)), (45000, [64, 200], False, (1, 0, 0)), (84000, [64, 100], False, (1, 0, 1)),
    (5000, [602, 256], False, (0, 1, 1)), (30000, [602, 47], False, (1, 0, 0))])
def test_large_layers_match_fp64(n, dims, project_first, fused, expected, calls):
    sg = random_graph(n)
    g = make_graph(sg)
    g.dg_graph_set_param("self_loops", int(fused))
    g.dg_graph_transpose()
    got, want = run(g, sg, dims, project_first, fused)
    # fp32 sums; a unit whose sum is within rounding of zero may fall on the other side of the ReLU
    close(got, want, 1e-6 if len(dims) == 2 else 1e-3)
    assert calls() == expected


@pytest.mark.parametrize("project_first", [False, True])
@pytest.mark.parametrize("fused", [False, True])
def test_large_layers_of_bf16_rows(project_first, fused, calls):
    sg = random_graph(8200)
    g = make_graph(sg)
    g.dg_graph_set_param("self_loops", int(fused))
    g.dg_graph_transpose()
    got, want = run(g, sg, [300, 256], project_first, fused, bf16=True)
    close(got, want, 2.0 ** -8)  # the rows that are added are rounded to bf16
    assert calls() == (1, 1, 1)


@pytest.mark.parametrize("project_first", [False, True])
def test_weights_whose_columns_lie_side_by_side(project_first, calls):
    sg = random_graph(8200)
    g = make_graph(sg)
    g.dg_graph_transpose()
    close(*run(g, sg, [300, 256], project_first, relayout=True), 1e-6)
    assert calls() == (1, 1, 1)


@pytest.mark.parametrize("scratch_mb,expected", [(0, (1, 1, 0)), (1, (1, 1, 0)), (6, (1, 1, 0)), (7, (1, 1, 1))])
def test_large_layers_within_a_scratch_limit(scratch_mb, expected, calls):
    sg = random_graph(8200)
    g = make_graph(sg)
    g.dg_graph_transpose()
    g.dg_graph_set_param("scratch_mb", scratch_mb)
    close(*run(g, sg, [300, 256]), 1e-6)
    assert calls() == expected


def test_gradients_of_a_large_layer_can_be_differentiated():
    n = 8200
    sg = random_graph(n)
    g = make_graph(sg)
    g.dg_graph_transpose()
    torch.manual_seed(0)
    model = graphsage.GraphSAGE(g, [256, 256]).to(DEV)
    X, labels = synth.features(n, 256, 3, DEV), torch.randint(0, 256, (n,), device=DEV)

    def penalty(logits, params):
        loss = torch.nn.functional.cross_entropy(logits, labels)
        return sum((d * d).sum() for d in torch.autograd.grad(loss, params, create_graph=True))

    got = torch.autograd.grad(penalty(model(X), list(model.parameters())), list(model.parameters()))
    W, b = (p.detach().double().requires_grad_(True) for p in model.parameters())
    close(got, torch.autograd.grad(penalty(reference_forward(sg, X, [W], [b]), [W, b]), [W, b]), 1e-5)


def test_large_layers_in_a_captured_epoch():
    """The products and their scratch in a CUDA graph, replayed on new features."""
    n, dims = 8200, [100, 256, 256]
    sg = random_graph(n)
    g = make_graph(sg)
    g.dg_graph_transpose()
    torch.manual_seed(0)
    model = graphsage.GraphSAGE(g, dims).to(DEV)
    X, dOut = synth.features(n, 100, 3, DEV), synth.features(n, 256, 4, DEV)
    params = list(model.parameters())
    step = lambda: torch.autograd.grad(model(X), params, dOut)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        grads = step()
    X.copy_(synth.features(n, 100, 5, DEV))
    graph.replay()
    torch.cuda.synchronize()
    for got, want in zip(grads, step()):
        assert torch.equal(got, want)
