"""The GraphSAGE epoch built on the aggregation primitive against a pure-torch reference
(index_add_ for the neighbour sum, autograd for everything): loss and every weight gradient."""
import pytest
import torch

from paper_2104_06700_b200 import binding, graphsage, synth
from parity_util import make_graph

pytestmark = pytest.mark.gpu
DEV = "cuda"


def reference_forward(sg, X, weights, biases):
    n = sg.n
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), (sg.rowptr[1:] - sg.rowptr[:-1]).to(DEV))
    cols = sg.colidx.to(DEV).long()
    deg1 = (sg.rowptr[1:] - sg.rowptr[:-1]).to(DEV).double() + 1.0
    H = X.double()
    for i, (W, b) in enumerate(zip(weights, biases)):
        agg = torch.zeros_like(H).index_add_(0, rows, H[cols])
        Z = (agg + H) / deg1.unsqueeze(1)
        H = Z @ W.double().t() + b.double()
        if i + 1 < len(weights):
            H = torch.relu(H)
    return H


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("project_first", [False, True])
@pytest.mark.parametrize("dims", [[64, 32, 7], [20, 16, 16, 5]])
def test_epoch_loss_and_gradients_match_torch_reference(dims, project_first, fused):
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    if fused:
        g.dg_graph_set_param("self_loops", 1)
    g.dg_graph_transpose()
    torch.manual_seed(0)
    model = graphsage.GraphSAGE(g, dims, project_first=project_first,
                                fused_aggregator=fused).to(DEV)
    X = synth.features(sg.n, dims[0], 3, DEV)
    labels = torch.randint(0, dims[-1], (sg.n,), device=DEV)
    train_idx = torch.arange(0, sg.n, 3, device=DEV)

    logits = model(X)
    loss = torch.nn.functional.cross_entropy(logits[train_idx], labels[train_idx])
    loss.backward()

    Ws = [l.weight.detach().clone().requires_grad_(True) for l in model.lin]
    bs = [l.bias.detach().clone().requires_grad_(True) for l in model.lin]
    ref_logits = reference_forward(sg, X, Ws, bs)
    ref_loss = torch.nn.functional.cross_entropy(ref_logits[train_idx], labels[train_idx])
    ref_loss.backward()

    assert abs(float(loss) - float(ref_loss)) <= 1e-4 * abs(float(ref_loss))
    for lin, W, b in zip(model.lin, Ws, bs):
        for got, want in ((lin.weight.grad, W.grad), (lin.bias.grad, b.grad)):
            scale = float(want.abs().max()) + 1e-12
            assert float((got.double() - want.double()).abs().max()) <= 1e-4 * scale


def test_epoch_function_trains():
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_transpose()
    torch.manual_seed(1)
    model = graphsage.GraphSAGE(g, [64, 32, 7]).to(DEV)
    X = synth.features(sg.n, 64, 4, DEV)
    labels = torch.randint(0, 7, (sg.n,), device=DEV)
    epoch = graphsage.make_epoch(model, X, labels, torch.arange(sg.n, device=DEV))
    losses = [float(epoch()) for _ in range(30)]
    assert losses[-1] < losses[0]
    assert graphsage.aggregation_calls([64, 32, 7]) == [("fwd", 64), ("fwd", 32), ("bwd", 32)]
    assert graphsage.aggregation_calls([64, 32, 7], True) == [("fwd", 32), ("bwd", 32),
                                                              ("fwd", 7), ("bwd", 7)]
    assert graphsage.aggregation_calls([16, 32, 32, 7], True) == [
        ("fwd", 16), ("fwd", 32), ("bwd", 32), ("fwd", 7), ("bwd", 7)]


def test_bf16_aggregation_stays_close_to_fp32():
    """Aggregating bf16-rounded activations changes the loss by bf16 rounding only."""
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_transpose()
    X = synth.features(sg.n, 64, 3, DEV)
    labels = torch.randint(0, 8, (sg.n,), device=DEV)
    losses = []
    for bf in (False, True):
        torch.manual_seed(0)
        model = graphsage.GraphSAGE(g, [64, 32, 8], bf16_aggregate=bf).to(DEV)
        logits = model(X)
        loss = torch.nn.functional.cross_entropy(logits, labels)
        loss.backward()
        losses.append((float(loss), model.lin[0].weight.grad.clone()))
    assert abs(losses[0][0] - losses[1][0]) <= 2e-2 * abs(losses[0][0])
    scale = float(losses[0][1].abs().max())
    assert float((losses[0][1] - losses[1][1]).abs().max()) <= 5e-2 * scale


def test_fused_aggregator_needs_the_matching_handle():
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    with pytest.raises(ValueError):
        graphsage.GraphSAGE(g, [8, 4], fused_aggregator=True)
    g.dg_graph_set_param("self_loops", 1)
    with pytest.raises(ValueError):
        graphsage.GraphSAGE(g, [8, 4])


@pytest.mark.parametrize("op", [binding.DG_OP_SUM, binding.DG_OP_MEAN])
def test_learnable_edge_weights_gradient_and_refresh(op):
    """The autograd wrapper returns the gradient with respect to the edge weights (one dot product
    per edge, dg_aggregate_edge_grad) next to the one for the features; after an in-place update of
    the weights dg_graph_update_weights brings the CSC of the backward pass up to date.  Reference:
    index_add_ with autograd in fp64."""
    sg = synth.make("tiny")
    rowptr, colidx = sg.rowptr.to(DEV), sg.colidx.to(DEV)
    w = sg.edge_w.to(DEV).clone().requires_grad_(True)
    g = binding.dg_graph_create(sg.n, sg.nnz, rowptr, colidx, w.detach())
    assert w.data_ptr() == g.edge_w.data_ptr()
    g.dg_graph_transpose()
    F = 48
    rows = torch.repeat_interleave(torch.arange(sg.n, device=DEV), rowptr[1:] - rowptr[:-1])
    deg = (rowptr[1:] - rowptr[:-1]).double().clamp(min=1).unsqueeze(1)

    def reference(H, wt):
        out = torch.zeros((sg.n, F), dtype=torch.float64, device=DEV)
        out.index_add_(0, rows, H.double()[colidx.long()] * wt.double().unsqueeze(1))
        return out / deg if op == binding.DG_OP_MEAN else out

    for step in range(2):
        H = synth.features(sg.n, F, 70 + step, DEV).requires_grad_(True)
        G = synth.features(sg.n, F, 80 + step, DEV)
        out = graphsage.aggregate(g, H, op, edge_w=w)
        (out * G).sum().backward()
        Hr = H.detach().clone().requires_grad_(True)
        wr = w.detach().clone().requires_grad_(True)
        (reference(Hr, wr) * G.double()).sum().backward()
        assert torch.allclose(out.detach().double(), reference(H.detach(), w.detach()),
                              rtol=1e-4, atol=1e-4)
        assert torch.allclose(H.grad.double(), Hr.grad.double(), rtol=1e-4, atol=1e-4)
        assert torch.allclose(w.grad.double(), wr.grad.double(), rtol=1e-4, atol=1e-3)
        with torch.no_grad():                       # an optimiser step on the weights, in place
            w -= 0.05 * w.grad
            w.grad = None
        g.dg_graph_update_weights()


@pytest.mark.parametrize("fused", [False, True])
def test_layers_call_a_linear_that_is_more_than_its_parameters(fused):
    """Hooks, parametrizations, a missing bias and modules in a Linear's place take part in forward and backward."""
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_set_param("self_loops", int(fused))
    g.dg_graph_transpose()
    X = synth.features(sg.n, 24, 3, DEV)
    dims = [24, 16, 16, 5]
    G = synth.features(sg.n, 5, 4, DEV)

    class Doubled(torch.nn.Linear):
        def forward(self, x):
            return 2.0 * super().forward(x)

    class Halved(torch.nn.Module):
        def forward(self, W):
            return 0.5 * W

    def changed(kind, model):
        """Changes the middle layer; the weight and bias it has in effect."""
        lin = model.lin[1]
        if kind == "hook":
            lin.register_forward_hook(lambda module, args, out: 2.0 * out)
            return 2.0 * lin.weight.detach(), 2.0 * lin.bias.detach()
        if kind == "pre-hook":
            lin.register_forward_pre_hook(lambda module, args: (2.0 * args[0],))
            return 2.0 * lin.weight.detach(), lin.bias.detach()
        if kind == "parametrization":
            torch.nn.utils.parametrize.register_parametrization(lin, "weight", Halved())
            return lin.weight.detach(), lin.bias.detach()
        if kind == "module":
            model.lin[1] = Doubled(16, 16).to(DEV)
            return 2.0 * model.lin[1].weight.detach(), 2.0 * model.lin[1].bias.detach()
        model.lin[1] = torch.nn.Linear(16, 16, bias=False).to(DEV)
        return model.lin[1].weight.detach(), torch.zeros(16, device=DEV)

    for kind in ("hook", "pre-hook", "parametrization", "module", "no bias"):
        torch.manual_seed(0)
        model = graphsage.GraphSAGE(g, dims, fused_aggregator=fused).to(DEV)
        weights = [l.weight.detach().double() for l in model.lin]
        biases = [l.bias.detach().double() for l in model.lin]
        weights[1], biases[1] = (t.double() for t in changed(kind, model))
        x = X.clone().requires_grad_(True)
        out = model(x)
        (out * G).sum().backward()
        xr = X.double().requires_grad_(True)
        want = reference_forward(sg, xr, weights, biases)
        (want * G.double()).sum().backward()
        for got, ref in ((out.detach(), want.detach()), (x.grad, xr.grad)):
            assert float((got.double() - ref).abs().max()) <= 1e-4 * float(ref.abs().max()), kind


def test_a_layer_under_autocast_gives_what_its_linear_gives():
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_transpose()
    model = graphsage.GraphSAGE(g, [24, 5]).to(DEV)
    X = synth.features(sg.n, 24, 3, DEV)
    with torch.autocast("cuda", torch.bfloat16):
        out = model(X)
    assert out.dtype == torch.bfloat16
    want = reference_forward(sg, X, [model.lin[0].weight], [model.lin[0].bias])
    # operands and result rounded to bf16: 2^-9 each of the terms, 24 of them
    assert float((out.double() - want).abs().max()) <= 24 * 3 * 2.0 ** -9 * float(X.abs().max())


def test_gradients_of_a_layer_can_be_differentiated():
    """A gradient penalty on the weights of a one-layer model (its input needs no gradient), against fp64."""
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_transpose()
    torch.manual_seed(0)
    model = graphsage.GraphSAGE(g, [24, 5]).to(DEV)
    X = synth.features(sg.n, 24, 3, DEV)
    labels = torch.randint(0, 5, (sg.n,), device=DEV)

    def penalty(logits, params):
        loss = torch.nn.functional.cross_entropy(logits, labels)
        return sum((d * d).sum() for d in torch.autograd.grad(loss, params, create_graph=True))

    got = torch.autograd.grad(penalty(model(X), list(model.parameters())), list(model.parameters()))
    W, b = (p.detach().double().requires_grad_(True) for p in model.parameters())
    want = torch.autograd.grad(penalty(reference_forward(sg, X, [W], [b]), [W, b]), [W, b])
    for x, y in zip(got, want):
        assert float((x.double() - y).abs().max()) <= 1e-4 * float(y.abs().max())


@pytest.mark.parametrize("bf16", [False, True])
def test_both_backward_forms_of_the_mean_with_own_rows(bf16):
    """aggregate(..., DG_OP_MEAN) on a handle with self loops: per-edge factors of the transposition, or dOut scaled row
    by row and the sum's backward pass (row_scale)."""
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_set_param("self_loops", 1)
    g.dg_graph_transpose()
    X, G = synth.features(sg.n, 24, 3, DEV), synth.features(sg.n, 24, 4, DEV)
    inv = 1.0 / ((sg.rowptr[1:] - sg.rowptr[:-1]).to(DEV).float() + 1.0).unsqueeze(1)
    eye, zero = torch.eye(24, device=DEV), torch.zeros(24, device=DEV)
    xr = X.double().requires_grad_(True)
    want = reference_forward(sg, xr, [eye], [zero])
    (want * G.double()).sum().backward()
    tol = 2.0 ** -8 if bf16 else 1e-5
    for scale in (None, inv):
        x = X.clone().requires_grad_(True)
        out = graphsage.aggregate(g, x, binding.DG_OP_MEAN, bf16, row_scale=scale)
        (out * G).sum().backward()
        for a, b in ((out.detach(), want.detach()), (x.grad, xr.grad)):
            assert float((a.double() - b).abs().max()) <= tol * float(b.abs().max())
