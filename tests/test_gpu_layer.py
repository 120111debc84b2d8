"""The elementwise passes around a layer's GEMM (dg_layer_fwd / dg_layer_bwd) against the same operations in
fp64, at the sizes where a thread's columns or rows run out: one vector, scalar columns, a second tile of
columns, one row, and more rows than the grid holds at once."""
import pytest
import torch

from paper_2104_06700_b200 import binding, graphsage

pytestmark = pytest.mark.gpu
DEV = "cuda"
EPS = 2.0 ** -24


def empty_graph(n):
    return binding.dg_graph_create(n, 0, torch.zeros(n + 1, dtype=torch.int64, device=DEV),
                                   torch.zeros(0, dtype=torch.int32, device=DEV), None)


@pytest.mark.parametrize("relu", [False, True])
@pytest.mark.parametrize("n,F", [(1, 1), (1, 256), (3, 4), (17, 47), (1023, 257), (1025, 1028), (5000, 256),
                                 (40000, 47), (100000, 64)])
def test_layer_passes_match_fp64(n, F, relu):
    gen = torch.Generator(device=DEV).manual_seed(n + F)
    Y, dOut = (torch.randn(n, F, device=DEV, generator=gen) for _ in range(2))
    scale = torch.rand(n, 1, device=DEV, generator=gen)
    bias = torch.randn(F, device=DEV, generator=gen)
    g = empty_graph(n)

    want = Y.double() * scale.double() + bias.double()
    bound = 2 * EPS * ((Y.double() * scale.double()).abs() + bias.double().abs())  # at most two roundings
    if relu:
        want = want.relu()
    out = g.dg_layer_fwd(Y.clone(), scale, bias, relu)
    assert bool(((out.double() - want).abs() <= bound).all())

    G, db = g.dg_layer_bwd(dOut, out if relu else None, scale)
    d = torch.where(out > 0, dOut, 0.0) if relu else dOut
    assert torch.equal(G, d * scale)
    # a sum of n terms in any order: (n - 1) roundings of partial sums, each at most the sum of |d|
    assert bool(((db.double() - d.double().sum(0)).abs() <= n * EPS * d.double().abs().sum(0)).all())
    G2, db2 = g.dg_layer_bwd(dOut, out if relu else None, scale)
    assert torch.equal(G, G2) and torch.equal(db, db2)


@pytest.mark.parametrize("n,F", [(1, 1), (2047, 33), (2048, 32), (70001, 260)])
def test_layer_backward_without_scratch(n, F):
    """The bias's gradient straight from dOut, before G takes its place."""
    gen = torch.Generator(device=DEV).manual_seed(n + F)
    dOut, out = (torch.randn(n, F, device=DEV, generator=gen) for _ in range(2))
    scale = torch.rand(n, 1, device=DEV, generator=gen)
    g = empty_graph(n)
    g.dg_graph_set_param("scratch_mb", 0)
    for mask in (None, out):
        d = dOut if mask is None else torch.where(out > 0, dOut, 0.0)
        G, db = g.dg_layer_bwd(dOut, mask, scale)
        assert torch.equal(G, d * scale)
        assert bool(((db.double() - d.double().sum(0)).abs() <= n * EPS * d.double().abs().sum(0)).all())


def test_nan_passes_through_and_arguments_are_checked():
    g = empty_graph(4)
    scale, bias = torch.ones(4, 1, device=DEV), torch.zeros(8, device=DEV)
    out = g.dg_layer_fwd(torch.full((4, 8), float("nan"), device=DEV), scale, bias, True)
    assert bool(out.isnan().all())
    G, _ = g.dg_layer_bwd(torch.ones(4, 8, device=DEV), out, scale)
    assert torch.equal(G, torch.ones(4, 8, device=DEV))  # as torch's ReLU
    for bad in (dict(row_scale=None), dict(bias=None)):
        with pytest.raises(binding.DgError):
            g.dg_layer_fwd(out, **{"row_scale": scale, "bias": bias, "relu": True, **bad})


@pytest.mark.parametrize("n", [8191, 8192, 8257, 20000])
def test_weight_gradient_in_slices(n):
    gen = torch.Generator(device=DEV).manual_seed(n)
    G, X = torch.randn(n, 130, device=DEV, generator=gen), torch.randn(n, 128, device=DEV, generator=gen)
    want = G.double().t() @ X.double()
    bound = n * EPS * (G.double().abs().t() @ X.double().abs())
    assert bool(((graphsage._weight_grad(G, X).double() - want).abs() <= bound).all())
