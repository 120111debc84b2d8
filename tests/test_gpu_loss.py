"""dg_cross_entropy_fwd / _bwd against torch's cross-entropy in fp64: classes at the edges of a warp and of the
registers, row counts at the edges of a warp's and a block's share, rows named twice, from the end, or ignored."""
import pytest
import torch

from paper_2104_06700_b200 import binding, graphsage, synth
from parity_util import make_graph

pytestmark = pytest.mark.gpu
DEV = "cuda"
EPS = 2.0 ** -24


def empty_graph(n):
    return binding.dg_graph_create(n, 0, torch.zeros(n + 1, dtype=torch.int64, device=DEV),
                                   torch.zeros(0, dtype=torch.int32, device=DEV), None)


@pytest.mark.parametrize("C", [1, 2, 32, 33, 47, 64, 65, 128, 129, 400])
@pytest.mark.parametrize("count", [1, 15, 16, 17, 128, 129, 5000])
def test_loss_and_gradient_match_fp64(count, C):
    n = 3000
    gen = torch.Generator(device=DEV).manual_seed(count + C)
    logits = torch.randn(n, C, device=DEV, generator=gen) * 4 + 30
    labels = torch.randint(0, C, (n,), device=DEV, generator=gen)
    index = torch.randint(-n, n, (count,), device=DEV, generator=gen)
    if count > 2:
        labels[index[count // 2]] = -100
        index[0] = index[count - 1]
    x = logits.double().requires_grad_(True)
    want = torch.nn.functional.cross_entropy(x[index], labels[index])
    (want * 0.5).backward()
    g = empty_graph(n)
    y = logits.clone().requires_grad_(True)
    loss = graphsage._CrossEntropy.apply(y, index, labels, g)
    (loss * 0.5).backward()
    # x - max is off by eps |x - max| < 64 eps (32 when rounded to nearest), expf and logf by a few eps of their
    # own, the sum of up to 400 terms by log2(32) + 400 / 32 eps; a gradient p / rows is off by as much of itself
    rel = (64 + 20 + 8) * EPS
    if bool(want.isnan()):
        assert bool(loss.isnan())
        return
    assert abs(float(loss) - float(want)) <= rel * (1 + abs(float(want)))
    counts = torch.zeros(n, device=DEV, dtype=torch.float64)
    counts.index_add_(0, index % n, torch.ones(count, device=DEV, dtype=torch.float64))
    rows = int((labels[index] != -100).sum())
    bound = rel * counts.unsqueeze(1) * 0.5 / rows
    assert bool(((y.grad.double() - x.grad).abs() <= bound).all())
    y2 = logits.clone().requires_grad_(True)
    loss2 = graphsage._CrossEntropy.apply(y2, index, labels, g)
    (loss2 * 0.5).backward()
    assert torch.equal(loss, loss2) and torch.equal(y.grad, y2.grad)


@pytest.mark.parametrize("C", [1, 47, 400])
@pytest.mark.parametrize("count", [1, 128, 129, 5000])
def test_loss_without_scratch(count, C):
    """One block walks all shares: the same statistics; the mean adds the same doubles in another order, so it is the
    same float up to its last rounding."""
    n = 3000
    gen = torch.Generator(device=DEV).manual_seed(count + C)
    logits = torch.randn(n, C, device=DEV, generator=gen) * 4 + 30
    labels = torch.randint(0, C, (n,), device=DEV, generator=gen)
    index = torch.randint(-n, n, (count,), device=DEV, generator=gen)
    g, without = empty_graph(n), empty_graph(n)
    without.dg_graph_set_param("scratch_mb", 0)
    want, stats = g.dg_cross_entropy_fwd(logits, index, labels)
    got, stats2 = without.dg_cross_entropy_fwd(logits, index, labels)
    assert torch.equal(stats, stats2)
    assert bool(((got - want).abs() <= 2 * EPS * want.abs()).all())


def test_out_of_range_targets_give_nan_and_nothing_else():
    g = empty_graph(10)
    logits = torch.zeros(10, 4, device=DEV)
    for index, label in ((10, 0), (-11, 0), (3, 4), (3, -1)):
        labels = torch.zeros(10, dtype=torch.int64, device=DEV)
        labels[3] = label
        idx = torch.tensor([0, index], device=DEV)
        result, stats = g.dg_cross_entropy_fwd(logits, idx, labels)
        assert bool(result[0].isnan())
        d = g.dg_cross_entropy_bwd(logits, idx, labels, result, stats, torch.ones((), device=DEV))
        assert bool((d[1:] == 0).all()) and bool((d[0] != 0).all())
    none = torch.zeros(0, dtype=torch.int64, device=DEV)
    result, stats = g.dg_cross_entropy_fwd(logits, none, labels)
    assert bool(result[0].isnan())
    assert not g.dg_cross_entropy_bwd(logits, none, labels, result, stats, torch.ones((), device=DEV)).any()


@pytest.mark.parametrize("mask", [False, True])
def test_epoch_takes_indices_and_masks(mask):
    sg = synth.make("tiny", weighted=False)
    g = make_graph(sg)
    g.dg_graph_transpose()
    torch.manual_seed(1)
    model = graphsage.GraphSAGE(g, [16, 8, 5]).to(DEV)
    X = synth.features(sg.n, 16, 4, DEV)
    labels = torch.randint(0, 5, (sg.n,), device=DEV)
    train = torch.arange(0, sg.n, 3, device=DEV)
    want = float(torch.nn.functional.cross_entropy(model(X)[train].double(), labels[train]))
    if mask:
        train = torch.zeros(sg.n, dtype=torch.bool, device=DEV).index_fill_(0, train, True)
    got = float(graphsage.make_epoch(model, X, labels, train)())
    assert abs(got - want) <= 1e-5 * want
    with pytest.raises(IndexError):
        graphsage.make_epoch(model, X, labels + 5, torch.arange(3, device=DEV))
