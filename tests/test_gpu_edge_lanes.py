"""The edge-weight gradient at the widths where the number of lanes per edge changes: whole and part-filled rounds of
every lane count, for each width of a load, against the oracle."""
import pytest
import torch

import oracle
from paper_2104_06700_b200 import binding, synth
from parity_util import assert_within_bound, make_graph, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def tiny():
    return synth.tiny(seed=3, n=700, nnz=9000)


# vectors of four, two and one float: 1 to 4, 8/9, 11, 16/17, 24/25, 32/33, 43, 48, 64/65 of them
@pytest.mark.parametrize("F", [k * v for v in (4, 2, 1) for k in (1, 2, 3, 4, 5, 8, 9, 11, 16, 17, 24, 25, 32, 33, 43, 48, 64, 65)
                               if v == 4 or k * v % (2 * v)])
def test_lanes_per_edge(tiny, F):
    g = make_graph(tiny)
    H, G = synth.features(tiny.n, F, 1, DEV), synth.features(tiny.n, F, 2, DEV)
    for op in (binding.DG_OP_SUM, binding.DG_OP_MEAN):
        dW = g.dg_aggregate_edge_grad(H, G, op)
        ref, mag = oracle.edge_weight_grad(to_np(tiny.rowptr), to_np(tiny.colidx), to_np(H), to_np(G), op)
        assert_within_bound(to_np(dW), ref, mag, f"F = {F}")
        assert torch.equal(dW, g.dg_aggregate_edge_grad(H, G, op))


# rows of 32 entries and more, where lanes are halved or not: 4, 8/9, 12/13, 16/17, 24/25, 32/33, 48/49 vectors
@pytest.mark.parametrize("budget", [1, 64])
@pytest.mark.parametrize("F", [4 * k for k in (4, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 48, 49)] + [13, 26, 47])
def test_lanes_per_edge_long_rows(F, budget):
    sg = synth.tiny(seed=4, n=6000, nnz=210_000)
    g = make_graph(sg)
    g.dg_graph_set_param("l2_budget_mb", budget)  # 1 MB: the matrix counts as one that L2 does not keep
    H, G = synth.features(sg.n, F, 1, DEV), synth.features(sg.n, F, 2, DEV)
    dW = g.dg_aggregate_edge_grad(H, G, binding.DG_OP_MEAN)
    ref, mag = oracle.edge_weight_grad(to_np(sg.rowptr), to_np(sg.colidx), to_np(H), to_np(G), binding.DG_OP_MEAN)
    assert_within_bound(to_np(dW), ref, mag, f"F = {F}")
    assert torch.equal(dW, g.dg_aggregate_edge_grad(H, G, binding.DG_OP_MEAN))
