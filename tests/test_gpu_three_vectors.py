"""Slices of 33 to 44 vectors, where a lane takes three of them, and the widths beside them, on graphs with rows long
enough for that: against the oracle, with weights, own rows, cut rows and padded copies."""
import numpy as np
import pytest
import torch

from paper_2104_06700_b200 import binding, synth
from parity_util import check_fwd_bwd, check_transpose
from test_gpu_chunks import graph_of, handle, host

pytestmark = pytest.mark.gpu
DEV = "cuda"
# rows around one and several pieces; mean degrees 24.2 and 23.8
LENGTHS = [0, 1, 7, 8, 9, 31, 32, 33, 64, 65, 161, 300, 1025, 3, 2]


@pytest.mark.parametrize("F", [128, 132, 136, 172, 176, 180, 171])
@pytest.mark.parametrize("weighted,self_loops", [(False, 0), (True, 0), (False, 1)])
@pytest.mark.parametrize("n", [72, 73])
def test_three_vectors_per_lane(F, weighted, self_loops, n):
    assert np.sum(LENGTHS) == 1741
    sg = graph_of(LENGTHS, n, F, weighted)
    g = handle(sg, self_loops)
    csc = check_transpose(g, *host(sg))
    H, G = synth.features(sg.n, F, 1, DEV), synth.features(sg.n, F, 2, DEV)
    for op in (binding.DG_OP_SUM, binding.DG_OP_MEAN):
        check_fwd_bwd(g, host(sg), H, G, op, csc, self_loops=bool(self_loops))


@pytest.mark.parametrize("blocks", [2, 8])
@pytest.mark.parametrize("weighted,self_loops", [(False, 0), (True, 0), (False, 1)])
def test_with_source_blocks(weighted, self_loops, blocks):
    """Three vectors per lane, and beside them the widths whose lane groups take neighbouring edges."""
    n, deg = 700, 80
    rng = np.random.default_rng(3)
    src = np.sort(np.stack([rng.choice(n, deg, replace=False) for _ in range(n)]), axis=1).astype(np.int32).reshape(-1)
    rowptr = np.arange(n + 1, dtype=np.int64) * deg
    w = rng.random(n * deg).astype(np.float32) if weighted else None
    g = binding.dg_graph_create(n, n * deg, torch.as_tensor(rowptr, device=DEV), torch.as_tensor(src, device=DEV),
                                None if w is None else torch.as_tensor(w, device=DEV))
    g.dg_graph_set_param("self_loops", self_loops)
    g.dg_graph_set_param("source_blocks", blocks)
    csc = check_transpose(g, rowptr, src, w)
    for F in (136, 172, 8, 16, 32, 48):
        H, G = synth.features(n, F, 1, DEV), synth.features(n, F, 2, DEV)
        for op in (binding.DG_OP_SUM, binding.DG_OP_MEAN):
            check_fwd_bwd(g, (rowptr, src, w), H, G, op, csc, self_loops=bool(self_loops))
