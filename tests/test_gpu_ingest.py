"""The CSC build where its last pass finds rows, counts columns and scans: row starts at every place of a block of 32
positions with empty rows between them, edge counts around a sort tile, vertex counts around a digit and around what one
block scans.  Bit-exact against the oracle's counting sort; the mean's factors through the
backward pass, within its bound."""
import numpy as np
import pytest
import torch

import oracle
from paper_2104_06700_b200 import binding, synth
from parity_util import assert_within_bound, check_transpose, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda"


def build(lengths, n, seed, weighted, self_loops):
    rng = np.random.default_rng(seed)
    deg = np.zeros(n, dtype=np.int64)
    deg[: len(lengths)] = lengths
    rowptr = np.concatenate([[0], np.cumsum(deg)])
    nnz = int(rowptr[-1])
    cols = (n * rng.random(nnz) ** 3).astype(np.int32)  # some columns long, most empty where n is large
    w = rng.random(nnz).astype(np.float32) if weighted else None
    g = binding.dg_graph_create(n, nnz, torch.as_tensor(rowptr, device=DEV), torch.as_tensor(cols, device=DEV),
                                None if w is None else torch.as_tensor(w, device=DEV))
    g.dg_graph_set_param("self_loops", self_loops)
    return g, rowptr, cols, w


def check(g, rowptr, cols, w, self_loops):
    colptr, rowidx, w_T = check_transpose(g, rowptr, cols, w)
    X = synth.features(g.n, 4, 3, DEV)
    ref, mag = oracle.ap_backward(rowptr, colptr, rowidx, w_T, to_np(X), binding.DG_OP_MEAN, self_loops=bool(self_loops))
    assert_within_bound(to_np(g.dg_aggregate_bwd(X, binding.DG_OP_MEAN)), ref, mag, "factors")


# rows of 1 to 70 entries with none to three empty rows between them: starts at every position of a block of 32
STAGGERED = [x for k in range(1, 71) for x in [k] + [0] * (k % 4)]


@pytest.mark.parametrize("weighted,self_loops", [(False, 0), (True, 0), (False, 1), (True, 1)])
@pytest.mark.parametrize("lengths,n", [(STAGGERED, 200), ([0] * 40 + STAGGERED[::-1], 300), ([1] * 100, 513),
                                       ([0, 33, 0, 0, 31, 32, 0], 70000), ([5000, 0, 1, 0, 200], 131073)],
                         ids=["staggered", "leading", "single", "blocks", "long"])
def test_rows_of_positions(lengths, n, weighted, self_loops):
    g, *csr = build(lengths, n, n, weighted, self_loops)
    check(g, *csr, self_loops)


# tiles of 4096 keys; 64 tiles of 256 digits, and 16383 vertices, are what one block scans
@pytest.mark.parametrize("nnz,n", [(4095, 256), (4096, 257), (4097, 512), (262144, 16383), (262145, 16384), (8193, 65537),
                                   (300000, 16385)])
def test_tiles_digits_and_scans(nnz, n):
    lengths = np.full(n, nnz // n)
    lengths[: nnz - int(lengths.sum())] += 1
    weighted = nnz % 2 == 1
    g, *csr = build(lengths, n, nnz, weighted, 0)
    check(g, *csr, 0)
