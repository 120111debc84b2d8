"""Which products of a layer go to the library: a rule on sizes, no GPU needed."""
from types import SimpleNamespace

import pytest
import torch

from paper_2104_06700_b200 import graphsage


def rule(n, K, N, scratch_mb=4096):
    graph = SimpleNamespace(n=n, dg_graph_get_param=lambda name: {"scratch_mb": scratch_mb}[name])
    return graphsage._by_library(graph, torch.empty(N, K, device="meta"))


@pytest.mark.parametrize("n,K,N,expected", [
    (8192, 256, 256, (True, True, True)), (8191, 256, 256, (False, False, False)), (10 ** 7, 39, 256, (False, False, False)),
    (245000, 256, 47, (True, True, False)), (245000, 64, 47, (True, False, True)), (245000, 47, 47, (True, False, False)),
    (245000, 602, 41, (True, False, False)), (4096, 602, 256, (False, True, True)), (4096, 256, 602, (True, False, True)),
    # wider than the library's calls take: torch's products serve these as ever
    (4096, 1 << 20, 64, (False, True, False)), (4096, (1 << 20) + 1, 64, (False, False, False)),
    (4096, 64, (1 << 20) + 4, (False, False, False))])
def test_products_by_size(n, K, N, expected):
    assert rule(n, K, N) == expected
    assert rule(n, K, N, scratch_mb=6) == (*expected[:2], False)


def test_a_callers_matmul_precision_is_kept():
    try:
        torch.set_float32_matmul_precision("high")
        assert rule(245000, 256, 256) == (False, False, False)
    finally:
        torch.set_float32_matmul_precision("highest")
    assert rule(245000, 256, 256) == (True, True, True)
