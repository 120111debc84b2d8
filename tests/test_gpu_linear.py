"""The matrix products of a layer on the tensor cores against fp64, at the sizes where a tile, a chunk of the sum, a slice
of the rows or a vector load runs out; infinities and NaN; without scratch."""
import pytest
import torch

from paper_2104_06700_b200 import binding
from test_gpu_layer import empty_graph

pytestmark = pytest.mark.gpu
DEV = "cuda"
EPS = 2.0 ** -24


def bound(depth, slices, magnitude):
    """Per chunk of 32 products: 12 tensor-core additions, each off by at most 2 EPS of the partial sum, and 4 EPS of what
    the split leaves out; then an fp32 addition per chunk and per slice."""
    return (28 + (depth + 31) // 32 + slices) * EPS * magnitude


def operands(n, K, N, offset=0):
    gen = torch.Generator(device=DEV).manual_seed(n + 7 * K + 31 * N)

    def matrix(r, c):  # `offset` floats behind a 16-byte boundary
        return torch.randn(r * c + offset, device=DEV, generator=gen)[offset:].view(r, c)

    return matrix(n, K), matrix(N, K), matrix(n, N), torch.rand(n, 1, device=DEV, generator=gen), matrix(1, N)[0]


def check(n, K, N, offset=0, scratch=True):
    X, W, G, scale, bias = operands(n, K, N, offset)
    g = empty_graph(n)
    if not scratch:
        g.dg_graph_set_param("scratch_mb", 0)
    Xd, Wd, Gd = X.double(), W.double(), G.double()
    want, size = Xd @ Wd.t(), Xd.abs() @ Wd.abs().t()
    assert bool(((g.dg_linear_fwd(X, W).double() - want).abs() <= bound(K, 1, size)).all())
    want = (want * scale.double() + bias.double()).relu()
    limit = bound(K, 1, size) * scale.double() + EPS * (size * scale.double() + bias.double().abs())
    assert bool(((g.dg_linear_fwd(X, W, scale, bias, True).double() - want).abs() <= limit).all())
    dX = g.dg_linear_bwd_input(G, W).double()
    assert bool(((dX - Gd @ Wd).abs() <= bound(N, 1, Gd.abs() @ Wd.abs())).all())
    dW = g.dg_linear_bwd_weight(G, X)
    assert bool(((dW.double() - Gd.t() @ Xd).abs() <= bound(n, 148, Gd.abs().t() @ Xd.abs())).all())
    assert torch.equal(dW, g.dg_linear_bwd_weight(G, X))


@pytest.mark.parametrize("n,K,N", [(1, 1, 1), (127, 31, 15), (128, 32, 16), (129, 33, 17), (513, 64, 47), (300, 100, 127),
                                   (640, 128, 128), (257, 129, 129), (1000, 255, 255), (511, 256, 256), (512, 257, 257),
                                   (700, 602, 41), (150, 41, 602), (40000, 100, 256)])
def test_products_match_fp64(n, K, N):
    check(n, K, N)


@pytest.mark.parametrize("offset", [1, 2])
@pytest.mark.parametrize("n,K,N", [(200, 64, 64), (130, 36, 260)])
def test_misaligned_matrices(n, K, N, offset):
    check(n, K, N, offset)


@pytest.mark.parametrize("n,K,N", [(129, 33, 17), (1500, 260, 130)])
def test_products_without_scratch(n, K, N):
    check(n, K, N, scratch=False)


def same_as_torch(got, want):
    """Where torch's result is infinite or NaN, the same; finite elsewhere."""
    finite = want.isfinite()
    assert torch.equal(got.isfinite(), finite)
    assert torch.equal(got[~finite].nan_to_num(9.0), want[~finite].nan_to_num(9.0))


# several tiles a block, a part-filled one among them, one and two passes of 128 columns
@pytest.mark.parametrize("n,K,N", [(20000, 100, 256), (20011, 260, 300), (20011, 256, 47)])
@pytest.mark.parametrize("kind", ["some", "all"])
def test_infinities_and_nan_in_many_tiles(n, K, N, kind):
    X, W, G, scale, bias = operands(n, K, N)
    if kind == "all":
        X.fill_(float("nan"))
        G[:, 3] = float("nan")
    else:
        X[n // 2:n // 2 + 200], X[n - 1, 0], X[3, K - 1] = float("nan"), float("inf"), -float("inf")
        G[5, N - 1], W[7, 7] = float("inf"), float("-inf")
    g = empty_graph(n)
    same_as_torch(g.dg_linear_fwd(X, W), X @ W.t())
    same_as_torch(g.dg_linear_fwd(X, W, scale, bias, True), (X @ W.t() * scale + bias).relu())
    same_as_torch(g.dg_linear_bwd_input(G, W), G @ W)
    same_as_torch(g.dg_linear_bwd_weight(G, X), G.t() @ X)


def test_sums_that_overflow():
    """Finite where the sum of the absolute products is, whatever the order."""
    X, W, G, scale, bias = operands(2000, 100, 60)
    X, W = X * 2.0 ** 62, W * 2.0 ** 60
    want, size = X.double() @ W.double().t(), X.double().abs() @ W.double().abs().t()
    fits = size < 3.0e38
    assert 0.05 < float(fits.double().mean()) < 0.5
    got = empty_graph(2000).dg_linear_fwd(X, W).double()
    assert bool(((got - want).abs() <= bound(100, 1, size))[fits].all())


def test_nan_costs_no_more_than_plain_arithmetic():
    """A diverged model's epochs end.  The factor is 3 to 8; an element at a time it was over 100."""
    n = 20000
    X, W, G, scale, bias = operands(n, 256, 256)
    g = empty_graph(n)
    nan = torch.full_like(X, float("nan"))

    def time(call):
        best = float("inf")
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            call()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    for call in (lambda x: g.dg_linear_fwd(x, W), lambda x: g.dg_linear_bwd_input(x, W),
                 lambda x: g.dg_linear_bwd_weight(x, x)):
        assert time(lambda: call(nan)) < 40 * time(lambda: call(X))


@pytest.mark.parametrize("limit", [1, 2])
def test_a_scratch_limit_costs_slices_and_not_all_of_them(limit):
    n, K, N = 40000, 256, 100  # 37 slices of 100 KiB
    X, W, G, scale, bias = operands(n, K, N)
    g = empty_graph(n)
    g.dg_graph_set_param("scratch_mb", limit)
    g.dg_linear_bwd_weight(G, X)
    before = binding.dg_kernel_launch_count()
    dW = g.dg_linear_bwd_weight(G, X)
    assert binding.dg_kernel_launch_count() - before == 2  # the products and the sum of the slices
    want, size = G.double().t() @ X.double(), G.double().abs().t() @ X.double().abs()
    assert bool(((dW.double() - want).abs() <= bound(n, 148, size)).all())


def test_infinities_and_nan():
    """As torch's GEMM, element for element."""
    X, W, G, scale, bias = operands(700, 70, 50)
    X[3, 5], X[200, 0], X[400, 69], X[500, 1] = float("inf"), float("nan"), -float("inf"), 3.3e38
    W[7, 7] = float("inf")
    g = empty_graph(700)
    for got, want in ((g.dg_linear_fwd(X, W), X @ W.t()), (g.dg_linear_bwd_input(G, W), G @ W),
                      (g.dg_linear_bwd_weight(G, X), G.t() @ X),
                      (g.dg_linear_fwd(X, W, scale, bias, True), (X @ W.t() * scale + bias).relu())):
        finite = want.isfinite()
        assert torch.equal(got.isfinite(), finite)
        assert torch.equal(got[~finite].nan_to_num(9.0), want[~finite].nan_to_num(9.0))


def test_no_wait_ran_out():
    g = empty_graph(3000)
    X, W, G, scale, bias = operands(3000, 300, 300)
    g.dg_linear_fwd(X, W)
    g.dg_linear_bwd_input(G, W)
    g.dg_linear_bwd_weight(G, X)
    assert g.dg_graph_get_param("expired_waits") == 0
    with pytest.raises(binding.DgError):
        g.dg_graph_set_param("expired_waits", 0)


def test_arguments_are_checked():
    X, W, G, scale, bias = operands(40, 8, 8)
    g = empty_graph(40)
    with pytest.raises(ValueError):
        g.dg_linear_fwd(X[1:], W)
    with pytest.raises(ValueError):
        g.dg_linear_bwd_weight(G[:, :4].contiguous(), X[1:])
    wide = torch.zeros(40, 12, device=DEV)  # holds enough values for every operand
    for call in (lambda: g.dg_linear_fwd(wide, W), lambda: g.dg_linear_fwd(X.view(8, 40), W),
                 lambda: g.dg_linear_fwd(X, W, bias=wide[0]), lambda: g.dg_linear_fwd(X, W, scale.repeat(2, 1)),
                 lambda: g.dg_linear_bwd_input(wide, W), lambda: g.dg_linear_bwd_weight(torch.zeros(41, 8, device=DEV), X)):
        with pytest.raises(ValueError):
            call()
    lib = binding.lib()
    assert lib.dg_linear_fwd(g._h, X.data_ptr(), 8, W.data_ptr(), 8, None, None, 0, X.data_ptr() + 16, None) \
        == binding.DG_ERR_INVALID_ARG
    assert lib.dg_linear_bwd_input(g._h, None, 8, W.data_ptr(), 8, X.data_ptr(), None) == binding.DG_ERR_INVALID_ARG
