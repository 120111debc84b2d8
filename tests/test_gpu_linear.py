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
    """Per chunk of 32 products: two tensor-core additions of products of the first parts and ten of 2^-8 of those and less,
    each off by at most 2 EPS of the partial sum, and EPS of what the split leaves out: 5.2 EPS; then an fp32 addition per
    chunk and per slice of the sum."""
    return (6 + (depth + 31) // 32 + slices) * EPS * magnitude


def slices_of(n, K, N):
    """(slices of the rows that the weights' gradient is summed in, their length)"""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slices = max(1, min(sms // ((N + 127) // 128 * ((K + 127) // 128)), (n + 511) // 512))
    return slices, -(-n // slices)


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
    slices, length = slices_of(n, K, N) if scratch else (1, n)
    assert bool(((dW.double() - Gd.t() @ Xd).abs() <= bound(length, slices, Gd.abs().t() @ Xd.abs())).all())
    assert torch.equal(dW, g.dg_linear_bwd_weight(G, X))


@pytest.mark.parametrize("n,K,N", [(1, 1, 1), (127, 31, 15), (128, 32, 16), (129, 33, 17), (513, 64, 47), (300, 100, 127),
                                   (640, 128, 128), (257, 129, 129), (1000, 255, 255), (511, 256, 256), (512, 257, 257),
                                   (700, 602, 41), (150, 41, 602), (40000, 100, 256),
                                   # blocks with several tiles: of two widths, of rows that leave as one stretch
                                   (20011, 64, 257), (20011, 300, 300), (40000, 256, 47), (40100, 41, 41), (20011, 48, 45)])
def test_products_match_fp64(n, K, N):
    check(n, K, N)


@pytest.mark.parametrize("offset", [1, 2])
@pytest.mark.parametrize("n,K,N", [(200, 64, 64), (130, 36, 260)])
def test_misaligned_matrices(n, K, N, offset):
    check(n, K, N, offset)


@pytest.mark.parametrize("n,K,N", [(129, 33, 17), (1500, 260, 130), (20011, 64, 257), (40000, 100, 47)])
def test_products_without_scratch(n, K, N):
    check(n, K, N, scratch=False)


def without_one(X, W, p, q):
    """X W^T less the products of X's part p and W's part q."""
    def part(x, which):
        for t in range(which + 1):
            piece = x.to(torch.bfloat16).float()
            x = (x - piece) * 256
        return piece.double() * 2.0 ** (-8 * which)

    return X.double() @ W.double().t() - part(X, p) @ part(W, q).t()


@pytest.mark.parametrize("nonzeros", [1, 2, 3, 16, 256])
def test_rows_of_few_numbers(nonzeros):
    """Their sums have no other rounding errors to hide a product that is left out."""
    n, K, N = 2000, 256, 256
    X, W, G, scale, bias = operands(n, K, N)
    G = G.contiguous()
    X = X * torch.zeros_like(X).scatter_(1, torch.rand_like(X).topk(nonzeros, 1).indices, 1.0)
    G = G * (X != 0)
    g = empty_graph(n)
    chunks = min(nonzeros, 8)
    for A, B, got in ((X, W, g.dg_linear_fwd(X, W)), (G, W.t().contiguous(), g.dg_linear_bwd_input(G, W))):
        want, size = A.double() @ B.double().t(), A.double().abs() @ B.double().abs().t()
        limit = (6 + chunks) * EPS * size
        assert bool(((got.double() - want).abs() <= limit).all())
        for p, q in ((0, 0), (0, 1), (1, 0), (1, 1), (0, 2), (2, 0)):  # the limit tells each of the six products
            assert nonzeros > 16 or bool(((without_one(A, B, p, q) - want).abs() > limit).any())
    dW, want, size = g.dg_linear_bwd_weight(G, X), G.double().t() @ X.double(), G.double().abs().t() @ X.double().abs()
    slices, length = slices_of(n, K, N)
    assert bool(((dW.double() - want).abs() <= bound(length, slices, size)).all())


def norm_error(got, want):
    return float((got.double() - want).norm() / want.norm())


@pytest.mark.parametrize("kind", ["normal", "one sign"] + [f"2^{e}" for e in (-100, -115, -122, -126)])
def test_errors_are_below_those_of_fp32_sums(kind):
    """2-norms against those of torch's fp32 products, in sums of 256 and of 20000; half of them at least where numbers have
    both signs.  Small operands against large ones: bf16 parts of fp32's smallest numbers."""
    n, K, N = 20000, 256, 256
    X, W, G, scale, bias = operands(n, K, N)
    if kind == "one sign":
        X, W, G = X.abs(), W.abs(), G.abs()
    elif kind != "normal":
        X = X * 2.0 ** int(kind[2:])
        G, W = G * 2.0 ** 60, W * 2.0 ** 60
    g = empty_graph(n)
    part = 1.0 if kind == "one sign" else 0.5
    for got, fp32, want in ((g.dg_linear_fwd(X, W), X @ W.t(), X.double() @ W.double().t()),
                            (g.dg_linear_bwd_input(G, W), G @ W, G.double() @ W.double()),
                            (g.dg_linear_bwd_weight(G, X), G.t() @ X, G.double().t() @ X.double())):
        assert norm_error(got, want) <= part * norm_error(fp32, want)


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
    slices = limit * 2 ** 20 // (K * N * 4)
    assert bool(((dW.double() - want).abs() <= bound(-(-n // slices), slices, size)).all())


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
