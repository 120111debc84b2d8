"""Where the rows are shared out in chunks, long rows are cut, matrices are copied into padded rows, and
the gradient of max / min goes through a bit mask: the sizes at which each of these changes its path,
against the CPU oracle element by element, with the bounds of the other parity tests."""
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2104_06700_b200 import binding, synth
from parity_util import assert_within_bound, check_fwd_bwd, check_transpose, to_np
from test_gpu_general import run_case

pytestmark = pytest.mark.gpu
DEV = "cuda"
OPS = (binding.DG_OP_SUM, binding.DG_OP_MEAN)


def graph_of(lengths, n, seed, weighted=False):
    """CSR with the given row lengths (the other rows are empty), random sorted sources."""
    rng = np.random.default_rng(seed)
    deg = np.zeros(n, dtype=np.int64)
    deg[: len(lengths)] = lengths
    rowptr = np.concatenate([[0], np.cumsum(deg)])
    cols = np.concatenate([np.sort(rng.integers(0, n, d)) for d in deg if d > 0] or [[]]).astype(np.int32)
    w = rng.random(cols.size).astype(np.float32) if weighted else None
    return synth.SynthGraph("rows", n, int(cols.size), 0, torch.as_tensor(rowptr, device=DEV),
                            torch.as_tensor(cols, device=DEV),
                            None if w is None else torch.as_tensor(w, device=DEV))


def host(sg):
    return to_np(sg.rowptr), to_np(sg.colidx), to_np(sg.edge_w)


def handle(sg, self_loops=0):
    g = binding.dg_graph_create(sg.n, sg.nnz, sg.rowptr, sg.colidx, sg.edge_w)
    g.dg_graph_set_param("self_loops", self_loops)
    return g


# lengths around one and several pieces of the smallest chunks (32 entries) and their cut threshold, with
# runs of empty rows between them; the last graph is one row
EDGES = [
    [1, 0, 0, 31, 32, 33, 0, 63, 64, 65, 159, 160, 161, 0, 0, 191, 192, 193, 1023, 1024, 1025, 5000],
    [0] * 300 + [70000] + [0] * 40 + [2] * 100 + [161] * 3,
    [3] * 2000 + [97, 4097],
    [2500],
]


@pytest.mark.parametrize("lengths", EDGES, ids=["edges", "star", "short", "one"])
@pytest.mark.parametrize("F", [1, 8, 47, 130, 260])
@pytest.mark.parametrize("self_loops", [0, 1])
def test_cut_rows(lengths, F, self_loops):
    sg = graph_of(lengths, len(lengths) + 70, F, weighted=F == 47)
    g = handle(sg, self_loops)
    csc = check_transpose(g, *host(sg))
    H, G = synth.features(sg.n, F, 1, DEV, nonneg=True), synth.features(sg.n, F, 2, DEV)
    for op in OPS:
        check_fwd_bwd(g, host(sg), H, G, op, csc, self_loops=bool(self_loops))
        assert torch.equal(g.dg_aggregate_fwd(H, op), g.dg_aggregate_fwd(H, op))


@pytest.mark.parametrize("lengths", EDGES, ids=["edges", "star", "short", "one"])
@pytest.mark.parametrize("F", [1, 32, 47, 130])
def test_calls_without_scratch(lengths, F):
    """"scratch_mb" = 0: the later pieces of cut rows are added by a kernel of their own, in either direction, for
    every operator pair, with weights, own rows and bf16 storage."""
    sg = graph_of(lengths, len(lengths) + 70, F, weighted=F == 47)
    H, G = synth.features(sg.n, F, 1, DEV, nonneg=True), synth.features(sg.n, F, 2, DEV)
    for self_loops in (0, 1):
        g = handle(sg, self_loops)
        g.dg_graph_set_param("scratch_mb", 0)
        csc = check_transpose(g, *host(sg))
        for op in OPS:
            check_fwd_bwd(g, host(sg), H, G, op, csc, self_loops=bool(self_loops))
            if F % 2 == 0:
                Hb, plain = H.to(torch.bfloat16), handle(sg, self_loops)
                got, want = g.dg_aggregate_fwd_bf16(Hb, op), plain.dg_aggregate_fwd_bf16(Hb, op)
                # non-negative terms: two orders of the same sum differ by at most twice its own bound
                assert bool(((got - want).abs() <= 2e-5 * want + 2e-7).all())
    for binary, cols, reduce in ((0, 1, 1), (1, F, 0), (2, 1, 2), (3, F, 1), (4, 1, 0), (4, F, 0), (5, 1, 1), (5, F, 2)):
        run_case(sg, F, cols, binary, reduce, seed=F, tie_heavy=binary != 5, params={"scratch_mb": 0})


def check_hub_of_equal_terms(params, F=64):
    """A row of 4 M equal terms, whose partial sums round the same way: one chain over its 40 thousand pieces is off by
    4e-5 of the sum.  The chains there are: 48 additions of a lane group, the groups, 32 slots, 170 totals of a warp, 8
    warps; fewer than 265, each off by at most 2^-24 of the sum."""
    n, hub = 1000, 4000000
    rowptr = torch.arange(n + 1, device=DEV)
    rowptr[8:] += hub - 1
    nnz = int(rowptr[-1])
    colidx = torch.arange(nnz, device=DEV).remainder(n).int()
    g = binding.dg_graph_create(n, nnz, rowptr, colidx, None)
    for name, value in params.items():
        g.dg_graph_set_param(name, value)
    for x in (0.1, 0.3, 0.9):
        H = torch.full((n, F), x, device=DEV)
        want = float(H[0, 0].double()) * hub
        for got in (g.dg_aggregate_fwd(H, binding.DG_OP_SUM),
                    g.dg_ap_fwd(H, torch.zeros(nnz, 1, device=DEV), binding.DG_BIN_ADD, binding.DG_RED_SUM)[0]):
            assert float((got[7].double() - want).abs().max()) <= 265 * 2.0 ** -24 * want


@pytest.mark.parametrize("params", [{}, {"scratch_mb": 0}], ids=["slots", "pieces"])
def test_pieces_of_a_hub_are_not_one_chain(params):
    check_hub_of_equal_terms(params)


def test_a_hub_is_cut_whatever_the_threshold():
    check_hub_of_equal_terms({"heavy_threshold": 1 << 30})


def test_cut_rows_of_larger_chunks():
    """1.6 M edges: chunks of 64 entries, rows over 128 are cut."""
    rng = np.random.default_rng(3)
    lengths = list(rng.integers(0, 200, 15000)) + [127, 128, 129, 90000]
    sg = graph_of(lengths, len(lengths) + 5, 1)
    g = handle(sg)
    csc = check_transpose(g, *host(sg))
    H, G = synth.features(sg.n, 36, 1, DEV), synth.features(sg.n, 36, 2, DEV)
    for op in OPS:
        check_fwd_bwd(g, host(sg), H, G, op, csc)


@pytest.mark.parametrize("F,shift", [(41, 0), (42, 0), (130, 0), (602, 0), (128, 1), (64, 2)])
@pytest.mark.parametrize("degree", [20, 70])
def test_padded_copies(F, shift, degree):
    """Mean degree 20: odd widths, and matrices that start 4 or 8 bytes off, are gathered from a padded
    copy; 70: the mean's backward pass divides the rows in the copy, and source blocks apply."""
    n = max(4200, (1 << 24) // (F * degree) + 1)
    rng = np.random.default_rng(F)
    sg = graph_of(rng.integers(degree - 10, degree + 14, n), n, F)
    assert sg.nnz >= degree * sg.n and sg.nnz * F >= 1 << 24
    for self_loops in (0, 1):
        g = handle(sg, self_loops)
        csc = check_transpose(g, *host(sg))
        rows = np.arange(0, sg.n, 7)
        buf = [synth.features(sg.n * F + 4, 1, 9 + i, DEV).flatten() for i in range(2)]
        H, G = (b[shift:shift + sg.n * F].view(sg.n, F) for b in buf)
        for op in OPS:
            check_fwd_bwd(g, host(sg), H, G, op, csc, rows=rows, self_loops=bool(self_loops))
        out = torch.zeros(sg.n * F + 4, device=DEV)  # an output that takes no vector stores
        got = g.dg_aggregate_fwd(H, binding.DG_OP_SUM, out=out[1:1 + sg.n * F].view(sg.n, F))
        torch.cuda.synchronize()
        ref, mag = oracle.ap_forward(*host(sg), to_np(H), binding.DG_OP_SUM, rows=rows,
                                     self_loops=bool(self_loops))
        assert_within_bound(to_np(got)[rows], ref, mag, "fwd into an unaligned output")
        assert float(out[0]) == 0.0 and float(out[1 + sg.n * F:].abs().max()) == 0.0
    dW = g.dg_aggregate_edge_grad(H, G, binding.DG_OP_SUM)
    torch.cuda.synchronize()
    ref, mag = oracle.edge_weight_grad(*host(sg)[:2], to_np(H), to_np(G), oracle.OP_SUM)
    assert_within_bound(to_np(dW), ref, mag, "dW")


@pytest.mark.parametrize("F", [1, 7, 16, 17, 32, 33, 96, 129, 256, 257, 300])
def test_extremum_gradient_mask(F):
    """One word per 32 features, up to eight at a time; rows of several windows and cut rows; ties."""
    sg = graph_of([5, 0, 33, 300, 1025, 2600, 0, 64] + [9] * 200, 230, F)
    for binary, cols in ((0, 1), (4, 1), (4, F), (5, F), (2, F)):
        run_case(sg, F, cols, binary, binding.DG_RED_MAX if F % 2 else binding.DG_RED_MIN, seed=F,
                 tie_heavy=binary != 5)


@pytest.mark.parametrize("F", [1, 8, 9, 16, 17, 33, 129, 300])
@pytest.mark.parametrize("degree", [9, 30, 70])
def test_extremum_gradient_on_both_sides_of_its_rule(F, degree):
    """The mask from 2^17 edges on, except for 9 to 16 features on longer rows; fewer edges compare arg (above)."""
    sg = graph_of([5, 0, 33, 300, 1025, 2600, 0, 64] + [degree] * (270000 // degree), 270000 // degree + 20, F)
    assert sg.nnz >= 1 << 17
    for binary, cols in ((0, 1), (4, 1)):
        run_case(sg, F, cols, binary, binding.DG_RED_MAX if F % 2 else binding.DG_RED_MIN, seed=F, tie_heavy=True)


@pytest.mark.parametrize("nnz", [1, 3, 4, 5, 7, 8, 9, 4095, 4096, 4097, 12289])
def test_csc_and_weight_refresh_remainders(nnz):
    """Four edges a thread in the refresh of the weights, eight in the column pointers, tiles of 4096."""
    sg = graph_of([nnz // 3, 0, nnz - nnz // 3], 40, nnz, weighted=True)
    g = handle(sg)
    check_transpose(g, *host(sg))
    sg.edge_w.mul_(0.5).add_(1.0)
    g.dg_graph_update_weights()
    torch.cuda.synchronize()
    _, _, w_T, perm = g.dg_graph_get_csc()
    assert torch.equal(w_T, sg.edge_w[perm.long()])
    G = synth.features(sg.n, 5, 3, DEV)
    csc = oracle.transpose(*host(sg))[:3]
    check_fwd_bwd(g, host(sg), G, G, binding.DG_OP_MEAN, csc)


@pytest.mark.parametrize("F", [8, 130])
def test_self_calls_are_the_attribute_for_one_call(F):
    """dg_aggregate_fwd_self / _bwd_self on a plain handle give what a handle with self_loops = 1 gives."""
    sg = graph_of(EDGES[0], 100, 5)
    plain, looped = handle(sg), handle(sg, 1)
    plain.dg_graph_transpose()
    looped.dg_graph_transpose()
    H = synth.features(sg.n, F, 1, DEV)
    for op in OPS:
        assert torch.equal(plain.dg_aggregate_fwd_self(H, op), looped.dg_aggregate_fwd(H, op))
    assert torch.equal(plain.dg_aggregate_bwd_self(H, binding.DG_OP_SUM),
                       looped.dg_aggregate_bwd(H, binding.DG_OP_SUM))
    with pytest.raises(binding.DgError) as e:
        plain.dg_aggregate_bwd_self(H, binding.DG_OP_MEAN)  # the factors were made without the loops
    assert e.value.status == binding.DG_ERR_NOT_TRANSPOSED
    assert torch.equal(looped.dg_aggregate_bwd_self(H, binding.DG_OP_MEAN),
                       looped.dg_aggregate_bwd(H, binding.DG_OP_MEAN))


@pytest.mark.parametrize("F", [8, 16])
def test_positions_up_to_the_last(F):
    """2^31 - 1 edges, the most a handle takes: a batch that starts in the last 32 positions ends beyond 2^31.  Rows
    of 2048 consecutive ids, so that every result has a closed form, and integer features, so that sums are exact.
    The wider matrix exceeds the L2 budget and takes the source-blocked kernels."""
    torch.cuda.empty_cache()
    n, deg, blocks = 1 << 20, 2048, 512
    nnz = n * deg - 1
    rowptr = (torch.arange(n + 1, device=DEV) * deg).clamp_(max=nnz)
    colidx = torch.arange(n, dtype=torch.int32, device=DEV).repeat(deg)[:nnz]
    g = binding.dg_graph_create(n, nnz, rowptr, colidx, None)
    g.dg_graph_transpose()
    _, rowidx_T, _, perm = g.dg_graph_get_csc()
    u = torch.arange(n, device=DEV)
    for lo in range(0, n, 1 << 15):  # column u: the rows congruent to u / 2048 modulo 512, in order
        cols = u[lo:lo + (1 << 15)].unsqueeze(1)
        rows = (cols // deg + blocks * torch.arange(deg, device=DEV)).flatten()[: nnz - lo * deg]
        at = slice(lo * deg, lo * deg + rows.numel())
        assert torch.equal(rowidx_T[at].long(), rows)
        assert torch.equal(perm[at].long(), rows * deg + (cols % deg).expand(-1, deg).flatten()[: rows.numel()])
    del rowidx_T, perm

    H = (u.unsqueeze(1) * 5 % 7 + torch.arange(F, device=DEV)).float()
    G = (u.unsqueeze(1) * 3 % 11 - torch.arange(F, device=DEV)).float()
    want = H.view(blocks, deg, F).sum(1).repeat(deg, 1)
    want[-1] -= H[-1]
    assert torch.equal(g.dg_aggregate_fwd(H, binding.DG_OP_SUM), want)
    want = G.view(deg, blocks, F).sum(0).repeat_interleave(deg, 0)
    want[-1] -= G[-1]
    assert torch.equal(g.dg_aggregate_bwd(G, binding.DG_OP_SUM), want)

    # the maximum of a block lies at its last id (which the last row does not have) for even features
    H[:, ::2] = (u % deg).float().unsqueeze(1)
    H[:, 1::2] = -H[:, ::2]
    fO, arg = g.dg_ap_fwd(H, None, binding.DG_BIN_COPY_LHS, binding.DG_RED_MAX)
    best = torch.tensor([deg - 1, 0] * (F // 2), device=DEV).repeat(n, 1)
    best[-1, ::2] = deg - 2
    assert torch.equal(arg.long(), u.unsqueeze(1) * deg + best)
    assert torch.equal(fO, best.float())
    dV, _ = g.dg_ap_bwd(G, H, None, binding.DG_BIN_COPY_LHS, binding.DG_RED_MAX, arg=arg)
    want = torch.zeros(n, F, device=DEV)
    sums = G.view(deg, blocks, F).sum(0)
    want.view(blocks, deg, F)[:, -1, ::2] = sums[:, ::2]
    want.view(blocks, deg, F)[:, 0, 1::2] = sums[:, 1::2]
    want[-1, ::2] -= G[-1, ::2]
    want[-2, ::2] = G[-1, ::2]
    assert torch.equal(dV, want)
    del fO, arg, dV, want, best

    H = (u.unsqueeze(1) * 5 % 7 + torch.arange(F, device=DEV)).float()
    fE = torch.ones(nnz, 1, device=DEV)
    for name, call in (("dot", lambda: g.dg_aggregate_edge_grad(H, G, binding.DG_OP_SUM)),
                       ("add", lambda: g.dg_ap_bwd(G, H, fE, binding.DG_BIN_ADD, binding.DG_RED_SUM)[1])):
        got = call().flatten()
        for lo in (0, n - 1024):
            X = H.view(blocks, deg, F)[u[lo:lo + 1024] % blocks] if name == "dot" else torch.ones(1024, deg, F, device=DEV)
            want = (X * G[lo:lo + 1024].unsqueeze(1)).sum(2).flatten()
            at = got[lo * deg:(lo + 1024) * deg]
            assert torch.equal(at, want[: at.numel()]), name
    del g, colidx
    torch.cuda.empty_cache()


def test_calls_on_two_streams():
    """Scratch comes from a pool shared by handles and streams; each call's is its own."""
    sg = graph_of(EDGES[0] * 40, 1000, 7)
    G = synth.features(sg.n, 47, 3, DEV)
    g = handle(sg)
    g.dg_graph_transpose()
    want = g.dg_aggregate_bwd(G, binding.DG_OP_MEAN).clone()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = []
    for i in range(20):
        with torch.cuda.stream(streams[i % 2]):
            got.append(g.dg_aggregate_bwd(G, binding.DG_OP_MEAN))
    torch.cuda.synchronize()
    assert all(torch.equal(x, want) for x in got)


def test_a_destroyed_handle_keeps_its_memory_until_its_kernels_are_done():
    """The short-lived handle works on a non-blocking stream behind a long queue and is destroyed at once; the plans of
    handles made meanwhile by other threads would take its place."""
    sg = graph_of(EDGES[0] * 40, 1000, 7)
    other = graph_of([200] * 150, 1000, 8)
    G = synth.features(sg.n, 47, 3, DEV)
    keep = handle(sg)
    keep.dg_graph_transpose()
    want = keep.dg_aggregate_bwd(G, binding.DG_OP_MEAN)
    torch.cuda.synchronize()
    busy = torch.randn(4096, 4096, device=DEV)
    side = torch.cuda.Stream()
    failed = []

    def make_handles():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(15):
                    g = handle(other)
                    g.dg_graph_transpose()
                    g.dg_aggregate_bwd(G, binding.DG_OP_SUM)
        except Exception as e:  # an assertion in a thread is not the test's
            failed.append(e)

    threads = [threading.Thread(target=make_handles) for _ in range(2)]
    for t in threads:
        t.start()
    got = []
    for _ in range(10):
        h = handle(sg)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            h.dg_graph_transpose()
            for _ in range(10):
                busy = busy @ busy * 1e-3
            got.append(h.dg_aggregate_bwd(G, binding.DG_OP_MEAN))
        h.dg_graph_destroy()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed and all(torch.equal(x, want) for x in got)
