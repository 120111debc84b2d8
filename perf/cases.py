"""Timed cases of the aggregation primitive: what full-batch GraphSAGE training asks of libdgagg.

A case is a dict of plain values.  ``kind`` says which public calls one pass makes:

  step      dg_aggregate_fwd and dg_aggregate_bwd (or the bf16 pair): one layer's aggregation in
            training, forward and backward
  ingest    dg_graph_create and dg_graph_transpose: what every new graph costs before its first step
  extremum  dg_ap_fwd with max / min and arg indices, then the gradient dV: the max-pooling aggregator
  edges     dg_ap_fwd with an |E| x F edge-feature matrix and sum, then both gradients
  weights   a training step of learnable scalar edge weights: forward, backward, the weights'
            gradient, an SGD update in place and dg_graph_update_weights
  epoch     one full-batch GraphSAGE epoch (graphsage.make_epoch): aggregations, Linear layers,
            loss, backward pass, Adam

``graph`` and ``scale`` name a generator of synth.py and its size (``n`` and ``nnz`` for the tiny
graph); ``F`` is the feature width.  Graphs, features and weights are drawn from the seed alone.
"""
from __future__ import annotations

import math

import torch

from paper_2104_06700_b200 import binding, graphsage, synth

OPS = {"sum": binding.DG_OP_SUM, "mean": binding.DG_OP_MEAN}
BINARIES = {"add": binding.DG_BIN_ADD, "sub": binding.DG_BIN_SUB, "mul": binding.DG_BIN_MUL}
REDUCERS = {"max": binding.DG_RED_MAX, "min": binding.DG_RED_MIN}

# widths the repository's configurations name: input features, hidden sizes, class counts
WIDTHS = [8, 16, 41, 47, 64, 100, 128, 172, 256, 602]
CLASSES = {"reddit_like": 41, "products_like": 47, "papers_like": 172}
LR = 1e-4  # of the edge weights' SGD update


def step(name, graph, scale, F, op="sum", dtype="f32", weighted=False, self_loops=False):
    return {"name": name, "kind": "step", "graph": graph, "scale": scale, "F": F, "op": op,
            "dtype": dtype, "weighted": weighted, "self_loops": self_loops}


def listed():
    tiny = {"graph": "tiny", "n": 4096, "nnz": 65536}
    return [
        # the smallest calls: a graph that fits a fraction of the chip, where launches and the host count
        {**step("tiny step", "tiny", 1.0, 64, "mean", weighted=True), **tiny},
        # a small graph at an odd class-count width (4-byte loads)
        step("small step", "products_like", 0.01, 47, "sum"),
        # the headline: dense-ish community graph at its input width
        step("reddit step", "reddit_like", 1.0, 602, "mean"),
        # the same width stored as bf16 (rows of 1204 bytes)
        step("reddit bf16 step", "reddit_like", 0.25, 602, "mean", dtype="bf16"),
        # sparse power-law graph whose features exceed the L2 many times
        step("products step", "products_like", 1.0, 100, "mean"),
        # narrow features, one scalar weight per edge: index and weight streams dominate
        step("proteins step", "proteins_like", 1.0, 8, "sum", weighted=True),
        # the largest matrices: citation-like graph with few edges per vertex, the GCN aggregator
        step("papers step", "papers_like", 0.05, 128, "mean", self_loops=True),
        # a new graph: CSR check, heavy lists, CSR -> CSC
        {"name": "products ingest", "kind": "ingest", "graph": "products_like", "scale": 1.0,
         "F": 1, "weighted": False, "self_loops": False},
        # max-pooling aggregator, forward and backward
        {"name": "products max", "kind": "extremum", "graph": "products_like", "scale": 0.25,
         "F": 100, "reduce": "max", "weighted": False, "self_loops": False},
        # full edge features: the |E| x F streams dominate
        {"name": "proteins edge features", "kind": "edges", "graph": "proteins_like", "scale": 0.1,
         "F": 64, "binary": "mul", "weighted": False, "self_loops": False},
        # learnable scalar edge weights
        {"name": "proteins weights", "kind": "weights", "graph": "proteins_like", "scale": 0.5,
         "F": 64, "op": "sum", "weighted": True, "self_loops": False},
        # the composite workload: 3 layers, hidden 256
        {"name": "products epoch", "kind": "epoch", "graph": "products_like", "scale": 0.1, "F": 100,
         "hidden": 256, "layers": 3, "project_first": False, "fused": False, "bf16": False,
         "weighted": False, "self_loops": False},
    ]


# ---- sizes and costs -------------------------------------------------------------------------

def sizes(case):
    """(vertices, edges) of the case's graph, by the generators' own rules."""
    if case["graph"] == "tiny":
        return case["n"], case["nnz"]
    n0, nnz0, _ = synth.CONFIG_SHAPES[case["graph"]]
    dense = case["graph"] in ("reddit_like", "proteins_like")
    n = max(64, int(round(n0 * (math.sqrt(case["scale"]) if dense else case["scale"]))))
    if case["graph"] == "papers_like":
        return n, max(64, int(round(nnz0 * case["scale"])))
    return n, 2 * max(64, int(round(nnz0 * case["scale"])) // 2)


def dims(case):
    """Layer widths of the epoch's model."""
    return [case["F"]] + [case["hidden"]] * (case["layers"] - 1) + [CLASSES[case["graph"]]]


def work(case):
    n, nnz = sizes(case)
    F, kind = case["F"], case["kind"]
    ptr, idx, mat = 8.0 * (n + 1), 4.0 * nnz, 4.0 * n * F
    w = idx if case["weighted"] else 0.0
    if kind == "step":  # pointers, indices, weights, the gathered matrix once, the result once; twice
        gathered = mat / 2 if case["dtype"] == "bf16" else mat
        return {"bytes": 2 * (ptr + idx + w + gathered + mat),
                "flops": 2.0 * nnz * F * (2 if case["weighted"] else 1)}
    if kind == "ingest":  # CSR in; colptr, row ids, permutation (and weights) out
        return {"bytes": 2 * ptr + 3 * idx + 2 * w, "flops": 0.0}
    if kind == "extremum":  # forward: fO and arg out; backward: dO and arg in, CSC with its permutation
        return {"bytes": (ptr + idx + 3 * mat) + (ptr + 2 * idx + 3 * mat), "flops": 2.0 * nnz * F}
    if kind == "edges":  # fE read by the forward pass and by dV (mul), dE written
        fE = 4.0 * nnz * F
        reads = 2 if case["binary"] == "mul" else 1
        return {"bytes": (ptr + idx + 2 * mat) + (ptr + 2 * idx + 2 * mat) + (ptr + idx + 2 * mat)
                + (reads + 1) * fE, "flops": 5.0 * nnz * F}
    if kind == "weights":  # forward, backward, dW, the update of w, the refreshed copy
        return {"bytes": 2 * (ptr + 2 * idx + 2 * mat) + (ptr + 2 * idx + 2 * mat) + 3 * idx + 3 * idx,
                "flops": 6.0 * nnz * F}
    d = dims(case)
    total, flops = 0.0, 0.0
    eb = 2.0 if case["bf16"] else 4.0
    for _, width in graphsage.aggregation_calls(d, case["project_first"]):
        total += ptr + idx + n * width * (eb + 4.0)
        flops += nnz * width
    for i in range(len(d) - 1):  # Linear: forward, gradient of the weights, gradient of the input
        total += (2 if i == 0 else 3) * 4.0 * n * (d[i] + d[i + 1])
        flops += (2 if i == 0 else 3) * 2.0 * n * d[i] * d[i + 1]
    return {"bytes": total, "flops": flops}


def gathered(case):
    """Gathered fp32 values of one pass: what the time of a pass goes with."""
    n, nnz = sizes(case)
    F, kind = case["F"], case["kind"]
    if kind == "ingest":
        return 200.0 * nnz
    if kind == "step":
        return 2.0 * nnz * F
    if kind == "epoch":
        d = dims(case)
        return (sum(1.0 * nnz * wd for _, wd in graphsage.aggregation_calls(d, case["project_first"]))
                + 60.0 * n * sum(d))
    return {"extremum": 8.0, "edges": 8.0, "weights": 4.0}[kind] * nnz * F


def draw(rng):
    """A case of the ranges above: any kind, any graph family, sizes spread over their logarithm."""
    most_bytes = max(work(c)["bytes"] for c in listed())
    most_time = max(gathered(c) for c in listed())
    while True:
        kind = rng.choice(["step"] * 5 + ["ingest", "extremum", "edges", "weights", "epoch"])
        graphs = ["reddit_like", "products_like", "papers_like"]
        if kind != "epoch":
            graphs += ["proteins_like", "tiny"]
        graph = rng.choice(graphs)
        F = rng.choice(WIDTHS) if rng.random() < 0.5 else int(round(math.exp(rng.uniform(math.log(8), math.log(602)))))
        case = {"kind": kind, "graph": graph, "F": 1 if kind == "ingest" else F,
                "weighted": kind == "weights" or rng.random() < 0.3, "self_loops": False}
        if graph == "tiny":
            case["n"] = int(round(math.exp(rng.uniform(math.log(256), math.log(4096)))))
            case["nnz"] = case["n"] * rng.randint(14, 24)
            case["scale"] = 1.0
        else:
            case["scale"] = round(math.exp(rng.uniform(math.log(5e-4), math.log(1.0))), 5)
        if kind == "step":
            case["op"] = rng.choice(["sum", "mean"])
            case["dtype"] = "bf16" if rng.random() < 0.3 else "f32"
            case["self_loops"] = rng.random() < 0.25
            if case["dtype"] == "bf16":
                case["F"] += F % 2  # the bf16 entry points take even widths
        elif kind == "extremum":
            case["reduce"], case["weighted"] = rng.choice(["max", "min"]), False
        elif kind == "edges":
            case["binary"], case["weighted"] = rng.choice(["mul", "mul", "add", "sub"]), False
        elif kind == "weights":
            case["op"] = rng.choice(["sum", "mean"])
        elif kind == "epoch":
            case["hidden"], case["layers"] = rng.choice([16, 64, 128, 256]), rng.choice([2, 3])
            case["project_first"], case["fused"] = rng.random() < 0.3, rng.random() < 0.3
            case["bf16"], case["weighted"] = rng.random() < 0.2, False
            case["self_loops"] = case["fused"]
        if work(case)["bytes"] <= most_bytes and gathered(case) <= most_time:
            return case


# ---- inputs and passes -----------------------------------------------------------------------

def endpoints(weights, gen):
    """count -> that many vertex ids with probability proportional to ``weights``.  The running sum
    is made on the host: on the GPU a floating-point cumsum need not round the same way twice, and a
    seed has to give the same graph every time."""
    cdf = torch.cumsum(weights.double().cpu(), 0)
    cdf = (cdf / cdf[-1]).to(weights.device)

    def pick(count):
        u = torch.rand(count, generator=gen, device=cdf.device, dtype=torch.float64)
        return torch.searchsorted(cdf, u, right=True).clamp_(max=cdf.numel() - 1)

    return pick


def undirected(case, seed, dev):
    """The Reddit- and Products-like graphs of synth.py (same construction, same sizes)."""
    n, nnz = sizes(case)
    gen = synth._gen(seed, dev)
    if case["graph"] == "reddit_like":  # 41 communities, 80 % of the edges inside one
        pick = endpoints(torch.exp(torch.randn(n, generator=gen, device=dev, dtype=torch.float64)), gen)
        bounds = (torch.arange(42, device=dev, dtype=torch.float64) * n / 41).floor().long()

        def pairs(count):
            a = pick(count)
            comm = torch.searchsorted(bounds, a, right=True) - 1
            r = torch.rand((2, count), generator=gen, device=dev, dtype=torch.float64)
            inside = bounds[comm] + (r[0] * (bounds[comm + 1] - bounds[comm]).double()).long()
            intra = torch.rand(count, generator=gen, device=dev) < 0.8
            return a, torch.where(intra, inside, (r[1] * n).long()).clamp_(max=n - 1)
    else:  # Chung-Lu, power law with exponent 2.1
        w = torch.rand(n, generator=gen, device=dev, dtype=torch.float64).clamp_(min=1e-12).pow(-1.0 / 1.1)
        mean = nnz / n
        for _ in range(8):  # rescale so that the capped weights average to the mean degree
            w = (w * (mean / w.mean())).clamp_(max=max(2.0e4 * case["scale"] ** 0.5, 2.0 * mean))
        pick = endpoints(w, gen)

        def pairs(count):
            return pick(count), pick(count)

    lo, hi = synth._exact_undirected(pairs, n, nnz // 2, gen, dev)
    rowptr, colidx, _ = synth._symmetric_csr(lo, hi, n, synth._relabel(n, False, gen, dev))
    return synth.SynthGraph(case["graph"], n, nnz, case["F"], rowptr, colidx, None, seed=seed)


def make_graph(case, seed, dev):
    if case["graph"] == "tiny":
        return synth.tiny(seed=seed, device=dev, n=case["n"], nnz=case["nnz"])
    if case["graph"] in ("reddit_like", "products_like"):
        return undirected(case, seed, dev)
    return synth.make(case["graph"], device=dev, scale=case["scale"], seed=seed)


def prepare(case, seed):
    kind, F, dev = case["kind"], case["F"], "cuda"
    sg = make_graph(case, seed, dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    w = None
    if case["weighted"]:
        w = sg.edge_w if sg.edge_w is not None else torch.rand(sg.nnz, generator=gen, device=dev)
    st = {"case": case}
    if kind == "ingest":
        st.update(n=sg.n, nnz=sg.nnz, rowptr=sg.rowptr, colidx=sg.colidx, w=w)
        return st
    g = binding.dg_graph_create(sg.n, sg.nnz, sg.rowptr, sg.colidx, w)
    if case["self_loops"]:
        g.dg_graph_set_param("self_loops", 1)
    g.dg_graph_transpose()
    st["g"] = g
    if kind == "epoch":
        d = dims(case)
        torch.manual_seed(seed)
        model = graphsage.GraphSAGE(g, d, project_first=case["project_first"], bf16_aggregate=case["bf16"],
                                    fused_aggregator=case["fused"]).to(dev)
        X = synth.features(sg.n, F, seed + 1, dev)
        labels = torch.randint(0, d[-1], (sg.n,), generator=gen, device=dev)
        train = torch.randperm(sg.n, generator=gen, device=dev)[: (2 * sg.n) // 3]
        st["model"], st["epoch"] = model, graphsage.make_epoch(model, X, labels, train)
        return st
    st["H"] = synth.features(sg.n, F, seed + 1, dev)
    st["dOut"] = synth.features(sg.n, F, seed + 2, dev)
    if kind == "step" and case["dtype"] == "bf16":
        st["H"], st["dOut"] = st["H"].to(torch.bfloat16), st["dOut"].to(torch.bfloat16)
    if kind == "edges":
        st["fE"] = torch.rand((sg.nnz, F), generator=gen, device=dev)
    if kind == "weights":
        st["w"] = w
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ingest":
        g = binding.dg_graph_create(state["n"], state["nnz"], state["rowptr"], state["colidx"], state["w"])
        g.dg_graph_transpose()
        return g.dg_graph_get_csc()
    if kind == "epoch":
        loss = state["epoch"]()
        params = list(state["model"].parameters())
        return {"loss": loss, "params": params, "grads": [p.grad for p in params]}
    g, H, dOut = state["g"], state["H"], state["dOut"]
    if kind == "step":
        op = OPS[case["op"]]
        if case["dtype"] == "bf16":
            return g.dg_aggregate_fwd_bf16(H, op), g.dg_aggregate_bwd_bf16(dOut, op)
        return g.dg_aggregate_fwd(H, op), g.dg_aggregate_bwd(dOut, op)
    if kind == "extremum":
        red = REDUCERS[case["reduce"]]
        fO, arg = g.dg_ap_fwd(H, None, binding.DG_BIN_COPY_LHS, red)
        dV, _ = g.dg_ap_bwd(dOut, H, None, binding.DG_BIN_COPY_LHS, red, arg=arg)
        return fO, arg, dV
    if kind == "edges":
        b = BINARIES[case["binary"]]
        fO, _ = g.dg_ap_fwd(H, state["fE"], b, binding.DG_RED_SUM)
        dV, dE = g.dg_ap_bwd(dOut, H, state["fE"], b, binding.DG_RED_SUM)
        return fO, dV, dE
    op, w = OPS[case["op"]], state["w"]
    out = g.dg_aggregate_fwd(H, op)
    dH = g.dg_aggregate_bwd(dOut, op)
    dW = g.dg_aggregate_edge_grad(H, dOut, op)
    w.sub_(dW, alpha=LR)
    g.dg_graph_update_weights()
    return out, dH, dW, w, g.dg_graph_get_csc()[2]


def tolerance(case):
    if case["kind"] == "ingest":  # integer work, and weights copied bit for bit
        return "exact"
    if case["kind"] == "epoch":
        # The first Adam steps move every parameter by about lr whatever its gradient's size, so a
        # gradient element within fp32 rounding of zero may move its parameter either way: single
        # elements by up to 2 lr, against a root mean square of the parameters of the same order.
        # (bf16 aggregation rounds activations that differ in the last fp32 bits to other bf16 values.)
        return {"rel": 5e-3, "max": 0.99}
    # sums in fp32 whatever the storage; the arg indices of an extremum are exact
    return {"rel": 1e-5}
