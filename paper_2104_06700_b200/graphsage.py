"""Full-batch GraphSAGE with the GCN aggregator (Section 5.1 of the paper, Models and
Parameters), as the composite workload the epoch-time metric is quoted on.

libdgagg runs the aggregation with the own row, the matrix products of large layers, the elementwise passes
of a layer and the loss; the products of small layers and Adam are torch's.  Per layer  z_v = (sum_{u in N(v)} h_u + h_v) / (deg(v) + 1),
h'_v = act(z_v W + b)  (aggregate first, then the Linear: Table 8 of the paper lists the aggregation
widths 100, 256, 256 for the 3-layer model, i.e. the layers' input widths), ReLU between layers, none
after the last, softmax cross-entropy on a training mask, Adam.  The features need no gradient, so an
L-layer epoch runs L forward and L-1 backward aggregations.  ``fused_aggregator`` is for handles with
the graph attribute "self_loops", which add the own row in every call.
"""
from __future__ import annotations

from typing import List, Sequence

import torch

from . import binding


class _Aggregate(torch.autograd.Function):
    """out = A H through dg_aggregate_fwd; the backward pass calls dg_aggregate_bwd.  With
    ``bf16`` the gathered matrices (H in the forward, dOut in the backward pass) are rounded to
    bf16 first and the bf16 entry points are used; sums and results stay fp32.

    ``row_scale`` (n x 1, only with op = mean on a handle with self loops): the backward pass
    multiplies dOut by it and runs the *sum* backward on the product instead of the mean
    backward.  Both give A^T D dOut + D dOut; the sum backward needs no per-edge factor, which
    on graphs with long rows saves more kernel time than the one elementwise pass costs."""

    @staticmethod
    def forward(ctx, H: torch.Tensor, graph: "binding.Graph", op: int, bf16: bool,
                row_scale, edge_w=None) -> torch.Tensor:
        ctx.graph, ctx.op, ctx.bf16, ctx.row_scale = graph, op, bf16, row_scale
        ctx.want_dw = edge_w is not None and edge_w.requires_grad
        if ctx.want_dw:
            if edge_w.data_ptr() != graph.edge_w.data_ptr():
                raise ValueError("edge_w must be the tensor the graph handle was created with")
            ctx.save_for_backward(H)
        if bf16:
            return graph.dg_aggregate_fwd_bf16(H.contiguous().to(torch.bfloat16), op)
        return graph.dg_aggregate_fwd(H.contiguous(), op)

    @staticmethod
    def backward(ctx, dOut: torch.Tensor):
        dH = None
        upstream = dOut
        if ctx.needs_input_grad[0]:
            op = ctx.op
            if ctx.row_scale is not None:
                dOut = dOut * ctx.row_scale
                op = binding.DG_OP_SUM
            if ctx.bf16:
                dH = ctx.graph.dg_aggregate_bwd_bf16(dOut.contiguous().to(torch.bfloat16), op)
            else:
                dH = ctx.graph.dg_aggregate_bwd(dOut.contiguous(), op)
        dW = None
        if ctx.want_dw:     # message passing onto the edges: one dot product per edge
            (H,) = ctx.saved_tensors
            dW = ctx.graph.dg_aggregate_edge_grad(H.contiguous(), upstream.contiguous(), ctx.op)
        return dH, None, None, None, None, dW


def _weight_grad(G: torch.Tensor, X: torch.Tensor) -> torch.Tensor:
    """G^T X: n rows reduced to a matrix of a layer's size.  As one product the fp32 GEMM leaves most of the chip
    idle; in 64 slices of the rows, summed, 245 k rows of 256 x 100 take 311 us instead of 504, 256 x 256
    597 / 718, 47 x 256 167 / 346 (32 slices: 319, 597, 221; 128: 409, 606, 165).  Below 2^27 products or
    8 k rows the launches cost more than that gives (12 k rows of 47 x 256: 39 us either way)."""
    n, slices = G.shape[0], 64
    if n < 8192 or n * G.shape[1] * X.shape[1] < 1 << 27:
        return G.t() @ X
    m = n // slices * slices
    dW = torch.bmm(G[:m].view(slices, -1, G.shape[1]).transpose(1, 2), X[:m].view(slices, -1, X.shape[1])).sum(0)
    return dW.addmm_(G[m:].t(), X[m:]) if m < n else dW


def _by_library(graph: "binding.Graph", weight: torch.Tensor):
    """Which products of a layer the library computes, and not torch's fp32 GEMMs: forward, gradient of the input, of the
    weights.  From 2^29 multiplications on it is faster, if neither width is small: tiles are 128 rows by whole steps of 16
    columns.  us library / torch, forward with its epilogue, gradients: 245 k rows of 256 x 256 189 / 660, 191 / 569, 267 / 594; of
    256 x 47 123 / 198, 103 / 173, -; 8 k of 256 x 256 23 / 31, 21 / 27, 31 / 36; but 100 k of 64 x 41 49 / 43, 39 / 29, 49 / 44;
    of 602 x 16 158 / 115, 160 / 94, 195 / 123.  Of the large ones torch keeps
      - those that fill few SMs: 4096 rows of 602 to 256 columns 40 / 36, 39 / 32; 8192 23 / 31;
      - gradients of narrow inputs, which have no epilogue to save: 245 k rows to 64 columns from 41 75 / 62, 100 k from 100
        45 / 39, from 602 171 / 156; and of wide ones from rows that allow no vectors: 33 k from 41 to 602 71 / 65;
      - gradients of weights of which one side is mostly padding to 128 and the other takes more than one tile, 245 k rows:
        47 x 256 174 / 165, 602 x 47 508 / 432 (47 x 128 99 / 117), or both are read number by number: 47 x 47 115 / 106;
        and those with little scratch, summed in few blocks: 256 x 256 with 5 and 4 MiB 481 and 597 / 594, 602 x 256 with 5 1507 / 1367.

    The library's calls take widths of up to 2^20.  A caller who allowed torch TF32 products (set_float32_matmul_precision, allow_tf32) keeps them: us
    library / TF32, 245 k rows of 256 x 256 194 / 168, 194 / 85, 267 / 101."""
    if graph.n * weight.numel() < 1 << 29:      # first: a small graph's epoch is host time
        return False, False, False
    N, K = weight.shape
    if (min(N, K) < 40 or max(N, K) > 1 << 20
            or torch.backends.cuda.matmul.fp32_precision not in ("none", "ieee")):
        return False, False, False
    small, big, tiles = min(N, K), max(N, K), (graph.n + 127) // 128
    return (tiles * ((N + 255) // 256) >= 64,
            tiles * ((K + 255) // 256) >= 64 and K > 64 and (N % 4 == 0 or K <= 256),
            (small > 64 or big <= 128 and (N % 4 == 0 or K % 4 == 0)) and graph.dg_graph_get_param("scratch_mb") >= 7)


def _with_own_row(graph: "binding.Graph", M: torch.Tensor, bf16: bool, transposed: bool) -> torch.Tensor:
    """(A + I) M, or with ``transposed`` (A^T + I) M.  bf16: the gathered rows are rounded; the own row too where
    the handle adds it itself."""
    if not bf16:
        call = graph.dg_aggregate_bwd_self if transposed else graph.dg_aggregate_fwd_self
        return call(M, binding.DG_OP_SUM)
    call = graph.dg_aggregate_bwd_bf16 if transposed else graph.dg_aggregate_fwd_bf16
    out = call(M.to(torch.bfloat16), binding.DG_OP_SUM)
    return out if graph.dg_graph_get_param("self_loops") else out.add_(M)


class _GcnLayer(torch.autograd.Function):
    """One layer  act(D (A M + M) W^T + b),  D = diag(1 / (deg + 1)),  with the own row added inside the
    aggregation kernel.  D is applied after the GEMM, forward together with bias and ReLU, backward together
    with the ReLU's mask and the sums of the bias: one elementwise pass over n x F each way, none forward where the
    library computes the product too (autograd's
    operations made two forward and three backward; 245 k vertices, 256 wide: 85 us a pass).

    ``project``: D ((A + I) (M W^T)) + b instead, the narrower product aggregated."""

    @staticmethod
    def forward(ctx, M, weight, bias, graph, inv_deg1, relu: bool, project: bool, bf16: bool):
        M = M.contiguous()
        if project:
            X = M
            large = _by_library(graph, weight)[0]
            Z = graph.dg_linear_fwd(M, weight.contiguous()) if large else M @ weight.t()
            out = graph.dg_layer_fwd(_with_own_row(graph, Z, bf16, False), inv_deg1, bias.contiguous(), relu)
        else:
            X = _with_own_row(graph, M, bf16, False)
            if _by_library(graph, weight)[0]:
                out = graph.dg_linear_fwd(X, weight.contiguous(), inv_deg1, bias.contiguous(), relu)
            else:
                out = graph.dg_layer_fwd(X @ weight.t(), inv_deg1, bias.contiguous(), relu)
        ctx.graph, ctx.relu, ctx.project, ctx.bf16 = graph, relu, project, bf16
        # M is the layer's input (another layer's output, which that one keeps) and costs no memory
        ctx.save_for_backward(X, weight, inv_deg1, out if relu else None, M, bias)
        return out

    @staticmethod
    def backward(ctx, dOut: torch.Tensor):
        X, weight, inv_deg1, out, M, bias = ctx.saved_tensors
        graph, needs = ctx.graph, ctx.needs_input_grad
        if torch.is_grad_enabled():     # create_graph: the gradients are differentiated in their turn
            again = _layer_by_operations(M, weight, bias, graph, inv_deg1, ctx.relu, ctx.project, ctx.bf16)
            inputs = [t for t, need in zip((M, weight, bias), needs) if need]
            grads = iter(torch.autograd.grad(again, inputs, dOut, create_graph=True))
            return (*[next(grads) if need else None for need in needs[:3]], None, None, None, None, None)
        G, db = graph.dg_layer_bwd(dOut.contiguous(), out, inv_deg1)
        if ctx.project and (needs[0] or needs[1]):
            G = _with_own_row(graph, G, ctx.bf16, True)
        _, input_grad, weight_grad = _by_library(graph, weight)
        dW = dM = None
        if needs[1]:
            dW = graph.dg_linear_bwd_weight(G, X) if weight_grad else _weight_grad(G, X)
        if needs[0]:
            dM = graph.dg_linear_bwd_input(G, weight.contiguous()) if input_grad else G @ weight
            if not ctx.project:
                dM = _with_own_row(graph, dM, ctx.bf16, True)
        return dM, dW, db if needs[2] else None, None, None, None, None, None


class _CrossEntropy(torch.autograd.Function):
    """torch's cross_entropy(logits[index], labels[index]) in two kernels forward and one backward."""

    @staticmethod
    def forward(ctx, logits, index, labels, graph):
        result, stats = graph.dg_cross_entropy_fwd(logits, index, labels)
        ctx.graph = graph
        ctx.save_for_backward(logits, index, labels, result, stats)
        return result[0].clone()

    @staticmethod
    def backward(ctx, grad: torch.Tensor):
        logits, index, labels, result, stats = ctx.saved_tensors
        return ctx.graph.dg_cross_entropy_bwd(logits, index, labels, result, stats, grad), None, None, None


def aggregate(graph: "binding.Graph", H: torch.Tensor, op: int = binding.DG_OP_SUM,
              bf16: bool = False, row_scale=None, edge_w=None) -> torch.Tensor:
    """Differentiable aggregation primitive (the graph must have been transposed).

    ``edge_w``: pass the weight tensor the handle was created with to get its gradient too
    (learnable edge weights).  The handle reads that tensor in place; after an optimiser step
    on it call ``graph.dg_graph_update_weights()`` so that the CSC used by the backward pass
    carries the new values."""
    return _Aggregate.apply(H, graph, op, bf16, row_scale, edge_w)


def _gcn(graph: "binding.Graph", M: torch.Tensor, inv_deg1: torch.Tensor, bf16: bool) -> torch.Tensor:
    """(sum of the neighbours' rows + own row) / (in-degree + 1), operation by operation."""
    total = aggregate(graph, M, binding.DG_OP_SUM, bf16)
    return (total if graph.dg_graph_get_param("self_loops") else total + M) * inv_deg1


def _layer_by_operations(M, weight, bias, graph, inv_deg1, relu: bool, project: bool, bf16: bool):
    """What _GcnLayer computes, from operations that autograd knows."""
    if project:
        out = _gcn(graph, M @ weight.t(), inv_deg1, bf16) + bias
    else:
        out = torch.nn.functional.linear(_gcn(graph, M, inv_deg1, bf16), weight, bias)
    return torch.relu(out) if relu else out


def _is_plain(lin: torch.nn.Module) -> bool:
    """Whether calling ``lin`` would compute x W^T + b from its parameters and do nothing else."""
    hooks = torch.nn.modules.module
    return (type(lin) is torch.nn.Linear and lin.bias is not None and "forward" not in lin.__dict__
            and not (lin._forward_hooks or lin._forward_pre_hooks or lin._backward_hooks or lin._backward_pre_hooks
                     or hooks._global_forward_hooks or hooks._global_forward_pre_hooks
                     or hooks._global_backward_hooks or hooks._global_backward_pre_hooks)
            and not torch.is_autocast_enabled())


class GraphSAGE(torch.nn.Module):
    """`dims` = [in, hidden, ..., classes]; one Linear per layer.

    ``project_first``: the aggregator is linear, so ((A H + H) / (deg+1)) W = (A (H W) + H W) /
    (deg+1): a layer whose output is narrower than its input may apply the Linear first and
    aggregate the narrower matrix.  Same function up to fp32 rounding, less aggregation work
    (602 -> 256 columns on the first Reddit-like layer); off by default because the paper
    aggregates first (its Table 8 counts the aggregation at the layers' input widths).

    A layer runs as one autograd function on its Linear's parameters; where that Linear has hooks, no bias,
    another type (a parametrization, a module put in its place) or runs under autocast, the module itself is
    called between the aggregation and the activation.
    """

    def __init__(self, graph: "binding.Graph", dims: Sequence[int], project_first: bool = False,
                 bf16_aggregate: bool = False, fused_aggregator: bool = False):
        super().__init__()
        self.graph = graph
        self.project_first = project_first
        self.bf16_aggregate = bf16_aggregate   # aggregate bf16-rounded activations (even widths)
        # for a handle whose "self_loops" attribute was set to 1 before dg_graph_transpose
        self.fused_aggregator = fused_aggregator
        if fused_aggregator and graph.dg_graph_get_param("self_loops") != 1:
            raise ValueError("fused_aggregator needs a graph handle with self_loops = 1")
        if not fused_aggregator and graph.dg_graph_get_param("self_loops") != 0:
            raise ValueError("this handle adds self loops itself: use fused_aggregator=True")
        self.lin = torch.nn.ModuleList(
            [torch.nn.Linear(dims[i], dims[i + 1]) for i in range(len(dims) - 1)])
        deg = (graph.rowptr[1:] - graph.rowptr[:-1]).to(torch.float32)
        self.register_buffer("inv_deg1", (1.0 / (deg + 1.0)).unsqueeze(1))

    def forward(self, H: torch.Tensor) -> torch.Tensor:
        for i, lin in enumerate(self.lin):
            project = self.project_first and lin.out_features < lin.in_features
            relu = i + 1 < len(self.lin)
            if _is_plain(lin):
                width = lin.out_features if project else lin.in_features
                H = _GcnLayer.apply(H, lin.weight, lin.bias, self.graph, self.inv_deg1, relu, project,
                                    self.bf16_aggregate and width % 2 == 0)
                continue
            if project:
                H = self._aggregated(torch.nn.functional.linear(H, lin.weight)) + lin.bias
            else:
                H = lin(self._aggregated(H))
            H = torch.relu(H) if relu else H
        return H

    def _aggregated(self, M: torch.Tensor) -> torch.Tensor:
        return _gcn(self.graph, M, self.inv_deg1, self.bf16_aggregate and M.shape[1] % 2 == 0)


def make_epoch(model: GraphSAGE, X: torch.Tensor, labels: torch.Tensor, train_idx: torch.Tensor,
               lr: float = 0.01, weight_decay: float = 5e-4):
    """Returns a function that runs one training epoch (forward, loss on the training vertices,
    backward, Adam step) and returns the loss tensor."""
    # one kernel for all parameters where they are on a GPU: a small graph's epoch is host time
    opt = torch.optim.Adam(model.parameters(), lr=lr, weight_decay=weight_decay,
                           fused=all(p.is_cuda for p in model.parameters()))

    n = model.graph.n
    # vertex indices and class indices, one row of logits each; masks, probabilities and the like are torch's
    plain = (train_idx.dtype == labels.dtype == torch.int64 and train_idx.dim() == labels.dim() == 1
             and train_idx.is_contiguous() and labels.is_contiguous() and labels.shape[0] == n
             and train_idx.is_cuda and labels.is_cuda)
    if plain and train_idx.numel():     # the kernel has no way to raise: it returns NaN
        if int(train_idx.min()) < -n or int(train_idx.max()) >= n:
            raise IndexError("train_idx holds an index outside the graph")
        y = labels[train_idx]
        if bool(((y != -100) & ((y < 0) | (y >= model.lin[-1].out_features))).any()):
            raise IndexError("labels holds a class outside the model's last layer")

    def epoch() -> torch.Tensor:
        opt.zero_grad(set_to_none=True)
        logits = model(X)
        if plain:
            loss = _CrossEntropy.apply(logits, train_idx, labels, model.graph)
        else:
            loss = torch.nn.functional.cross_entropy(logits[train_idx], labels[train_idx])
        loss.backward()
        opt.step()
        return loss.detach()

    return epoch


def aggregation_calls(dims: Sequence[int], project_first: bool = False) -> List[tuple]:
    """(direction, width) of every aggregation one epoch runs, for work accounting.  Aggregating
    first, layer 1 needs no backward aggregation (the features carry no gradient); projecting
    first, the aggregated matrix depends on the layer's weights, so it does."""
    calls = []
    for i in range(len(dims) - 1):
        first = project_first and dims[i + 1] < dims[i]
        w = dims[i + 1] if first else dims[i]
        calls.append(("fwd", w))
        if i > 0 or first:
            calls.append(("bwd", w))
    return calls
