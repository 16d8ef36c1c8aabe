"""The work a user has this package do, as timed cases: single graphs in each
precision, packed batches, and differentiable distances (forward + backward).

Sizes are those of the package's configurations, tests and benchmark (n = 1024,
4096, 16384; 4096 graphs of 16..512 vertices; 256 graphs of 256 vertices) and
generic odd ones beside them.  Weights: integers U[1, 100] (with ties), reals
U[0.5, 2), int32 U[1, 2^26]; a missing edge is +inf (I32_INF), the diagonal 0.
A solve works in place, so a pass first restores the weights, as a program does
that keeps them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2105_07298_gb300 as apsp
from paper_2105_07298_gb300.batched import packed_numel, packed_offsets

DEVICE = "cuda"


def listed():
    return [
        # One graph no larger than a block: a call's latency.
        dict(name="f32_n97_path", kind="single", dtype="f32", n=97, path=True, weights="int", p=0.3),
        # The smallest configuration of the benchmark, distances and paths.
        dict(name="f32_n1024_path", kind="single", dtype="f32", n=1024, path=True, weights="int", p=0.3),
        # Distances alone, a ragged odd size whose rows are not 16-byte aligned.
        dict(name="f32_n2049_dist", kind="single", dtype="f32", n=2049, path=False, weights="real", p=0.4),
        # The n sweep: a mid size, and the largest that stays well below 2 s.
        dict(name="f32_n4096_path", kind="single", dtype="f32", n=4096, path=True, weights="int", p=0.5),
        dict(name="f32_n16384_path", kind="single", dtype="f32", n=16384, path=True, weights="int", p=0.5),
        # Double precision: real weights (no sum is a float), and integers.
        dict(name="f64_n1000_path", kind="single", dtype="f64", n=1000, path=True, weights="real", p=0.4),
        dict(name="f64_n4096_path", kind="single", dtype="f64", n=4096, path=True, weights="int", p=0.5),
        # Exact int32 weights beyond 2^24.
        dict(name="i32_n2048_path", kind="single", dtype="i32", n=2048, path=True, weights="wide", p=0.5),
        # The batched workload: uneven graphs, one plan run many times.
        dict(name="batched_4096_path", kind="batched", graphs=4096, lo=16, hi=512, path=True, plan=True,
             weights="int", p=0.3),
        # A batch of small graphs given once: distances only, plan and run in one call.
        dict(name="batched_1000_small", kind="batched", graphs=1000, lo=16, hi=64, path=False, plan=False,
             weights="int", p=0.3),
        # Training through distances: an even stack, and an uneven packed batch.
        dict(name="grad_256x256", kind="stack", graphs=256, n=256, p=0.4),
        dict(name="grad_packed_300", kind="packed", graphs=300, lo=20, hi=200, p=0.4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "batched", "batched", "stack", "packed"])
    p = round(rng.uniform(0.2, 0.6), 2)
    if kind == "single":
        dtype = rng.choice(["f32", "f32", "f64", "i32"])
        n = _log_int(rng, 40, {"f32": 12000, "f64": 6000, "i32": 4500}[dtype])
        weights = "wide" if dtype == "i32" else rng.choice(["int", "real"])
        return dict(kind=kind, dtype=dtype, n=n, path=rng.random() < 0.7, weights=weights, p=p)
    if kind == "batched":
        return dict(kind=kind, graphs=_log_int(rng, 60, 4096), lo=16, hi=_log_int(rng, 48, 512),
                    path=rng.random() < 0.6, plan=rng.random() < 0.6, weights=rng.choice(["int", "real"]), p=p)
    if kind == "stack":
        return dict(kind=kind, graphs=_log_int(rng, 8, 256), n=_log_int(rng, 24, 384), p=p)
    return dict(kind=kind, graphs=_log_int(rng, 30, 600), lo=16, hi=_log_int(rng, 48, 400), p=p)


# ---------------------------------------------------------------- inputs
_TYPES = {"f32": torch.float32, "f64": torch.float64, "i32": torch.int32}


def _fill(count, weights, p, dtype, gen):
    """``count`` independent entries: an edge weight with probability p, else no edge."""
    if weights == "int":
        w = torch.randint(1, 101, (count,), generator=gen, device=DEVICE, dtype=torch.int32).to(dtype)
    elif weights == "wide":
        w = torch.randint(1, (1 << 26) + 1, (count,), generator=gen, device=DEVICE, dtype=torch.int32).to(dtype)
    else:
        real = dtype if dtype.is_floating_point else torch.float32
        w = torch.rand(count, generator=gen, device=DEVICE, dtype=real) * 1.5 + 0.5
    none = apsp.I32_INF if dtype == torch.int32 else math.inf
    w[torch.rand(count, generator=gen, device=DEVICE) >= p] = none
    return w


def _sizes(case):
    """Vertex counts of a packed batch: uniform on [lo, hi], the same for every seed."""
    rng = np.random.default_rng((case["graphs"], case["lo"], case["hi"]))
    return rng.integers(case["lo"], case["hi"] + 1, size=case["graphs"]).astype(np.int64)


def _packed(case, gen):
    """(packed weights, sizes, offsets); the up to three entries between graphs are 0."""
    sizes = _sizes(case)
    off = packed_offsets(sizes)
    W = _fill(packed_numel(sizes), case.get("weights", "real"), case["p"], torch.float32, gen)
    diag = np.concatenate([o + np.arange(n) * (n + 1) for n, o in zip(sizes, off)])
    gaps = [np.arange(o + n * n, o + (n * n + 3) // 4 * 4) for n, o in zip(sizes[:-1], off[:-1])]
    W[torch.from_numpy(np.concatenate([diag] + gaps)).to(DEVICE)] = 0.0
    return W, sizes, off


def _weights(case, seed):
    """The case's weights: a matrix, a stack, or (packed buffer, sizes, offsets)."""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    if case["kind"] == "single":
        n = case["n"]
        W = _fill(n * n, case["weights"], case["p"], _TYPES[case["dtype"]], gen).view(n, n)
        W.fill_diagonal_(0)
        return W
    if case["kind"] == "stack":
        n = case["n"]
        W = _fill(case["graphs"] * n * n, "real", case["p"], torch.float32, gen).view(case["graphs"], n, n)
        W.diagonal(dim1=1, dim2=2).zero_()
        return W
    return _packed(case, gen)


def _upstream(W, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(seed + 1000003)
    return torch.randn(W.shape, generator=gen, device=DEVICE)


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "single":
        W = _weights(case, seed)
        state.update(W=W, D=torch.empty_like(W))
        if case["path"]:
            state["P"] = torch.empty(W.shape, dtype=torch.int32, device=DEVICE)
    elif case["kind"] == "batched":
        W, sizes, off = _weights(case, seed)
        state.update(W=W, D=torch.empty_like(W), sizes=sizes, off=off)
        if case["path"]:
            state["P"] = torch.full(W.shape, -1, dtype=torch.int32, device=DEVICE)
        if case["plan"]:
            state["plan"] = apsp.BatchedPlan(sizes, off)
    elif case["kind"] == "stack":
        W = _weights(case, seed)
        state.update(W=W.requires_grad_(), g=_upstream(W, seed))
    else:
        W, sizes, off = _weights(case, seed)
        state.update(W=W.requires_grad_(), g=_upstream(W, seed), sizes=sizes, off=off)
    return state


def run(state):
    kind = state["case"]["kind"]
    if kind == "stack":
        D = apsp.shortest_path_distances(state["W"])
        (grad,) = torch.autograd.grad(D, state["W"], state["g"])
        return {"dist": D, "grad": grad}
    if kind == "packed":
        D = apsp.shortest_path_distances_packed(state["W"], state["sizes"], state["off"])
        (grad,) = torch.autograd.grad(D, state["W"], state["g"])
        return {"dist": D, "grad": grad}
    D, P = state["D"], state.get("P")
    D.copy_(state["W"])
    if kind == "single":
        apsp.apsp_fw(D, P)
    elif "plan" in state:
        state["plan"].run(D, P)
    else:
        apsp.apsp_fw_batched(D, state["sizes"], state["off"], P)
    return {"dist": D} if P is None else {"dist": D, "path": P}


# ---------------------------------------------------------------- cost and results
def work(case):
    """2 operations (add, compare) per relaxation, n^3 of them; weights read, distances
    (and paths, or gradients) written."""
    kind = case["kind"]
    if kind in ("batched", "packed"):
        n = _sizes(case).astype(np.float64)
        n2, n3 = float(np.sum(n ** 2)), float(np.sum(n ** 3))
    else:
        count = case.get("graphs", 1)
        n2, n3 = count * float(case["n"]) ** 2, count * float(case["n"]) ** 3
    if kind in ("stack", "packed"):  # weights and upstream read, distances and gradient written
        return {"bytes": 16.0 * n2, "flops": 2.0 * n3 + n2}
    size = 8 if case.get("dtype") == "f64" else 4
    return {"bytes": n2 * (2 * size + (4 if case["path"] else 0)), "flops": 2.0 * n3}


def tolerance(case):
    """About four times what was measured.  Single graphs: distances and paths are those of the
    sequential blocked algorithm, bit for bit (the C header's contract).  Batched integer
    weights: every sum is exact.  Batched real weights: the order of additions is free (3e-8 and
    at most 1.2e-7 from 64 bits), and a path entry may move where two sums differ by rounding
    alone.  Gradients: FP32 atomic sums in no fixed order (1e-7 from pass to pass), and a pair
    whose two best paths differ by rounding alone may put its whole gradient on the other one
    (4e-4 from 64 bits where that happened once in 16.7 million pairs)."""
    if case["kind"] == "single":
        return "exact"
    if case["kind"] == "batched":
        return "exact" if case["weights"] == "int" else {"rel": 1.2e-7, "max": 5e-7, "differ": 1e-3}
    return {"rel": 1.6e-3, "max": 0.9}


def _fw64(D, pred=None):
    """Floyd-Warshall in 64 bits on a (B, n, n) stack, in place; with ``pred``, the last
    vertex before j on the path of each (i, j) too."""
    for k in range(D.shape[-1]):
        cand = D[:, :, k:k + 1] + D[:, k:k + 1, :]
        if pred is not None:
            torch.where(cand < D, pred[:, k:k + 1, :].expand_as(pred), pred, out=pred)
        torch.minimum(D, cand, out=D)
    return D


def _grad64(D, pred, g):
    """dL/dW of each graph: every reachable pair's g added to the edges of its path."""
    B, n, _ = D.shape
    ok = torch.isfinite(D) & ~torch.eye(n, dtype=torch.bool, device=DEVICE)
    b, i, j = ok.nonzero(as_tuple=True)
    gv = g[b, i, j]
    grad = torch.zeros(B * n * n, dtype=torch.float64, device=DEVICE)
    while len(b):
        u = pred[b, i, j]
        grad.index_add_(0, (b * n + u) * n + j, gv)
        more = u != i
        b, i, j, gv = b[more], i[more], u[more], gv[more]
    return grad.view(B, n, n)


def _solve64(W, g=None):
    """64-bit distances of a (B, n, n) stack, and its gradient for the upstream g."""
    D = W.double()
    if g is None:
        return _fw64(D), None
    n = W.shape[-1]
    pred = torch.arange(n, device=DEVICE)[None, :, None].expand(W.shape).contiguous()
    _fw64(D, pred)
    return D, _grad64(D, pred, g.double())


def exact(case, seed):
    kind = case["kind"]
    W = _weights(case, seed)
    if kind == "single":
        if case["n"] > 8192:
            return None
        W64 = W.double()
        if case["dtype"] == "i32":
            W64[W == apsp.I32_INF] = math.inf
        D = _fw64(W64[None])[0]
        if case["dtype"] == "i32":
            D = torch.where(torch.isinf(D), float(apsp.I32_INF), D).to(torch.int32)
        return {"dist": D, "path": None} if case["path"] else {"dist": D}
    if kind == "stack":
        D, grad = _solve64(W, _upstream(W, seed))
        return {"dist": D, "grad": grad}
    W, sizes, off = W
    g = _upstream(W, seed) if kind == "packed" else None
    D, grad = W.double(), torch.zeros(W.shape, dtype=torch.float64, device=DEVICE)
    order = np.argsort(sizes, kind="stable")
    for at in range(0, len(order), 64):  # graphs of like size together, padded with lone vertices
        ids = order[at:at + 64]
        n = int(sizes[ids].max())
        Ws = torch.full((len(ids), n, n), math.inf, dtype=torch.float64, device=DEVICE)
        Ws.diagonal(dim1=1, dim2=2).zero_()
        gs = torch.zeros_like(Ws) if g is not None else None
        part = [(t, int(sizes[q]), int(off[q])) for t, q in enumerate(ids)]
        for t, m, o in part:
            Ws[t, :m, :m] = W[o:o + m * m].view(m, m)
            if g is not None:
                gs[t, :m, :m] = g[o:o + m * m].view(m, m)
        Ds, grads = _solve64(Ws, gs)
        for t, m, o in part:
            D[o:o + m * m] = Ds[t, :m, :m].reshape(-1)
            if g is not None:
                grad[o:o + m * m] = grads[t, :m, :m].reshape(-1)
    if kind == "packed":
        return {"dist": D, "grad": grad}
    return {"dist": D, "path": None} if case["path"] else {"dist": D}
