"""The calls whose speed is followed: what a program asks of this library, from
the smallest graph to the largest, in every element type, single, batched, on
host buffers and inside a training step.

A case names its kind (which entry point it goes through), its sizes and its
weights.  Weights are those of the repository's own workloads: int32 U[1, hi],
fp32 and fp64 uniform in (0, 1] (fp32 in [1, 2) under training), int64
U[1, 1e12]; an edge is present with probability p, the diagonal is 0 and a
missing edge is the type's INF.
"""
import math

import numpy as np
import torch

import paper_2403_18619_gb300 as fw
from paper_2403_18619_gb300 import autograd as fw_autograd

DTYPES = {"i32": torch.int32, "f32": torch.float32, "i64": torch.int64, "f64": torch.float64}
INF = {"i32": fw.INF_I32, "i64": fw.INF_I64, "f32": math.inf, "f64": math.inf}


def listed():
    return [
        # one small graph, answered at once: latency and launches are all there is
        dict(name="i32_n64", kind="solve", dtype="i32", n=64, p=0.3, hi=100, pred=True),
        # the small dense workload: bound by the chain of its rounds
        dict(name="i32_n1024", kind="solve", dtype="i32", n=1024, p=1.0, hi=100, pred=True),
        # an ordinary graph whose weights and results live in host memory
        dict(name="i32_host_n4096", kind="host", dtype="i32", n=4096, p=0.5, hi=1000, pred=True),
        # a large dense graph: the headline recipe (p = 0.9, U[1, 1e4]) at half its side
        dict(name="i32_n16384", kind="solve", dtype="i32", n=16384, p=0.9, hi=10000, pred=True),
        # the paper's own element type and its common size, with the path matrix
        dict(name="f32_n8192", kind="solve", dtype="f32", n=8192, p=0.5, hi=0, pred=True),
        # distances only (metric closures, graph features), a size no block divides
        dict(name="f32_dist_n5000", kind="solve", dtype="f32", n=5000, p=0.5, hi=0, pred=False),
        # the paper's double-precision runs
        dict(name="f64_n4096", kind="solve", dtype="f64", n=4096, p=0.5, hi=0, pred=True),
        # 64-bit integer weights (exact sums of large lengths), a size no block divides
        dict(name="i64_n3000", kind="solve", dtype="i64", n=3000, p=0.5, hi=10**12, pred=True),
        # many graphs of uneven size through one kept plan (a data set's graphs)
        dict(name="i32_batch128", kind="batched", dtype="i32", batch=128, lo=64, n=2048, p=0.3,
             hi=100, pred=True, sizes=11),
        # a training step: forward and backward of a batch of graphs through autograd
        dict(name="f32_train32x1024", kind="train", dtype="f32", batch=32, n=1024, p=0.1, hi=0),
        # the backward alone, as a program with its own solve calls it
        dict(name="f32_backward64x1024", kind="backward", dtype="f32", batch=64, n=1024, p=0.1,
             hi=0),
        # the paper's path bookkeeping (P_ij = k) from the solved last hops
        dict(name="intermediate_n8192", kind="intermediate", dtype="i32", n=8192, p=0.5, hi=1000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _int_weight(rng, n):
    """Largest int32 weight of a drawn graph: 100 up to what n allows ((n-1) * hi < 2^29)."""
    return _log_int(rng, 100, max(101, min(10**6, (2**29 - 1) // max(1, n - 1))))


def draw(rng):
    kind = rng.choice(["solve_i32", "solve_i32", "solve_i32", "solve_f32", "solve_f32",
                       "solve_f64", "solve_i64", "host", "batched", "train", "backward",
                       "intermediate"])
    p = rng.choice([0.1, 0.3, 0.5, 0.9, 1.0])
    if kind == "solve_i32":
        n = _log_int(rng, 33, 12000)
        return dict(kind="solve", dtype="i32", n=n, p=p, hi=_int_weight(rng, n),
                    pred=rng.random() < 0.8)
    if kind == "solve_f32":
        return dict(kind="solve", dtype="f32", n=_log_int(rng, 33, 8192), p=p, hi=0,
                    pred=rng.random() < 0.6)
    if kind == "solve_f64":
        return dict(kind="solve", dtype="f64", n=_log_int(rng, 100, 4096), p=p, hi=0,
                    pred=rng.random() < 0.7)
    if kind == "solve_i64":
        return dict(kind="solve", dtype="i64", n=_log_int(rng, 100, 4096), p=p,
                    hi=_log_int(rng, 100, 10**12), pred=rng.random() < 0.7)
    if kind == "host":
        n = _log_int(rng, 100, 4096)
        return dict(kind="host", dtype="i32", n=n, p=p, hi=_int_weight(rng, n),
                    pred=rng.random() < 0.8)
    if kind == "batched":
        top = _log_int(rng, 200, 2048)
        dtype = rng.choice(["i32", "i32", "f32"])
        return dict(kind="batched", dtype=dtype, batch=rng.randint(8, 128), lo=min(64, top),
                    n=top, p=p, hi=_int_weight(rng, top) if dtype == "i32" else 0,
                    pred=rng.random() < 0.8, sizes=rng.randint(1, 10**6))
    if kind == "intermediate":
        return dict(kind="intermediate", dtype="i32", n=_log_int(rng, 200, 8192), p=p, hi=1000)
    n = _log_int(rng, 60, 1200)
    batch = max(2, min(64, int(32 * (1024 / n) ** 2 * rng.random())))
    return dict(kind=kind, dtype="f32", batch=batch, n=n, p=p, hi=0)


# ------------------------------------------------------------------ inputs ---

def _weights(case, n, gen, device="cuda"):
    """One n x n weight matrix (rows padded to 16 bytes), drawn on the GPU."""
    dtype, hi = case["dtype"], case["hi"]
    full = torch.zeros((n, fw.padded(n)), dtype=DTYPES[dtype], device="cuda")
    W = full[:, :n]
    if dtype in ("i32", "i64"):
        W.random_(1, hi + 1, generator=gen)
    elif case["kind"] in ("train", "backward"):
        W.uniform_(1.0, 2.0, generator=gen)
    else:
        W.uniform_(0.0, 1.0, generator=gen)
        W.neg_().add_(1)  # [0, 1) -> (0, 1]
    if case["p"] < 1.0:
        W.masked_fill_(torch.rand((n, n), generator=gen, device="cuda") >= case["p"], INF[dtype])
    W.fill_diagonal_(0)
    if device == "cpu":
        out = torch.empty(full.shape, dtype=full.dtype, pin_memory=True)
        out.copy_(full)
        return out[:, :n]
    return W


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _batch_weights(case, gen):
    """(B, n, n) fp32 weights with contiguous rows."""
    return torch.stack([_weights(case, case["n"], gen) for _ in range(case["batch"])])


def _sizes(case):
    r = np.random.RandomState(case["sizes"])
    return [int(x) for x in r.randint(case["lo"], case["n"] + 1, case["batch"])]


def _strided(t):
    """t (B, n, n) as a view with rows padded to 16 bytes."""
    B, n, _ = t.shape
    full = torch.zeros((B, n, fw.padded(n)), dtype=t.dtype, device=t.device)
    full[:, :, :n] = t
    return full[:, :, :n]


def prepare(case, seed):
    kind, gen = case["kind"], _gen(seed)
    if kind == "solve":
        return dict(case=case, W=_weights(case, case["n"], gen))
    if kind == "host":
        n, shape = case["n"], (case["n"], fw.padded(case["n"]))
        W = _weights(case, n, gen, device="cpu")
        D = torch.zeros(shape, dtype=torch.int32, pin_memory=True)[:, :n]
        P = torch.zeros(shape, dtype=torch.int32, pin_memory=True)[:, :n] if case["pred"] else None
        return dict(case=case, W=W, D=D, P=P)
    if kind == "batched":
        # every graph in one slab, so that a new batch arrives by one copy
        ns = _sizes(case)
        lds = [fw.padded(n) for n in ns]
        ends = np.cumsum([n * ld for n, ld in zip(ns, lds)])
        W = torch.zeros(int(ends[-1]), dtype=DTYPES[case["dtype"]], device="cuda")
        D, P = torch.zeros_like(W), torch.zeros(W.shape, dtype=torch.int32, device="cuda")
        dists, preds = [], []
        for n, ld, end in zip(ns, lds, ends):
            at = slice(int(end) - n * ld, int(end))
            W[at].view(n, ld)[:, :n] = _weights(case, n, gen)
            dists.append(D[at].view(n, ld)[:, :n])
            preds.append(P[at].view(n, ld)[:, :n])
        code = fw.FW_I32 if case["dtype"] == "i32" else fw.FW_F32
        plan = fw.BatchedPlan(ns, lds, code)
        return dict(case=case, W=W, D=D, P=P, dists=dists, preds=preds if case["pred"] else None,
                    plan=plan)
    if kind == "intermediate":
        _, P = fw.solve(_weights(case, case["n"], gen))
        return dict(case=case, P=P)
    W = _batch_weights(case, gen)
    G = torch.randn(W.shape, generator=gen, device="cuda")
    if kind == "train":
        return dict(case=case, W=W.requires_grad_(), G=G)
    with torch.no_grad():
        D, P = fw_autograd.shortest_paths(W)
    return dict(case=case, G=_strided(G), D=_strided(D), P=_strided(P))


def run(state):
    kind = state["case"]["kind"]
    if kind == "solve":
        D, P = fw.solve(state["W"], with_pred=state["case"]["pred"])
        return {"dist": D, "pred": P}
    if kind == "host":
        fw.fw_solve_host_io(state["W"], state["D"], state["P"])
        return {"dist": state["D"], "pred": state["P"]}
    if kind == "batched":
        state["D"].copy_(state["W"])
        state["plan"].solve(state["dists"], state["preds"])
        return {"dist": state["D"], "pred": state["P"] if state["case"]["pred"] else None}
    if kind == "intermediate":
        return {"mid": fw.fw_intermediate(state["P"])}
    if kind == "train":
        D, P = fw_autograd.shortest_paths(state["W"])
        (grad,) = torch.autograd.grad(D, state["W"], state["G"])
        return {"dist": D, "pred": P, "grad": grad}
    grad = torch.empty_strided(state["G"].shape, state["G"].stride(), device="cuda")
    fw.fw_backward_strided(state["G"], state["D"], state["P"], grad)
    return {"grad": grad}


def work(case):
    """Two operations (add, min) per relaxation, n^3 relaxations per solve;
    weights in, distances and predecessors out (the backward: dL/dD and the
    predecessors in, dL/dW out, an add per entry along the tree and one into
    its edge)."""
    kind, size = case["kind"], 8 if case["dtype"] in ("i64", "f64") else 4
    if kind == "batched":
        ns = _sizes(case)
        return {"bytes": float(sum(n * n for n in ns)) * (2 * size + 4 * case["pred"]),
                "flops": 2.0 * sum(n**3 for n in ns)}
    n2 = float(case["n"]) ** 2 * case.get("batch", 1)
    if kind == "intermediate":
        return {"bytes": 8 * n2, "flops": n2}
    if kind == "backward":
        return {"bytes": 12 * n2, "flops": 2 * n2}
    if kind == "train":  # W and dL/dD in; distances, predecessors and dL/dW out
        return {"bytes": 20 * n2, "flops": 2 * n2 * case["n"] + 2 * n2}
    return {"bytes": n2 * (2 * size + 4 * case["pred"]), "flops": 2 * n2 * case["n"]}


# ------------------------------------------------------- 64-bit references ---

def _plain_fw(W, pred):
    """Floyd-Warshall of (B, n, n) fp64 weights, one vertex at a time: distances
    and, if asked for, the last hops (strict improvement)."""
    B, n, _ = W.shape
    D, P, via = W.clone(), None, torch.empty_like(W)
    if pred:
        rows = torch.arange(n, dtype=torch.int32, device=W.device).view(1, n, 1).expand(B, n, n)
        eye = torch.eye(n, dtype=torch.bool, device=W.device)
        P = torch.where(torch.isfinite(W) & ~eye, rows, torch.full_like(rows, -1))
    for k in range(n):
        torch.add(D[:, :, k:k + 1], D[:, k:k + 1, :], out=via)
        if pred:
            P = torch.where(via < D, P[:, k:k + 1, :], P)
        torch.minimum(D, via, out=D)
    return D, P


def _plain_grad(G, D, P):
    """dL/dW of dL/dD = G through the trees of P, in fp64: every source's
    vertices from the farthest inwards add their subtree's sum to their last
    hop's, then each sum goes to the edge it arrived by."""
    B, n, _ = D.shape
    P = P.reshape(B * n, n).long()
    tree = P >= 0
    E = torch.where(tree, G.double().reshape(B * n, n), torch.zeros((), dtype=torch.float64,
                                                                    device=G.device))
    far = torch.where(tree, D.reshape(B * n, n), torch.full((), -1.0, dtype=torch.float64,
                                                            device=D.device))
    order = torch.argsort(far, dim=1, descending=True)
    rows = torch.arange(B * n, device=D.device)
    for t in range(n):
        v = order[:, t]
        hop = P[rows, v]
        add = torch.where(hop >= 0, E[rows, v], torch.zeros_like(E[:, 0]))
        E[rows, hop.clamp(min=0)] += add
    E = torch.where(tree, E, torch.zeros_like(E)).view(B, n, n)
    grad = torch.zeros((B, n, n), dtype=torch.float64, device=D.device)
    grad.scatter_add_(1, P.clamp(min=0).view(B, n, n), E)
    return grad


def exact(case, seed):
    """The floating-point outputs in 64 bits (whole numbers have one value only)."""
    kind, gen = case["kind"], _gen(seed)
    if case["dtype"] not in ("f32", "f64") or kind == "batched":
        return None
    if kind == "solve":
        D, _ = _plain_fw(_weights(case, case["n"], gen).double().unsqueeze(0), False)
        return {"dist": D[0], "pred": None}
    W = _batch_weights(case, gen)
    G = torch.randn(W.shape, generator=gen, device="cuda")
    D, P = _plain_fw(W.double(), True)
    grad = _plain_grad(G, D, P)
    return {"dist": D, "pred": None, "grad": grad} if kind == "train" else {"grad": grad}
