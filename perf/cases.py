"""Performance cases: what programs have this framework do, through its public calls.

A case is one call (or the short chain of calls that a program makes per step) of the
Bi-GCN library at one size. ``listed()`` holds twelve of them, ``draw`` gives more of the
same kinds over the same ranges:

* ``forward``   the two-layer forward (runner.GCN2Forward), one pass over a whole graph as a
                transductive node classifier makes it; launched directly, or replayed as the
                CUDA graph that the runner captures; with and without predicted classes.
* ``layer``     one binarized layer with a caller's workspace: one step of a deeper model.
* ``static``    the same layer on the library's own scratch, for programs that may not
                allocate: small graphs, where the cost is launches and latency.
* ``weighted``  the layer over a weighted adjacency (similarity or interaction graphs).
* ``mean``, ``sage``  the inductive layers (neighbour mean, GraphSAGE-mean).
* ``backward``  one layer's back-propagation, the gradients of its weights and its input.
* ``weights``, ``features``  the ablation layers (one operand of the product kept real).
* ``steps``     the step calls one after another over weights packed once, as a program does
                that keeps its packed model and needs the intermediate results.

Inputs are drawn on the GPU from the seed: Gaussian features, sparse binary ones (bags of
words) or sparse exponential ones with normalised rows (tf-idf), centred by their own
batch-normalisation statistics; weights N(0, 1/K); symmetric graphs without self-loops, either
uniform or with power-law expected degrees.
"""
from __future__ import annotations

import math

import torch

from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300.runner import GCN2Forward

DEV = "cuda"
BN_EPS = 1e-5

# The largest listed layer: no drawn case has more features to read, or more entries to gather.
MAX_FEATURES = (1 << 20) * 4096
MAX_ENTRIES = 114_600_000


def listed():
    return [
        # The smallest call: a small graph with odd sizes in a serving loop that may not allocate.
        dict(name="static_small", kind="static", N=1001, K=203, F=19, degree=4.0, hub=60,
             features="normal"),
        # Transductive node classification on citation graphs (bag-of-words features), the sizes
        # of the paper's Cora, Citeseer and PubMed: a few tens of microseconds of work each.
        dict(name="forward_cora", kind="forward", N=2708, K=1433, F=64, out=7, degree=4.0,
             hub=168, features="binary", density=0.0127, replay=False, pred=True),
        dict(name="forward_citeseer", kind="forward", N=3327, K=3703, F=64, out=6, degree=2.8,
             hub=99, features="binary", density=0.0085, replay=True, pred=False),
        dict(name="forward_pubmed", kind="forward", N=19717, K=500, F=64, out=3, degree=4.5,
             hub=171, features="exp", density=0.10, replay=False, pred=False),
        # The same on a social graph of Reddit's size, 114.6 million CSR entries with hubs.
        dict(name="forward_reddit", kind="forward", N=232965, K=602, F=128, out=41, degree=491.9,
             hub=20000, features="normal", replay=True, pred=True),
        # One layer of a deeper model on a million nodes: narrow, and wide over long features.
        dict(name="layer_1m_512_64", kind="layer", N=1 << 20, K=512, F=64, degree=16.0, hub=0,
             features="normal"),
        dict(name="layer_1m_4096_256", kind="layer", N=1 << 20, K=4096, F=256, degree=16.0, hub=0,
             features="normal"),
        # A weighted graph of ordinary size with nothing a round number.
        dict(name="weighted_100k", kind="weighted", N=100003, K=300, F=100, degree=50.0, hub=3000,
             features="normal"),
        # GraphSAGE-mean's first layer on the social graph.
        dict(name="sage_reddit", kind="sage", N=232965, K=602, F=128, degree=491.9, hub=20000,
             features="normal"),
        # Training: one layer's backward on the social graph.
        dict(name="backward_reddit", kind="backward", N=232965, K=602, F=128, degree=491.9,
             hub=20000, features="normal"),
        # The paper's ablation: only the features binarized.
        dict(name="features_65k", kind="features", N=65521, K=1000, F=96, degree=16.0, hub=500,
             features="normal"),
        # Step by step over weights that were packed once.
        dict(name="steps_170k", kind="steps", N=169343, K=128, F=256, degree=13.8, hub=10000,
             features="normal"),
    ]


KINDS = ("forward", "forward", "forward", "layer", "layer", "static", "weighted", "mean", "sage",
         "backward", "weights", "features", "steps")


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(KINDS)
    N = _log_int(rng, 1000, 20000) if kind == "static" else _log_int(rng, 1000, 1 << 20)
    K = _log_int(rng, 64, 4096)
    F = _log_int(rng, 8, 128 if kind in ("forward", "static") else 256)
    K = max(16, min(K, MAX_FEATURES // N))
    # Node-classification graphs: sparse when they are small, up to hundreds of entries a row.
    top = 8.0 if N < 5000 else min(492.0, MAX_ENTRIES / N)
    degree = round(math.exp(rng.uniform(math.log(2.0), math.log(top))), 2)
    if N * degree * F > MAX_ENTRIES * 128:
        degree = round(MAX_ENTRIES * 128 / (N * F), 2)
    case = dict(kind=kind, N=N, K=K, F=F, degree=degree,
                hub=rng.choice([0, min(N // 4, int(40 * degree))]),
                features=rng.choice(["normal", "normal", "binary", "exp"]))
    if case["features"] != "normal":    # a dozen features or more in every node's bag
        case["density"] = round(max(rng.uniform(0.01, 0.1), 12.0 / K), 4)
    if kind == "forward":
        case.update(out=_log_int(rng, 2, 64), replay=rng.random() < 0.5, pred=rng.random() < 0.5)
    return case


# ------------------------------------------------------------------ inputs ----
def _features(c, g):
    """X (N x K) and its batch-normalisation affine (scale, shift)."""
    N, K = c["N"], c["K"]
    if c["features"] == "normal":
        X = torch.randn((N, K), generator=g, device=DEV)
    else:
        keep = torch.rand((N, K), generator=g, device=DEV) < c["density"]
        if c["features"] == "binary":
            X = keep.float()
        else:
            X = torch.empty((N, K), device=DEV).exponential_(generator=g) * keep
            X /= X.norm(dim=1, keepdim=True).clamp_min(1e-20)
        del keep
    rows = max(1, (1 << 26) // K)
    s1 = torch.zeros(K, dtype=torch.float64, device=DEV)
    s2 = torch.zeros(K, dtype=torch.float64, device=DEV)
    for r in range(0, N, rows):
        x = X[r:r + rows].double()
        s1 += x.sum(0)
        s2 += x.square().sum(0)
    mean = s1 / N
    s = 1.0 / torch.sqrt((s2 / N - mean * mean).clamp_min(0.0) + BN_EPS)
    return X, s.float(), (-mean * s).float()


def _graph(c, g):
    """Symmetric CSR without self-loops of about N * degree entries: uniform endpoints, or
    (hub > 0) endpoints drawn by power-law expected degrees of at most ``hub``."""
    N = c["N"]
    target = int(round(N * c["degree"] / 2))
    M = int(target * (1.12 if c["hub"] else 1.02)) + 64
    if c["hub"]:
        w = torch.rand(N, generator=g, device=DEV, dtype=torch.float64).pow(-1.0 / 1.5)
        for _ in range(20):
            w = torch.clamp(w * (c["degree"] / w.mean()), max=float(c["hub"]))
        cum = torch.cumsum(w, 0)
        cum /= cum[-1].clone()

        def ends():
            r = torch.rand(M, generator=g, device=DEV, dtype=torch.float64)
            return torch.searchsorted(cum, r).clamp_max(N - 1)
    else:
        def ends():
            return torch.randint(0, N, (M,), generator=g, device=DEV)
    u, v = ends(), ends()
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.unique((lo * N + hi)[lo != hi])
    del u, v, lo, hi
    if key.numel() > target:
        key = key[torch.randperm(key.numel(), generator=g, device=DEV)[:target]]
    lo, hi = key // N, key % N
    key = torch.sort(torch.cat([lo * N + hi, hi * N + lo]))[0]
    del lo, hi
    rows = key // N
    rowptr = torch.zeros(N + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=N), 0)
    return rowptr, (key - rows * N).to(torch.int32)


def _edge_weights(rowptr, colidx, g):
    """Symmetric weights between 0.5 and 2: a hash of the sum of the two ends' keys."""
    N = rowptr.numel() - 1
    key = torch.randint(0, 1 << 31, (N,), generator=g, device=DEV)
    row = torch.repeat_interleave(torch.arange(N, device=DEV), rowptr.diff())
    h = key[row] + key[colidx.long()]
    h = ((h ^ (h >> 16)) * 0x45D9F3B) & 0xFFFFFFFF
    h = ((h ^ (h >> 16)) * 0x45D9F3B) & 0xFFFFFFFF
    return 0.5 + 1.5 * ((h >> 8) & 0xFFFFFF).float() / float(1 << 24)


def _inputs(c, seed):
    """What both ``prepare`` and ``exact`` start from."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    d = {}
    d["X"], d["s"], d["t"] = _features(c, g)
    K, F = c["K"], c["F"]

    def weights(k, f):
        return torch.randn((k, f), generator=g, device=DEV) / math.sqrt(k)

    d["W"] = weights(K, F)
    d["rowptr"], d["colidx"] = _graph(c, g)
    kind = c["kind"]
    if kind == "forward":
        d["W2"] = weights(F, c["out"])
    if kind == "sage":
        d["W2"] = weights(K, F)
    if kind == "weighted":
        d["values"] = _edge_weights(d["rowptr"], d["colidx"], g)
    if kind == "backward":          # gradients of a mean loss: small against the clip at 1
        d["dH"] = torch.randn((c["N"], F), generator=g, device=DEV) * 1e-3
    return d


def _bytes(n):
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    c, d = case, _inputs(case, seed)
    N, K, F, kind = c["N"], c["K"], c["F"], c["kind"]
    d["case"] = c
    if kind == "forward":
        m = GCN2Forward(N, K, F, c["out"], d["colidx"].numel(), DEV)
        m.load(X=d.pop("X"), s=d.pop("s"), t=d.pop("t"), W1=d.pop("W"), W2=d.pop("W2"),
               rowptr=d.pop("rowptr"), colidx=d.pop("colidx"))
        d["model"] = m
        d["pred"] = torch.empty(N, dtype=torch.int32, device=DEV) if c["pred"] else None
        if c["replay"]:
            if c["pred"]:           # the runner's capture has no predictions: capture the call
                _launch(d)
                torch.cuda.synchronize()
                m.graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(m.graph):
                    _launch(d)
            else:
                m.capture()
        return d
    d["H"] = torch.empty((N, F), device=DEV)
    if kind == "layer":
        d["ws"] = _bytes(B.bigcn_layer_workspace_bytes(N, K, F))
    elif kind == "weighted":
        d["ws"] = _bytes(B.bigcn_weighted_layer_workspace_bytes(N, K, F))
    elif kind in ("mean", "sage"):
        d["ws"] = _bytes(B.bigcn_inductive_layer_workspace_bytes(kind, N, K, F))
    elif kind in ("weights", "features"):
        d["ws"] = _bytes(B.bigcn_layer_ablation_workspace_bytes(kind, N, K, F))
    elif kind == "backward":
        d["ws"] = _bytes(B.bigcn_layer_backward_workspace_bytes(N, K, F))
        d["dW"], d["dX"] = torch.empty((K, F), device=DEV), torch.empty((N, K), device=DEV)
    elif kind == "steps":
        d["wbits"], d["beta"] = B.pack_weights(d.pop("W"))
        d["bits"] = torch.empty((N, B.words_for(K)), dtype=torch.int64, device=DEV)
        d["alpha"], d["Z"] = torch.empty(N, device=DEV), torch.empty((N, F), device=DEV)
    return d


def _launch(d):
    m = d["model"]
    if d["pred"] is None:
        m.launch()
    else:
        B.bigcn_forward_2layer(m.X, m.s, m.t, m.W1, m.W2, m.rowptr, m.colidx, m.workspace,
                               m.logits, pred=d["pred"])


def run(d):
    kind = d["case"]["kind"]
    if kind == "forward":
        m = d["model"]
        if d["case"]["replay"]:
            m.replay()
        else:
            _launch(d)
        return {"logits": m.logits} if d["pred"] is None else {"logits": m.logits,
                                                               "pred": d["pred"]}
    X, s, t, rp, ci, H = d["X"], d["s"], d["t"], d["rowptr"], d["colidx"], d["H"]
    if kind == "layer":
        B.bigcn_layer_forward(X, s, t, d["W"], rp, ci, d["ws"], H)
    elif kind == "static":
        B.bigcn_layer_forward_static(X, s, t, d["W"], rp, ci, H)
    elif kind == "weighted":
        B.bigcn_weighted_layer_forward(X, s, t, d["W"], rp, ci, d["values"], d["ws"], H)
    elif kind in ("mean", "sage"):
        B.bigcn_inductive_layer_forward(kind, X, s, t, d["W"], rp, ci, d["ws"], H,
                                        W_neigh=d.get("W2"))
    elif kind in ("weights", "features"):
        B.bigcn_layer_forward_ablation(kind, X, s, t, d["W"], rp, ci, d["ws"], H)
    elif kind == "backward":
        B.bigcn_layer_backward(X, s, t, d["W"], rp, ci, d["dH"], d["ws"], d["dW"], dX=d["dX"])
        return {"dW": d["dW"], "dX": d["dX"]}
    elif kind == "steps":
        B.bigcn_pack_rows(X, s, t, d["bits"], d["alpha"])
        B.bigcn_xnor_gemm(d["bits"], d["alpha"], d["wbits"], d["beta"], d["case"]["K"], d["Z"])
        B.bigcn_spmm_norm(rp, ci, d["Z"], H)
        return {"bits": d["bits"], "alpha": d["alpha"], "Z": d["Z"], "H": H}
    return {"H": H}


def work(case):
    c = case
    N, K, F, kind = c["N"], c["K"], c["F"], c["kind"]
    nnz = 2 * int(round(N * c["degree"] / 2))
    b = 4 * N * K + 8 * K + 8 * (N + 1) + 4 * nnz           # features, affine, CSR
    f = 2 * N * K * F + 2 * (nnz + N) * F                   # product, aggregation
    if kind == "forward":
        b += 4 * K * F + 4 * F * c["out"] + 4 * N * c["out"] + (4 * N if c["pred"] else 0)
        f += 2 * N * F * c["out"] + 2 * (nnz + N) * c["out"]
        return {"bytes": b, "flops": f}
    b += 4 * K * F + 4 * N * F                              # weights, H (or dH)
    if kind == "weighted":
        b += 4 * nnz
    elif kind == "sage":
        b += 4 * K * F
        f += 2 * N * K * F
    elif kind == "backward":
        b += 4 * K * F + 4 * N * K
        f += 2 * N * K * F
    elif kind == "steps":
        words = (K + 63) // 64
        b += 8 * words * (N + F) + 4 * N + 4 * F + 4 * N * F - 4 * K * F
    return {"bytes": b, "flops": f}


def tolerance(case):
    # About four times the error measured against ``exact``. Sums of fp32 terms over exact
    # integer dots: 1e-7. A real operand of the product (fp32 in three bf16 parts): 3e-6; the
    # weight gradient, a sum over all nodes whose terms cancel: 2e-5. A two-layer forward
    # binarizes the hidden layer: where one of its N F sums is within rounding of zero (a few
    # 1e-7 of them), another order of the additions gives the other sign, which moves a dot of
    # about sqrt(F) by 2 in all of that node's logits: few values, but each by up to its size.
    kind = case["kind"]
    if kind == "forward":
        n = case["N"] * case["F"]
        return {"rel": min(0.02, 4.0 * math.sqrt((1.0 + 4e-7 * n) / n)), "max": 0.99,
                "differ": 1e-3}
    if kind == "backward":
        return {"rel": 1e-4, "max": 4e-3}
    if kind in ("weights", "features"):
        return {"rel": 1e-5, "max": 4e-4}
    return {"rel": 1e-6, "max": 4e-5}


# ------------------------------------------------- the same in 64-bit torch ----
def _sign(y):
    return torch.where(y >= 0, 1.0, -1.0).to(torch.float64)


def _product(X, s, t, Ws, weights_real=False, features_real=False):
    """zeta of Eqs. 10-12 for each weight matrix, rows in chunks, in 64 bits: the signs'
    product first (exact integers), then the row and column scales."""
    N, K = X.shape
    out = [torch.empty((N, W.shape[1]), dtype=torch.float64, device=DEV) for W in Ws]
    ops = [W.double() if weights_real else _sign(W) for W in Ws]
    col = [1.0 if weights_real else W.double().abs().mean(0) for W in Ws]
    rows = max(1, (1 << 27) // K)
    for r in range(0, N, rows):
        y = X[r:r + rows].double()
        if s is not None:
            y = y * s.double() + t.double()
        a = 1.0 if features_real else y.abs().mean(1, keepdim=True)
        if not features_real:
            y = _sign(y)
        for o, w, b in zip(out, ops, col):
            o[r:r + rows] = (y @ w) * a * b
    return out


def _aggregate(rowptr, colidx, Z, values=None, mode="gcn"):
    N = rowptr.numel() - 1
    vals = (torch.ones(colidx.numel(), dtype=torch.float64, device=DEV) if values is None
            else values.double())
    A = torch.sparse_csr_tensor(rowptr, colidx.long(), vals, (N, N))
    deg = (rowptr.diff().double() if values is None
           else (A @ torch.ones((N, 1), dtype=torch.float64, device=DEV)).squeeze(1))
    deg = deg.unsqueeze(1)
    if mode == "gcn":
        d = 1.0 / torch.sqrt(1.0 + deg)
        Zd = Z * d
        return d * (Zd + A @ Zd)
    if mode == "mean":
        return (Z + A @ Z) / (1.0 + deg)
    return (A @ Z) / deg.clamp_min(1.0)                     # GraphSAGE's neighbour mean


def exact(case, seed):
    c, d = case, _inputs(case, seed)
    X, s, t, W, rp, ci = d["X"], d["s"], d["t"], d["W"], d["rowptr"], d["colidx"]
    kind = c["kind"]
    if kind == "forward":
        H1 = _aggregate(rp, ci, _product(X, s, t, [W])[0])
        out = _aggregate(rp, ci, _product(H1, None, None, [d["W2"]])[0])
        return {"logits": out, "pred": out.argmax(1)} if c["pred"] else {"logits": out}
    if kind == "sage":
        zs, zn = _product(X, s, t, [W, d["W2"]])
        return {"H": zs + _aggregate(rp, ci, zn, mode="sage")}
    if kind == "backward":
        G = _aggregate(rp, ci, d["dH"].double())
        beta = W.double().abs().mean(0)
        dX = G @ (_sign(W) * beta).T
        dX = torch.where(dX.abs() < 1.0, dX, 0.0)
        dWt = torch.zeros(W.shape, dtype=torch.float64, device=DEV)
        rows = max(1, (1 << 27) // c["K"])
        for r in range(0, c["N"], rows):
            y = X[r:r + rows].double() * s.double() + t.double()
            dWt += (_sign(y) * y.abs().mean(1, keepdim=True)).T @ G[r:r + rows]
        sW = _sign(W)
        dW = sW * (dWt * sW).sum(0) / c["K"] + beta * dWt * (W.abs() < 1.0)
        return {"dW": dW, "dX": dX}
    Z = _product(X, s, t, [W], weights_real=kind == "features",
                        features_real=kind == "weights")[0]
    H = _aggregate(rp, ci, Z, d.get("values"), "mean" if kind == "mean" else "gcn")
    if kind == "steps":
        y = X.double() * s.double() + t.double()
        return {"bits": None, "alpha": y.abs().mean(1), "Z": Z, "H": H}
    return {"H": H}
