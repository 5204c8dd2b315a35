"""Aggregations over byte dots whose row scales or edge weights are unlike one another:
the tensor-core walk holds a weight as two fp16 parts on a scale of its output row, and
has to give what fp32 multiply-adds give. References in fp64 over the exact dots."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev
from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300 import inputs

pytestmark = pytest.mark.gpu

AGGS = ["gcn", "mean", "sage", "weighted"]


def reference(c, agg, v=None, Wn=None):
    """H, and the sum of the magnitudes of its terms."""
    X, rp, ci = c["X"].astype(np.float64), c["rowptr"], c["colidx"]
    N = len(rp) - 1
    row = np.repeat(np.arange(N), np.diff(rp))
    alpha = np.abs(c["X"]).mean(1, dtype=np.float32).astype(np.float64)[:, None]
    S = np.where(X >= 0, 1.0, -1.0)

    def zeta(W):
        return (S @ np.where(W >= 0, 1.0, -1.0)) * alpha * np.abs(W.astype(np.float64)).mean(0)

    a = np.ones(len(ci)) if v is None else v.astype(np.float64)
    deg = np.bincount(row, a, N)[:, None]
    Z = zeta(Wn if agg == "sage" else c["W"])
    out = []
    for z in (Z, np.abs(Z)):
        if agg in ("gcn", "weighted"):
            d = 1.0 / np.sqrt(1.0 + deg)
            s = z * d
            np.add.at(s, row, a[:, None] * (z * d)[ci])
            s = s * d
        else:
            s = z.copy() if agg == "mean" else np.zeros_like(z)
            np.add.at(s, row, z[ci])
            if agg == "mean":
                s = s / (1.0 + deg)
            else:
                self_ = zeta(c["W"])
                s = s / np.maximum(deg, 1.0) + (self_ if z is Z else np.abs(self_))
        out.append(s)
    return out


def run(c, agg, dev, v=None, Wn=None):
    N, K = c["X"].shape
    F = c["W"].shape[1]
    X, W, rp, ci = (to_dev(c[k]) for k in ("X", "W", "rowptr", "colidx"))
    H = torch.full((N, F), float("nan"), device=dev)
    ws = lambda n: torch.full((n,), 0xAB, dtype=torch.uint8, device=dev)
    if agg == "gcn":
        B.bigcn_layer_forward(X, None, None, W, rp, ci, ws(B.bigcn_layer_workspace_bytes(N, K, F)),
                              H)
    elif agg == "weighted":
        B.bigcn_weighted_layer_forward(X, None, None, W, rp, ci, to_dev(v),
                                       ws(B.bigcn_weighted_layer_workspace_bytes(N, K, F)), H)
    else:
        B.bigcn_inductive_layer_forward(agg, X, None, None, W, rp, ci, ws(
            B.bigcn_inductive_layer_workspace_bytes(agg, N, K, F)), H, W_neigh=to_dev(Wn))
    return H.cpu().numpy().astype(np.float64)


def make(N, K, F, deg, agg, seed):
    c = inputs.layer_case(N, K, F, seed=seed, mean_degree=deg, hub_degree=N // 3, centred=False)
    v = inputs.edge_weights(c["rowptr"], c["colidx"], seed) if agg == "weighted" else None
    Wn = inputs.weights(K, F, seed=seed + 1) if agg == "sage" else None
    return c, v, Wn


# One-row windows (long rows, few rows), eight-row windows, two column slabs (GraphSAGE
# of 144 features: uint16 dots on the CUDA cores)
SHAPES = [(700, 200, 40, 80.0), (3000, 200, 40, 6.0), (700, 200, 144, 80.0)]


@pytest.mark.parametrize("agg", AGGS)
@pytest.mark.parametrize("N,K,F,deg", SHAPES)
def test_infinite_row_scale(cuda_device, agg, N, K, F, deg):
    """A row whose mean |y| overflows has an infinite scale: where it is gathered, H is
    Inf of the dot's sign, or NaN where the dot is zero or two infinities cancel."""
    c, v, Wn = make(N, K, F, deg, agg, seed=N + F)
    c["X"][::61] = np.where(c["X"][::61] >= 0, 3e38, -3e38)
    with np.errstate(invalid="ignore", over="ignore"):
        ref, mag = reference(c, agg, v, Wn)
    got = run(c, agg, cuda_device, v, Wn)
    assert np.isinf(ref).any() and np.isnan(ref).any() and np.isfinite(ref).any()
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    inf = np.isinf(ref)
    assert np.array_equal(got[inf], ref[inf])
    ok = np.isfinite(ref)
    assert (np.abs(got[ok] - ref[ok]) <= 1e-5 * mag[ok] + 1e-30).all()


@pytest.mark.parametrize("agg", AGGS)
@pytest.mark.parametrize("N,K,F,deg", SHAPES)
@pytest.mark.parametrize("powers", [[-35], [-36], [-33, -34, -35, -36, -37]])
def test_tiny_row_scales(cuda_device, agg, N, K, F, deg, powers):
    """Row scales so small that the weights' power-of-two scale ends at a float's largest
    exponent (below 2^-113), alone and among larger ones that raise it."""
    c, v, Wn = make(N, K, F, deg, agg, seed=N + F + len(powers))
    p = np.asarray(powers)[np.arange(N) // 64 % len(powers)]
    c["X"] = (c["X"] * 10.0 ** p[:, None]).astype(np.float32)
    ref, mag = reference(c, agg, v, Wn)
    got = run(c, agg, cuda_device, v, Wn)
    # n additions, truncated (tensor cores) or rounded to 24 bits, and a few roundings of
    # the scales; what lies below the normal range loses bits, 2^-149 at each step
    n = np.diff(c["rowptr"]).max() + 8
    bad = np.abs(got - ref) > n * (2.0 ** -23 * mag + 2.0 ** -149)
    assert not bad.any(), (int(bad.sum()), got[bad][:4], ref[bad][:4])


# Weight ratios up to 10^(max - min) within a row
@pytest.mark.parametrize("agg", AGGS)
@pytest.mark.parametrize("N,K,F,deg", SHAPES + [(700, 600, 40, 80.0), (3000, 600, 128, 6.0)])
@pytest.mark.parametrize("powers", [[0, -8], [0, -10], [0, -12, -24], [30, -36], [35, 0, -35]])
def test_unlike_weights(cuda_device, agg, N, K, F, deg, powers):
    """Where the dots of a row's large neighbours are zero, the small ones' sum is all
    there is: each column is held to the magnitudes of its own terms."""
    c, v, Wn = make(N, K, F, deg, agg, seed=N + F + len(powers))
    g = np.random.default_rng(N)
    if K > 256:         # some wide rows
        r = np.arange(0, N, 5)
        c["X"][r] = np.abs(c["X"][r]) * np.where(c["W"].T[r % F] >= 0, 1, -1)

    def draw(n):                # few large ones
        return 10.0 ** np.asarray(powers)[
            np.where(g.random(n) < 0.03, 0, g.integers(1, len(powers), n))]

    if agg == "weighted" and max(powers) - min(powers) < 39:     # the edges' own weights
        v = (v * draw(len(v))).astype(np.float32)
    else:
        c["X"] = (c["X"] * draw(N)[:, None]).astype(np.float32)
    ref, mag = reference(c, agg, v, Wn)
    got = run(c, agg, cuda_device, v, Wn)
    n = np.diff(c["rowptr"]).max() + 8
    bad = np.abs(got - ref) > n * (2.0 ** -23 * mag + 2.0 ** -149)
    assert not bad.any(), (int(bad.sum()), got[bad][:4], ref[bad][:4])
