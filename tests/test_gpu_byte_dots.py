"""Layers whose product stays factored in byte planes: a dot is 2 v + (K & 1), v
in one byte where it fits and in two for the rows marked wide. Rows planted at
dots of +-K (wide from K = 258 on: v reaches 128 at dot 256) among ordinary ones,
at the widths where a 16-feature tile, a column slab or a staged row's chunk
count ends, through the kernels that write the planes (the split and whole-row
fronts, the CUDA-core and the tcgen05 product) and both window forms of the
aggregation that reads them (one long row, eight short ones, heavy rows)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import check_sum, to_dev
from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300 import inputs

pytestmark = pytest.mark.gpu


def planted_case(N, K, F, deg, hub, every, seed):
    """A layer case in which every ``every``-th row of X has the signs of a weight
    column, or their opposites (dots +-K with that column)."""
    c = inputs.layer_case(N, K, F, seed=seed, mean_degree=deg, hub_degree=hub, centred=False)
    rows = np.arange(0, N, every)
    cols = rows // every % F
    sign = np.where(rows // every % 2 == 0, 1.0, -1.0).astype(np.float32)
    c["X"][rows] = np.abs(c["X"][rows]) * np.where(c["W"].T[cols] >= 0, 1, -1) * sign[:, None]
    return c


def sampled(N, n, seed):
    if N <= n:
        return np.arange(N)
    g = np.random.default_rng(seed)
    return np.unique(np.concatenate([np.arange(9), np.arange(N - 9, N),
                                     g.choice(N, size=n, replace=False)]))


# (N, K, F, mean degree, hub, a planted row every)
LAYERS = [
    (700, 257, 1, 4.0, 0, 3),           # whole-row front, one-row windows; dots fit a byte
    (700, 258, 15, 4.0, 90, 3),         # the first wide dots
    (3000, 511, 16, 6.0, 0, 2),         # eight-row windows
    (3000, 512, 17, 6.0, 400, 1),       # every row wide, a heavy row
    (1100, 300, 64, 90.0, 0, 5),        # long rows
    (1100, 2047, 65, 90.0, 900, 5),     # split front, five tiles in eight chunks
    (1100, 2048, 128, 70.0, 0, 7),
    (2000, 254, 256, 70.0, 0, 4),       # CUDA-core product in column tiles: never wide
    (2500, 3072, 64, 9.0, 0, 4),        # CUDA-core product, wide
    (152 * 128 + 77, 130, 33, 5.0, 0, 9),       # tcgen05 products
    (152 * 128 + 1, 1030, 128, 6.0, 500, 2),
    (152 * 128 + 200, 600, 144, 66.0, 0, 9),    # two column slabs of five tiles (one short)
    (152 * 128 + 77, 3072, 256, 70.0, 0, 50),   # warp-specialised product, two slabs
    (152 * 128 + 77, 700, 256, 70.0, 0, 50),    # two slabs, one-row windows
]


@pytest.mark.parametrize("N,K,F,deg,hub,every", LAYERS)
def test_layer_with_wide_rows(cuda_device, N, K, F, deg, hub, every):
    c = planted_case(N, K, F, deg, hub, every, seed=N + K + F)
    d = {k: to_dev(v) for k, v in c.items() if v is not None}
    ws = torch.full((B.bigcn_layer_workspace_bytes(N, K, F),), 0xAB, dtype=torch.uint8,
                    device=cuda_device)
    ldh = F + 1                          # odd: feature pairs of H unaligned
    H = torch.full((N, ldh), float("nan"), device=cuda_device)[:, :F]
    B.bigcn_layer_forward(d["X"], None, None, d["W"], d["rowptr"], d["colidx"], ws, H)
    torch.cuda.synchronize()
    assert B.device_timeouts() == 0
    rows = sampled(N, 600, K)
    ref = oracle.layer_forward(c["X"], c["W"], c["rowptr"], c["colidx"], rows=rows)
    nterms = int(np.diff(c["rowptr"])[rows].max()) + 1
    check_sum(H.cpu().numpy()[rows], ref["H"], ref["absterm"],
              f"layer with wide rows {N}x{K}x{F}", nterms)


# (N, K, Fh, Fo, mean degree): row scales kept in the rows' padding or apart (Fo mod 16)
FORWARDS = [(900, 602, 128, 41, 5.0), (900, 1433, 64, 12, 90.0), (3100, 602, 127, 13, 6.0),
            (3100, 300, 33, 64, 80.0), (30000, 500, 64, 3, 4.0), (30000, 258, 20, 48, 4.0)]


@pytest.mark.parametrize("N,K,Fh,Fo,deg", FORWARDS)
def test_forward_with_wide_rows(cuda_device, N, K, Fh, Fo, deg):
    c = planted_case(N, K, Fh, deg, 300, 4, seed=N + K + Fo)
    W2 = inputs.weights(Fh, Fo, seed=N + 1)
    d = {k: to_dev(v) for k, v in c.items() if v is not None}
    ws = torch.full((B.bigcn_forward_2layer_workspace_bytes(N, K, Fh, Fo),), 0xAB,
                    dtype=torch.uint8, device=cuda_device)
    H1 = torch.full((N, Fh), float("nan"), device=cuda_device)
    out = torch.full((N, Fo), float("nan"), device=cuda_device)
    pred = torch.full((N,), -1, dtype=torch.int32, device=cuda_device)
    B.bigcn_forward_2layer(d["X"], None, None, d["W"], to_dev(W2), d["rowptr"], d["colidx"], ws,
                           out, H1=H1, pred=pred)
    torch.cuda.synchronize()
    r1 = oracle.layer_forward(c["X"], c["W"], c["rowptr"], c["colidx"])
    n = int(np.diff(c["rowptr"]).max()) + 1
    check_sum(H1.cpu().numpy(), r1["H"], r1["absterm"], f"wide rows H1 {N}x{K}x{Fh}", n)
    # Layer 2 on the GPU's own H1 (signs of values within rounding of zero may differ).
    r2 = oracle.layer_forward(H1.cpu().numpy(), W2, c["rowptr"], c["colidx"])
    check_sum(out.cpu().numpy(), r2["H"], r2["absterm"], f"wide rows logits {N}x{K}x{Fo}", n)
    assert np.array_equal(pred.cpu().numpy(), out.cpu().numpy().argmax(1))


# The other aggregators over the same planes: (N, K, F, mean degree, hub, planted every)
AGGREGATORS = [
    (700, 258, 5, 4.0, 90, 3),          # fronts, GraphSAGE's halves padded from 5 to 16
    (3000, 511, 50, 6.0, 400, 2),       # eight-row windows, a heavy row
    (1100, 300, 64, 90.0, 900, 5),      # one-row windows
    (700, 200, 100, 4.0, 90, 3),        # weighted: the CUDA-core product in column tiles
    (152 * 128 + 77, 1030, 100, 6.0, 0, 9),     # tcgen05 products (two halves: 224 columns)
    (152 * 128 + 77, 600, 144, 70.0, 0, 9),     # two column slabs (GraphSAGE: uint16 dots)
]


@pytest.mark.parametrize("N,K,F,deg,hub,every", AGGREGATORS)
@pytest.mark.parametrize("agg", ["mean", "sage", "weighted"])
def test_aggregators_with_wide_rows(cuda_device, agg, N, K, F, deg, hub, every):
    c = planted_case(N, K, F, deg, hub, every, seed=N + K + F)
    rp, ci = c["rowptr"], c["colidx"]
    d = {k: to_dev(v) for k, v in c.items() if v is not None}
    H = torch.full((N, F), float("nan"), device=cuda_device)
    rows = sampled(N, 600, K)
    if agg == "weighted":
        vals = inputs.edge_weights(rp, ci, K)
        vals[::7] = 0.0
        ws = torch.full((B.bigcn_weighted_layer_workspace_bytes(N, K, F),), 0xAB,
                        dtype=torch.uint8, device=cuda_device)
        B.bigcn_weighted_layer_forward(d["X"], None, None, d["W"], d["rowptr"], d["colidx"],
                                       to_dev(vals), ws, H)
        ref = oracle.layer_forward_weighted(c["X"], c["W"], rp, ci, vals, rows=rows)
    else:
        Wn = inputs.weights(K, F, seed=K + F) if agg == "sage" else None
        ws = torch.full((B.bigcn_inductive_layer_workspace_bytes(agg, N, K, F),), 0xAB,
                        dtype=torch.uint8, device=cuda_device)
        B.bigcn_inductive_layer_forward(agg, d["X"], None, None, d["W"], d["rowptr"],
                                        d["colidx"], ws, H, W_neigh=to_dev(Wn))
        ref = oracle.layer_forward_inductive(c["X"], c["W"], rp, ci, agg, W_neigh=Wn, rows=rows)
    torch.cuda.synchronize()
    assert B.device_timeouts() == 0
    check_sum(H.cpu().numpy()[rows], ref["H"], ref["absterm"],
              f"{agg} layer with wide rows {N}x{K}x{F}", int(np.diff(rp)[rows].max()) + 2)
