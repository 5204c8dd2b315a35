"""Calls large enough that a second kernel stands by for data with many wide rows (byte
dots: see test_gpu_byte_dots.py), on both sides of the share from which it takes over: every
row wide, some, few (left to the tensor-core walk's own pass), none. And wide rows whose
halves lack one of the dot (odd K above 2048)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import check_sum, to_dev
from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300 import inputs
from paper_2010_07565_gb300.runner import GCN2Forward, fused_kernel_names
from test_gpu_byte_dots import planted_case, sampled

pytestmark = pytest.mark.gpu


def layer(dev, agg, c, seed):
    N, K = c["X"].shape
    F = c["W"].shape[1]
    rp, ci = c["rowptr"], c["colidx"]
    d = {k: to_dev(v) for k, v in c.items() if v is not None}
    H = torch.full((N, F), float("nan"), device=dev)
    rows = sampled(N, 500, seed)
    ws = lambda n: torch.full((n,), 0xAB, dtype=torch.uint8, device=dev)
    if agg == "weighted":
        v = inputs.edge_weights(rp, ci, seed)
        B.bigcn_weighted_layer_forward(d["X"], None, None, d["W"], d["rowptr"], d["colidx"],
                                       to_dev(v), ws(B.bigcn_weighted_layer_workspace_bytes(N, K, F)),
                                       H)
        ref = oracle.layer_forward_weighted(c["X"], c["W"], rp, ci, v, rows=rows)
    elif agg == "gcn":
        B.bigcn_layer_forward(d["X"], None, None, d["W"], d["rowptr"], d["colidx"],
                              ws(B.bigcn_layer_workspace_bytes(N, K, F)), H)
        ref = oracle.layer_forward(c["X"], c["W"], rp, ci, rows=rows)
    else:
        Wn = inputs.weights(K, F, seed=seed) if agg == "sage" else None
        B.bigcn_inductive_layer_forward(agg, d["X"], None, None, d["W"], d["rowptr"], d["colidx"],
                                        ws(B.bigcn_inductive_layer_workspace_bytes(agg, N, K, F)),
                                        H, W_neigh=to_dev(Wn))
        ref = oracle.layer_forward_inductive(c["X"], c["W"], rp, ci, agg, W_neigh=Wn, rows=rows)
    torch.cuda.synchronize()
    assert B.device_timeouts() == 0
    check_sum(H.cpu().numpy()[rows], ref["H"], ref["absterm"],
              f"{agg} layer, wide rows {N}x{K}x{F}", int(np.diff(rp)[rows].max()) + 2)


# (N, K, F, mean degree, hub): N F of 4 million and more; eight-row windows taken from one
# counter by persistent blocks that also walk the heavy rows, one-row windows, two column
# slabs, few features
SIZES = [(110011, 300, 47, 12.0, 900), (33001, 511, 127, 70.0, 3000), (30011, 600, 144, 70.0, 0),
         (281003, 260, 15, 3.0, 90)]


@pytest.mark.parametrize("agg", ["gcn", "mean", "sage", "weighted"])
@pytest.mark.parametrize("every", [1, 3, 100, 20000])
@pytest.mark.parametrize("N,K,F,deg,hub", SIZES)
def test_layer(cuda_device, agg, N, K, F, deg, hub, every):
    if agg == "sage" and F > 128:
        F = 128
    layer(cuda_device, agg, planted_case(N, K, F, deg, hub, every, seed=N + K + every), K + every)


@pytest.mark.parametrize("agg", ["gcn", "mean", "sage", "weighted"])
@pytest.mark.parametrize("N,K,F,deg", [(1500, 2049, 64, 80.0), (2500, 2305, 48, 6.0),
                                       (2500, 3071, 64, 6.0), (152 * 128 + 5, 2051, 64, 6.0)])
@pytest.mark.parametrize("every", [1, 7])
def test_odd_dots_beyond_fp16(cuda_device, agg, N, K, F, deg, every):
    layer(cuda_device, agg, planted_case(N, K, F, deg, 300, every, seed=N + K + every), K + every)


@pytest.mark.parametrize("N,K,Fh,Fo,deg,every", [
    (66003, 300, 64, 7, 6.0, 2), (66003, 300, 64, 16, 6.0, 100), (33001, 602, 127, 41, 70.0, 3),
    (33001, 602, 128, 64, 70.0, 1), (270001, 260, 16, 3, 3.0, 5), (66003, 300, 64, 7, 6.0, 30000)])
def test_forward(cuda_device, N, K, Fh, Fo, deg, every):
    c = planted_case(N, K, Fh, deg, 900, every, seed=N + K + Fo)
    W2 = inputs.weights(Fh, Fo, seed=N + 1)
    d = {k: to_dev(v) for k, v in c.items() if v is not None}
    ws = torch.full((B.bigcn_forward_2layer_workspace_bytes(N, K, Fh, Fo),), 0xAB,
                    dtype=torch.uint8, device=cuda_device)
    out = torch.full((N, Fo), float("nan"), device=cuda_device)
    pred = torch.full((N,), -1, dtype=torch.int32, device=cuda_device)
    for H1 in (None, torch.full((N, Fh), float("nan"), device=cuda_device)):
        B.bigcn_forward_2layer(d["X"], None, None, d["W"], to_dev(W2), d["rowptr"], d["colidx"],
                               ws, out, H1=H1, pred=pred)
        if H1 is None:
            first = out.clone()
    assert torch.equal(first, out)
    rows = sampled(N, 400, K)
    r1 = oracle.layer_forward(c["X"], c["W"], c["rowptr"], c["colidx"], rows=rows)
    n = int(np.diff(c["rowptr"]).max()) + 1
    check_sum(H1.cpu().numpy()[rows], r1["H"], r1["absterm"], f"many wide rows H1 {N}x{K}x{Fh}", n)
    # Layer 2 on the GPU's own H1 (signs of values within rounding of zero may differ).
    r2 = oracle.layer_forward(H1.cpu().numpy(), W2, c["rowptr"], c["colidx"], rows=rows)
    check_sum(out.cpu().numpy()[rows], r2["H"], r2["absterm"], f"many wide rows logits {N}x{Fo}", n)
    assert np.array_equal(pred.cpu().numpy(), out.cpu().numpy().argmax(1))


@pytest.mark.parametrize("N,F,deg,hub", [(66003, 64, 6.0, 400), (33001, 127, 70.0, 5000)])
@pytest.mark.parametrize("every", [1, 50, 40000])
def test_unlike_weights(cuda_device, N, F, deg, hub, every):
    """Rows of weights up to 1e20 apart: all (left to the second kernel), some, few; each
    column held to the magnitudes of its own terms."""
    K = 200
    c = inputs.layer_case(N, K, F, seed=N, mean_degree=deg, hub_degree=hub, centred=False)
    rp, ci = c["rowptr"], c["colidx"]
    v = inputs.edge_weights(rp, ci, 3)
    row = np.repeat(np.arange(N), np.diff(rp))
    g = np.random.default_rng(N)
    v = np.where(row % every == 0, v * 10.0 ** g.integers(-10, 11, len(v)), v).astype(np.float32)
    d = {k: to_dev(x) for k, x in c.items() if x is not None}
    H = torch.full((N, F), float("nan"), device=cuda_device)
    ws = torch.full((B.bigcn_weighted_layer_workspace_bytes(N, K, F),), 0xAB, dtype=torch.uint8,
                    device=cuda_device)
    B.bigcn_weighted_layer_forward(d["X"], None, None, d["W"], d["rowptr"], d["colidx"], to_dev(v),
                                   ws, H)
    # fp64 on the GPU, over the exact dots
    S = torch.where(d["X"] >= 0, 1.0, -1.0).double()
    Z = (S @ torch.where(d["W"] >= 0, 1.0, -1.0).double()) * d["X"].double().abs().mean(
        1, keepdim=True) * d["W"].double().abs().mean(0)
    A = torch.sparse_csr_tensor(d["rowptr"], d["colidx"].long(), to_dev(v).double(), (N, N))
    dinv = 1.0 / torch.sqrt(1.0 + A @ torch.ones((N, 1), dtype=torch.float64, device=cuda_device))
    ref = dinv * (Z * dinv + A @ (Z * dinv))
    mag = dinv * (Z.abs() * dinv + A @ (Z.abs() * dinv))
    n = int(np.diff(rp).max()) + 8
    bad = (H.double() - ref).abs() > n * (2.0 ** -23 * mag + 2.0 ** -149)
    assert not bool(bad.any()), int(bad.sum())


@pytest.mark.parametrize("power", [-37, 36])
def test_row_scales_at_the_ends_of_fp32(cuda_device, power):
    """The second kernel's weights are the row scales themselves."""
    N, K, F = 66003, 300, 64
    c = planted_case(N, K, F, 6.0, 400, 3, seed=5)
    c["X"] = (c["X"] * 10.0 ** power).astype(np.float32)
    if power > 0:               # (|y| sums of 300 terms and sums of dots stay finite)
        c["X"] *= 0.1
        c["W"] *= np.float32(1e-3)
    d = {k: to_dev(x) for k, x in c.items() if x is not None}
    H = torch.full((N, F), float("nan"), device=cuda_device)
    ws = torch.full((B.bigcn_layer_workspace_bytes(N, K, F),), 0xAB, dtype=torch.uint8,
                    device=cuda_device)
    B.bigcn_layer_forward(d["X"], None, None, d["W"], d["rowptr"], d["colidx"], ws, H)
    rows = sampled(N, 500, K)
    ref = oracle.layer_forward(c["X"], c["W"], c["rowptr"], c["colidx"], rows=rows)
    n = int(np.diff(c["rowptr"]).max()) + 8
    err = np.abs(H.cpu().numpy()[rows].astype(np.float64) - ref["H"])
    # (the oracle sums the row scale in fp64; products below the normal range lose bits)
    assert (err <= (n + K) * (2.0 ** -23 * ref["absterm"] + 2.0 ** -149)).all()


def test_forward_kernels_of_a_large_graph(cuda_device):
    """The stand-by kernel is timed, and counted, with the aggregation it stands by for."""
    N, K, Fh, Fo = 66003, 300, 64, 7
    assert fused_kernel_names(N, K, Fh, Fo) == fused_kernel_names(3000, K, Fh, Fo)
    c = inputs.layer_case(N, K, Fh, seed=4)
    m = GCN2Forward(N, K, Fh, Fo, len(c["colidx"]), cuda_device)
    m.load(X=to_dev(c["X"]), s=to_dev(c["s"]), t=to_dev(c["t"]), W1=to_dev(c["W"]),
           W2=to_dev(inputs.weights(Fh, Fo, 5)), rowptr=to_dev(c["rowptr"]),
           colidx=to_dev(c["colidx"]))
    events = [torch.cuda.Event(enable_timing=True, external=True)
              for _ in range(len(m.kernel_names) + 1)]
    m.capture(events)
    m.replay()
    torch.cuda.synchronize()
    assert all(a.elapsed_time(b) > 0 for a, b in zip(events, events[1:]))
