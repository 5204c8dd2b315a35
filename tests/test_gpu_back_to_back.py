"""Calls back to back on one stream over one workspace, inputs changing from call to call.
The kernels of a call overlap at their ends and the next call begins while the last one
drains: each output has to be, bit for bit, what the same call gives by itself."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev
from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300 import inputs

pytestmark = pytest.mark.gpu

CALLS = 60


def call(kind, X, d, ws, H):
    if kind == "layer":
        B.bigcn_layer_forward(X, d["s"], d["t"], d["W"], d["rowptr"], d["colidx"], ws, H)
    elif kind == "static":
        B.bigcn_layer_forward_static(X, d["s"], d["t"], d["W"], d["rowptr"], d["colidx"], H)
    elif kind == "weighted":
        B.bigcn_weighted_layer_forward(X, d["s"], d["t"], d["W"], d["rowptr"], d["colidx"], d["v"],
                                       ws, H)
    elif kind == "forward":
        B.bigcn_forward_2layer(X, d["s"], d["t"], d["W"], d["W2"], d["rowptr"], d["colidx"], ws, H)
    else:
        B.bigcn_inductive_layer_forward(kind, X, d["s"], d["t"], d["W"], d["rowptr"], d["colidx"],
                                        ws, H, W_neigh=d["Wn"] if kind == "sage" else None)


# The fronts, the CUDA-core and the tcgen05 products, uint16 and fp32 rows, the second kernel
@pytest.mark.parametrize("N,K,F", [(301, 203, 19), (2708, 1433, 64), (5000, 300, 64),
                                   (152 * 128 + 77, 300, 40), (3000, 3100, 48), (200, 33000, 8),
                                   (66003, 200, 64)])
@pytest.mark.parametrize("kind", ["layer", "static", "weighted", "mean", "sage", "forward"])
def test_calls_overlap(cuda_device, kind, N, K, F):
    c = inputs.layer_case(N, K, F, seed=N + K, mean_degree=6.0, hub_degree=min(N // 3, 900))
    d = {k: to_dev(x) for k, x in c.items()}
    d["v"] = to_dev(inputs.edge_weights(c["rowptr"], c["colidx"], 5))
    d["Wn"], d["W2"] = to_dev(inputs.weights(K, F, 7)), to_dev(inputs.weights(F, 5, 8))
    size = {"layer": B.bigcn_layer_workspace_bytes(N, K, F),
            "static": B.bigcn_layer_workspace_bytes(N, K, F),
            "weighted": B.bigcn_weighted_layer_workspace_bytes(N, K, F),
            "forward": B.bigcn_forward_2layer_workspace_bytes(N, K, F, 5)}.get(kind)
    if size is None:
        size = B.bigcn_inductive_layer_workspace_bytes(kind, N, K, F)
    if kind == "static" and size > B.STATIC_SCRATCH_BYTES:
        pytest.skip("does not fit the static scratch")
    ws = torch.full((size,), 0xAB, dtype=torch.uint8, device=cuda_device)
    out = 5 if kind == "forward" else F
    # Inputs unlike one another: other signs, other scales, and (K >= 258) every row wide.
    Xs = [d["X"], -2.0 * d["X"].roll(1, 0), 0.25 * d["X"].roll(3, 1)]
    cols = torch.arange(N, device=cuda_device) % F
    Xs.append(d["X"].abs() * torch.where(d["W"].t()[cols] >= 0, 1.0, -1.0) + d["t"] * 0)
    alone = []
    for X in Xs:
        H = torch.full((N, out), float("nan"), device=cuda_device)
        call(kind, X, d, ws, H)
        torch.cuda.synchronize()
        alone.append(H)
        assert torch.isfinite(H).all()
    Hs = [torch.full((N, out), float("nan"), device=cuda_device) for _ in range(CALLS)]
    order = np.random.default_rng(N).integers(0, len(Xs), CALLS)
    torch.cuda.synchronize()
    for H, q in zip(Hs, order):
        call(kind, Xs[q], d, ws, H)
    torch.cuda.synchronize()
    assert B.device_timeouts() == 0
    for i, (H, q) in enumerate(zip(Hs, order)):
        assert torch.equal(H, alone[q]), f"call {i} (input {q})"
