"""Column indices out of range: skipped, with the row's degree unchanged, where an
aggregation loads 32 entries at a time. Lists of 31 to 97 entries, whose blocks of 32
hold one bad index, all but one, or none but bad ones (the self-loop is the first
entry of a list, so index 31 of the CSR row begins its second block)."""
import numpy as np
import pytest
import torch

from gpu_helpers import check_sum, to_dev
from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300 import inputs

pytestmark = pytest.mark.gpu


def bad_graph(N, seed):
    """CSR with planted out-of-range columns, and the mask of the good entries."""
    g = np.random.default_rng(seed)
    lens = g.choice([0, 5, 31, 32, 40, 63, 64, 96], size=N)
    lens[:8] = [31, 32, 40, 63, 64, 95, 96, 97]
    rp = np.zeros(N + 1, np.int64)
    rp[1:] = np.cumsum(lens)
    ci = g.integers(0, N, size=rp[-1]).astype(np.int32)
    bad = [-1, N, -2 ** 31, 2 ** 31 - 1]
    for i in range(N):
        b, n = rp[i], lens[i]
        if n < 31:
            continue
        form = i % 4
        at = {0: [31], 1: range(31, min(n, 63)), 2: range(30, n - 1), 3: range(0, n)}[form]
        for q in at:
            if q < n:
                ci[b + q] = bad[(i + q) % 4]
    return rp, ci, (ci >= 0) & (ci < N)


def reference(rp, ci, good, Z):
    """D^-1/2 (A + I) D^-1/2 Z without the bad entries, degrees with them; and the
    sums of the terms' magnitudes."""
    N = len(rp) - 1
    row = np.repeat(np.arange(N), np.diff(rp))
    d = 1.0 / np.sqrt(1.0 + np.diff(rp))
    out = []
    for z in (Z * d[:, None], np.abs(Z) * d[:, None]):
        s = z.copy()
        np.add.at(s, row[good], z[ci[good]])
        out.append(s * d[:, None])
    return out


@pytest.mark.parametrize("F", [1, 41, 128, 256])
@pytest.mark.parametrize("prescaled", [False, True])
def test_fp32_rows(cuda_device, F, prescaled):
    N = 400
    rp, ci, good = bad_graph(N, F)
    Z = np.random.default_rng(F + 1).standard_normal((N, F)).astype(np.float32)
    ref, mag = reference(rp, ci, good, Z.astype(np.float64))
    H = torch.full((N, F), float("nan"), device=cuda_device)
    if prescaled:
        Zp = (Z / np.sqrt(1.0 + np.diff(rp))[:, None]).astype(np.float32)
        B.bigcn_spmm_prescaled(to_dev(rp), to_dev(ci), to_dev(Zp), H)
    else:
        B.bigcn_spmm_norm(to_dev(rp), to_dev(ci), to_dev(Z), H)
    check_sum(H, ref, mag, f"out-of-range columns, F={F}, prescaled={prescaled}", 98)


# K: byte planes on the tensor cores; uint16 dots on the CUDA cores
@pytest.mark.parametrize("K", [200, 3100])
@pytest.mark.parametrize("F", [16, 64, 128])
def test_layer(cuda_device, K, F):
    N = 400
    rp, ci, good = bad_graph(N, K + F)
    c = inputs.layer_case(N, K, F, seed=K + F, centred=False)
    S, SB = np.where(c["X"] >= 0, 1.0, -1.0), np.where(c["W"] >= 0, 1.0, -1.0)
    Z = (S @ SB) * np.abs(c["X"].astype(np.float64)).mean(1, keepdims=True) * np.abs(
        c["W"].astype(np.float64)).mean(0)
    ref, mag = reference(rp, ci, good, Z)
    ws = torch.empty(B.bigcn_layer_workspace_bytes(N, K, F), dtype=torch.uint8, device=cuda_device)
    H = torch.full((N, F), float("nan"), device=cuda_device)
    B.bigcn_layer_forward(to_dev(c["X"]), None, None, to_dev(c["W"]), to_dev(rp), to_dev(ci), ws, H)
    check_sum(H, ref, mag, f"out-of-range columns, layer K={K}, F={F}", 98)
