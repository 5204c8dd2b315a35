"""GPU: the stores of the ablation products' unsplit tiles (one k-block, so no
cluster split) at every store width, and the weight gradient's contraction over
nodes at the edges of its tiles.
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import check_sum as check, to_dev
from paper_2010_07565_gb300 import binding as B
from paper_2010_07565_gb300 import inputs

pytestmark = pytest.mark.gpu


def features(N, K, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    return (1.5 * g.standard_normal((N, K)) + 0.2).astype(np.float32)


def strided(N, F, ldz, skip, dev):
    """An N x F view of row stride ldz that starts `skip` floats into its buffer."""
    buf = torch.full((skip + N * ldz,), -7.0, device=dev)
    return buf, buf[skip:].as_strided((N, F), (ldz, 1), skip)


# Row strides and starts that allow stores of 16, 8 and 4 bytes; columns that
# end inside a store, at a tile's edge and in a second or third column tile.
STORES = [(128, 64, 64, 0), (129, 66, 68, 0), (257, 602, 602, 0), (300, 255, 256, 2),
          (127, 257, 257, 0), (1, 5, 8, 1), (255, 130, 130, 4)]


@pytest.mark.parametrize("N,F,ldz,skip", STORES)
def test_unsplit_tiles_store_their_rows(cuda_device, N, F, ldz, skip):
    K = 50
    X = features(N, K, N + F)
    Wt = inputs.weights(K, F, seed=F)
    SB, beta = oracle.weight_binarize(Wt)
    beta32 = beta.astype(np.float32)
    ref, mag = oracle.real_binary_product(X, SB, beta32.astype(np.float64), with_absterm=True)
    buf, Z = strided(N, F, ldz, skip, cuda_device)
    B.bigcn_real_binary_gemm(to_dev(X), None, None, to_dev(oracle.pack(SB)), to_dev(beta32), Z)
    torch.cuda.synchronize()
    check(Z.cpu().numpy(), ref, mag, f"X W~ {N}x{F} stride {ldz}", nterms=K)
    rows = buf[skip:].view(N, ldz)
    assert torch.all(buf[:skip] == -7.0) and torch.all(rows[:, F:] == -7.0)

    SF, alpha = oracle.sign(X), oracle.row_scale(X).astype(np.float32)
    ref, mag = oracle.binary_real_product(SF, alpha.astype(np.float64), Wt, with_absterm=True)
    ws = torch.empty(B.bigcn_binary_real_gemm_workspace_bytes(K, F), dtype=torch.uint8,
                     device=cuda_device)
    buf, Z = strided(N, F, ldz, skip, cuda_device)
    B.bigcn_binary_real_gemm(to_dev(oracle.pack(SF)), to_dev(alpha), K, to_dev(Wt), ws, Z)
    torch.cuda.synchronize()
    check(Z.cpu().numpy(), ref, mag, f"H~ W {N}x{F} stride {ldz}", nterms=K)
    rows = buf[skip:].view(N, ldz)
    assert torch.all(buf[:skip] == -7.0) and torch.all(rows[:, F:] == -7.0)
    assert B.device_timeouts() == 0


# Nodes, features and columns at and one past their tiles of 64, 128 and 64 to 256.
GRADIENTS = [(63, 64, 64), (65, 65, 65), (193, 129, 129), (128, 31, 257), (4097, 97, 128)]


@pytest.mark.parametrize("N,K,F", GRADIENTS)
def test_weight_gradient_at_tile_edges(cuda_device, N, K, F):
    case = inputs.layer_case(N, K, F, seed=N + K, mean_degree=3.0, hub_degree=0)
    dH = np.random.Generator(np.random.PCG64(F)).standard_normal((N, F)).astype(np.float32)
    d = {k: to_dev(v) for k, v in case.items()}
    ws = torch.empty(B.bigcn_layer_backward_workspace_bytes(N, K, F), dtype=torch.uint8,
                     device=cuda_device)
    dW = torch.full((K, F), float("nan"), device=cuda_device)
    B.bigcn_layer_backward(d["X"], d["s"], d["t"], d["W"], d["rowptr"], d["colidx"], to_dev(dH),
                           ws, dW)
    torch.cuda.synchronize()
    ref = oracle.layer_backward(case["X"], case["W"], case["rowptr"], case["colidx"],
                                dH.astype(np.float64), case["s"], case["t"])
    scale = np.broadcast_to(ref["Wg_abs"] * (1.0 + ref["beta"]), dW.shape)
    check(dW.cpu().numpy().astype(np.float64), ref["dW"], scale, f"dW {N}x{K}x{F}", nterms=N + K)
    assert B.device_timeouts() == 0
