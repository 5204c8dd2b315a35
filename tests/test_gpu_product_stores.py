"""GPU: the stores of the ablation products' unsplit tiles (one k-block, so no
cluster split) at every store width.
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
