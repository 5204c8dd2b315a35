"""GPU row packing around the row counts where a warp goes from one row at a time
to two and to four together, against the oracle's signs and row scales.
"""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import to_dev
from paper_2010_07565_gb300 import binding as B

pytestmark = pytest.mark.gpu

PER_ROW = 4 * 8     # warps per SM that take several rows each


@pytest.mark.parametrize("K", [1, 65, 300, 513])
@pytest.mark.parametrize("together,extra", [(2, -1), (2, 0), (2, 1), (4, -1), (4, 0), (4, 3)])
@pytest.mark.parametrize("centred", [False, True])
def test_rows_packed_together(cuda_device, together, extra, K, centred):
    N = together * PER_ROW * torch.cuda.get_device_properties(0).multi_processor_count + extra
    g = np.random.Generator(np.random.PCG64(N + K))
    X = g.standard_normal((N, K)).astype(np.float32)
    s = (0.5 + g.random(K)).astype(np.float32) if centred else None
    t = g.standard_normal(K).astype(np.float32) if centred else None
    Y = oracle.centre(X, s, t) if centred else X
    words = (K + 63) // 64 + 1                      # one padding word a row
    bits = torch.full((N, words), -1, dtype=torch.int64, device=cuda_device)
    alpha = torch.full((N,), float("nan"), device=cuda_device)
    B.bigcn_pack_rows(to_dev(X), to_dev(s), to_dev(t), bits, alpha)
    torch.cuda.synchronize()
    got = bits.cpu().numpy().view(np.uint64)
    assert np.array_equal(got[:, :-1], np.asarray(oracle.pack(oracle.sign(Y))).view(np.uint64))
    assert not got[:, -1].any()
    # K fp32 roundings of a sum of non-negative terms, and the division's.
    assert np.allclose(alpha.cpu().numpy(), oracle.row_scale(Y), rtol=(K + 2) * 2.0 ** -24, atol=0)


@pytest.mark.parametrize("together", [1, 2, 4])
@pytest.mark.parametrize("K,words", [(64, 2), (33, 18), (65, 40), (300, 64)])
def test_rows_longer_than_their_signs(cuda_device, together, K, words):
    """Words past the signs are written as zeros however many a row has."""
    N = together * PER_ROW * torch.cuda.get_device_properties(0).multi_processor_count + 3
    X = np.random.default_rng(K).standard_normal((N, K)).astype(np.float32)
    bits = torch.full((N, words), -1, dtype=torch.int64, device=cuda_device)
    alpha = torch.full((N,), float("nan"), device=cuda_device)
    B.bigcn_pack_rows(to_dev(X), None, None, bits, alpha)
    got = bits.cpu().numpy().view(np.uint64)
    n = (K + 63) // 64
    assert np.array_equal(got[:, :n], np.asarray(oracle.pack(oracle.sign(X))).view(np.uint64))
    assert not got[:, n:].any()


@pytest.mark.parametrize("K", [2048, 2049, 2354])
@pytest.mark.parametrize("centred", [False, True])
@pytest.mark.parametrize("extra", [-1, 0, 3])
def test_long_rows_packed_four_together(cuda_device, K, centred, extra):
    """From 2048 features eight chunks of each row at a time, with a last, partial batch."""
    N = 4 * PER_ROW * torch.cuda.get_device_properties(0).multi_processor_count + extra
    gen = torch.Generator(device=cuda_device)
    gen.manual_seed(K)
    X = torch.randn((N, K), generator=gen, device=cuda_device)
    s = 0.5 + torch.rand(K, generator=gen, device=cuda_device) if centred else None
    t = torch.randn(K, generator=gen, device=cuda_device) if centred else None
    bits, alpha = B.pack_rows(X, s, t)
    rows = np.unique(np.concatenate([np.arange(9), np.arange(N - 9, N), np.arange(0, N, 97)]))
    cpu = lambda a: None if a is None else a.cpu().numpy()
    Y = oracle.centre(X[rows].cpu().numpy(), cpu(s), cpu(t)) if centred else X[rows].cpu().numpy()
    assert np.array_equal(bits.cpu().numpy().view(np.uint64)[rows],
                          np.asarray(oracle.pack(oracle.sign(Y))).view(np.uint64))
    assert np.allclose(alpha.cpu().numpy()[rows], oracle.row_scale(Y), rtol=(K + 2) * 2.0 ** -24,
                       atol=0)
