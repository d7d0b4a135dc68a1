"""The channeliser's tiles: few records of a small array, widths that end inside
a tile, more tiles than CTAs, and shards of one to four bins per record (whose
rows may start off the 128-byte boundary of a tensor store), against the FP64
FFT.

Tolerance: log2(F) butterfly levels of FP32 with table twiddles, below 2e-6 of a
record's largest element norm (FFT_TOL of the parity tests: 5e-6)."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,F,L,recs,shard", [
    (64, 512, 16, 12, None), (2, 512, 16, 1, None), (18, 512, 512, 3, None), (30, 1024, 64, 5, None),
    (6, 1024, 16, 151, None), (250, 512, 16, 9, None), (64, 512, 512, 4, (5, 1)), (64, 512, 512, 4, (6, 2)),
    (64, 1024, 1024, 3, (7, 1)), (64, 512, 128, 4, (9, 1)), (8, 2048, 2048, 2, (3, 1)), (8, 2048, 1024, 2, (3, 1)),
    (8, 2048, 512, 2, (4, 2))])
def test_channelised_bins(N, F, L, recs, shard):
    kw = dict(s_begin=shard[0], s_count=shard[1]) if shard else {}
    M = max(16, 1 << (N - 1).bit_length())
    plan = P.Plan(N=N, F=F, L=L, M=M, u=[0.1], W=[1], K=[1], P_train=recs, P_test=0, fc=10e9, fs=1e9, fd=10e9, delta=1.0,
                  **kw)
    s0, Ls = shard if shard else (0, L)
    B = F // L
    g = torch.Generator(device="cuda").manual_seed(N + F)
    x = torch.view_as_complex(torch.randn(recs * F * N, 2, generator=g, device="cuda"))
    xc = torch.full((recs * F * N + 4,), 9.0, dtype=torch.complex64, device="cuda")
    P.bs_channelize(plan, x, xc)
    assert plan.device_status() == 0
    n = recs * Ls * B * N
    assert (xc[n:] == 9.0).all()
    X = np.fft.fft(x.cpu().numpy().astype(np.complex128).reshape(recs, F, N), axis=1, norm="ortho")
    q = (np.arange(s0 * B, (s0 + Ls) * B) - F // 2) % F
    ref = X[:, q]
    got = xc[:n].cpu().numpy().reshape(recs, Ls * B, N)
    scale = np.linalg.norm(X, axis=1).max()
    assert np.abs(got - ref).max() <= 2e-6 * scale
