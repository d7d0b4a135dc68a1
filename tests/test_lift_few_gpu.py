"""The lift on both sides of the line between an element per thread and the
table kernel: the same bits from a plan of few pairs and from one of many that
holds the same pairs, over element counts around a block of 256, windows of one
beam and of the widest, M above N, and against FP64.

Tolerance: a W-term Horner sum of FP32 FMAs, W 2^-24 of each term's magnitude,
doubled for the two twiddles."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,T,L,W", [(1, 32, 100, 128, 1), (4, 16, 100, 256, 9), (48, 64, 100, 128, 3), (100, 128, 100, 128, 32),
                                       (256, 256, 64, 256, 5), (257, 512, 40, 256, 9), (700, 1024, 20, 256, 9), (1024, 1024, 10, 256, 16),
                                       (1025, 2048, 8, 256, 2)])
def test_few_and_many_pairs_agree(N, M, T, L, W):
    kw = dict(N=N, F=4 * L, L=L, M=M, u=np.sin(np.linspace(-0.9, 0.9, T)), W=[W] * T, K=[4] * T, P_train=1, P_test=0, fc=10e9,
              fs=1e9, fd=10e9, delta=10.0)
    whole, part = P.Plan(**kw), P.Plan(s_begin=1, s_count=1, **kw)
    g = torch.Generator(device="cuda").manual_seed(N + W)
    c = torch.view_as_complex(torch.randn(T, L, W, 2, generator=g, device="cuda"))
    ch = torch.full((T * L * N + 4,), 3.0, dtype=torch.complex64, device="cuda")
    cp = torch.full((T * N + 4,), 3.0, dtype=torch.complex64, device="cuda")
    P.bs_lift(whole, c.reshape(-1), ch)
    P.bs_lift(part, c[:, 1].contiguous().reshape(-1), cp)
    torch.cuda.synchronize()
    assert (ch[T * L * N:] == 3.0).all() and (cp[T * N:] == 3.0).all()
    got = cp[:T * N].reshape(T, N)
    assert torch.equal(torch.view_as_real(ch[:T * L * N].reshape(T, L, N)[:, 1].contiguous()), torch.view_as_real(got))
    start = part.offsets()["start"]
    n = np.arange(N)
    for t in range(T):
        m = (start[t] + np.arange(W)) % M
        w = c[t, 1].cpu().numpy().astype(np.complex128)
        ref = (w[:, None] * np.exp(2j * np.pi * ((m[:, None] * n) % M) / M)).sum(0) / np.sqrt(M)
        assert np.abs(got[t].cpu().numpy() - ref).max() <= 2 * W * 2.0 ** -24 * np.abs(w).sum() / np.sqrt(M)
