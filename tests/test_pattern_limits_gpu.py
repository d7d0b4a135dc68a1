"""Beam patterns around the SIMT kernel's shared-memory limit: element plus
direction counts whose range of directions, rounded up to whole warps' passes,
reaches 48 KB with more pairs than the directions are split for.

Tolerance: that of the SIMT kernel's rotations, (N / 16 + 8) 2^-23 of a
pattern's maximum of 1 (2e-6 at least)."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,D", [(1024, 3, 5088), (1024, 3, 5120), (1024, 3, 5121), (2048, 3, 4096), (4096, 4, 2016),
                                   (4096, 4, 2017), (4096, 4, 2048), (4000, 4, 2120), (4090, 1, 2049)])
def test_pattern_at_the_shared_memory_limit(N, T, D):
    L = 128
    M = 1 << (N - 1).bit_length()
    plan = P.Plan(N=N, F=4 * L, L=L, M=M, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[3] * T, K=[4] * T, P_train=1, P_test=1,
                  fc=10e9, fs=1e9, fd=10e9, delta=10.0)
    g = torch.Generator(device="cuda").manual_seed(D)
    ch = torch.view_as_complex(torch.randn(T, L, N, 2, generator=g, device="cuda"))
    u = torch.linspace(-1.0, 1.0, D, dtype=torch.float64, device="cuda")
    pat = torch.full((T * L * D + 8,), 3.0, device="cuda")
    P.bs_beam_pattern(plan, ch.reshape(-1), u, pat)
    assert plan.device_status() == 0 and (pat[T * L * D:] == 3.0).all()
    p = pat[:T * L * D].cpu().numpy().reshape(T, L, D)
    for s in (0, L - 1):
        c = ch[:, s].cpu().numpy().astype(np.complex128)
        f = 10e9 + (((s - L // 2 + 1) - 0.5) / L) * 1e9
        e = np.exp(1j * np.pi * np.outer(np.arange(N), u.cpu().numpy() * (f / 10e9)))
        ref = np.abs(c.conj() @ e) / (np.linalg.norm(c, axis=1, keepdims=True) * np.sqrt(N))
        assert np.abs(p[:, s] - ref).max() <= max(2e-6, (N / 16 + 8) * 2.0 ** -23)
