"""Beam patterns where the rule between the SIMT kernel and the tensor-core
tiles can go wrong: both sides of its line, direction counts around the SIMT
kernel's warps and ranges and the tile of 192, few and many elements, a shard.

Tolerance, of a pattern's maximum of 1: each rotation by 32 elements adds at
most 2^-22 to a steering value, N / 32 of them half of that on average over the
sum, (N / 32) 2^-23; the sum's N / 32 steps of two FMAs and the reduction add
(N / 32 + 8) 2^-23.  The tensor-core tiles stay below 2e-6."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


def _plan(N, T, L, **kw):
    M = 1 << max(4, (N - 1).bit_length())
    return P.Plan(N=N, F=max(16, 4 * L), L=L, M=M, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[3] * T, K=[4] * T, P_train=1,
                  P_test=1, fc=10e9, fs=1e9, fd=10e9, delta=10.0, **kw)


@pytest.mark.parametrize("N,T,L,D,scale", [
    (1, 1, 2, 1, 1.0), (31, 1, 2, 33, 1e-30), (48, 3, 16, 31, 1.0), (48, 16, 32, 31, 1.0), (48, 16, 32, 64, 1.0),
    (100, 12, 64, 32, 1e30), (129, 4, 8, 193, 1.0), (33, 65, 8, 65, 1.0), (1000, 3, 4, 700, 1.0), (16, 2, 2, 6128, 1.0),
    (16, 2, 2, 6129, 1.0)])
def test_pattern_paths_match_fp64(N, T, L, D, scale):
    whole = _plan(N, T, L)
    g = torch.Generator(device="cuda").manual_seed(N + D)
    ch = torch.view_as_complex(torch.randn(T, L, N, 2, generator=g, device="cuda") * scale)
    u = torch.linspace(-1.0, 1.0, D, dtype=torch.float64, device="cuda")
    pat = torch.full((T * L * D + 8,), 3.0, device="cuda")
    P.bs_beam_pattern(whole, ch.reshape(-1), u, pat)
    assert whole.device_status() == 0 and (pat[T * L * D:] == 3.0).all()
    p = pat[:T * L * D].cpu().numpy().reshape(T, L, D)
    c64 = ch.cpu().numpy().astype(np.complex128)
    for s in range(L):
        f = 10e9 + (((s - L // 2 + 1) - 0.5) / L) * 1e9
        e = np.exp(1j * np.pi * np.outer(np.arange(N), u.cpu().numpy() * (f / 10e9)))
        ref = np.abs(c64[:, s].conj() @ e) / (np.linalg.norm(c64[:, s], axis=1, keepdims=True) * np.sqrt(N))
        assert np.abs(p[:, s] - ref).max() <= max(2e-6, (N / 16 + 8) * 2.0 ** -23)
    part = _plan(N, T, L, s_begin=L // 2, s_count=L - L // 2)
    pp = torch.empty(T * (L - L // 2) * D, device="cuda")
    P.bs_beam_pattern(part, ch[:, L // 2:].contiguous().reshape(-1), u, pp)
    assert np.array_equal(pp.cpu().numpy().reshape(T, -1, D), p[:, L // 2:])
