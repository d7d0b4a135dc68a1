"""Beam patterns on the tensor-core tiles, with pairs enough that the rule
takes them there (1.4 times its line or more): element counts around the
16-element stage and the 64-element chunk, odd rows, the first full workload's
N, targets around the 64-target tile, directions around 16, 64 and the tile of
192, correlators at extreme scales, a shard, and a NaN row staying its own.

Tolerance: the kernel's 2e-6 of a pattern's maximum of 1 (six products of a
split pair 2^-24, truncated steps of a chunk 2^-23 each, at most 16 chunks in
FP32, steering values of 4 roundings)."""
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
    (1, 65, 64, 17, 1.0), (15, 70, 64, 16, 1e-30), (17, 65, 64, 191, 1e18), (63, 64, 64, 192, 1.0), (65, 63, 64, 193, 1.0),
    (130, 129, 32, 385, 1e-18), (301, 37, 64, 181, 1.0), (512, 65, 64, 63, 1e30), (1023, 20, 64, 181, 1.0),
    (1024, 64, 16, 181, 1.0), (1024, 63, 64, 65, 1e-30)])
def test_pattern_tiles_match_fp64(N, T, L, D, scale):
    whole, part = _plan(N, T, L), _plan(N, T, L, s_begin=L // 2, s_count=L // 4)
    g = torch.Generator(device="cuda").manual_seed(N + D)
    ch = torch.view_as_complex(torch.randn(T, L, N, 2, generator=g, device="cuda") * scale)
    bad = L // 2 + 1
    ch[T - 2, bad, N // 2] = float("nan")
    u = torch.linspace(-1.0, 1.0, D, dtype=torch.float64, device="cuda")
    pat = torch.full((T * L * D + 8,), 3.0, device="cuda")
    P.bs_beam_pattern(whole, ch.reshape(-1), u, pat)
    assert whole.device_status() == 0 and (pat[T * L * D:] == 3.0).all()
    p = pat[:T * L * D].cpu().numpy().reshape(T, L, D)
    nan = np.zeros((T, L), bool)
    nan[T - 2, bad] = True
    assert np.array_equal(np.isnan(p).any(-1), nan) and np.isnan(p[T - 2, bad]).all()
    for s in sorted({0, 1, bad, L - 1}):
        f = 10e9 + (((s - L // 2 + 1) - 0.5) / L) * 1e9
        e = np.exp(1j * np.pi * np.outer(np.arange(N), u.cpu().numpy() * (f / 10e9)))
        ok = ~nan[:, s]
        c = ch[:, s].cpu().numpy().astype(np.complex128)[ok]
        ref = np.abs(c.conj() @ e) / (np.linalg.norm(c, axis=1, keepdims=True) * np.sqrt(N))
        assert np.abs(p[ok, s] - ref).max() <= 2e-6
    pp = torch.empty(T * (L // 4) * D, device="cuda")
    P.bs_beam_pattern(part, ch[:, L // 2:L // 2 + L // 4].contiguous().reshape(-1), u, pp)
    assert np.array_equal(pp.cpu().numpy().reshape(T, -1, D), p[:, L // 2:L // 2 + L // 4], equal_nan=True)
