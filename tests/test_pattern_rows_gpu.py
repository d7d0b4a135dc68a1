"""Beam patterns of correlators whose elements differ in scale by more than
FP32's exponents allow to be squared together: tapers that rise from almost
nothing, residues in front of a row, leading zeros before a tiny rest, ramps
over the whole exponent range, on both sides of the rule between the SIMT
kernel and the tensor-core tiles (by a factor of two or more in the pairs).

Tolerance, of a pattern's maximum of 1: that of the two kernels at these
sizes (2e-6 of the tiles; (N / 16 + 8) 2^-23 of the SIMT kernel's rotations)."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


def _rows(N):
    """[16][N] real envelopes."""
    n = np.arange(N)
    gauss = [np.exp(-0.5 * ((n - (N - 1) / 2) / (N * s)) ** 2) for s in (0.054, 0.049)]
    residue = np.where(n < 16, 1e-20, 1.0)
    zeros = np.where(n < 16, 0.0, 1e-30)
    up = 10.0 ** np.linspace(-37, 17, N)
    steps = np.where(n < N // 2, 1e-25, 1.0)
    rows = np.stack(gauss + [residue, zeros, up, up[::-1], steps, np.where(n == N - 1, 1e10, 1e-10)])
    return np.concatenate([rows, rows])


@pytest.mark.parametrize("N,L,D", [(1024, 128, 181), (1024, 2, 31), (100, 128, 100), (100, 4, 64), (37, 256, 193)])
def test_pattern_of_uneven_rows(N, L, D):
    env = _rows(N)
    T = len(env)
    M = 1 << (N - 1).bit_length()
    plan = P.Plan(N=N, F=max(16, 4 * L), L=L, M=M, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[3] * T, K=[4] * T, P_train=1, P_test=1,
                  fc=10e9, fs=1e9, fd=10e9, delta=10.0)
    rng = np.random.default_rng(N + L)
    ch = (env[:, None] * np.exp(2j * np.pi * rng.uniform(size=(T, L, N)))).astype(np.complex64)
    u = np.linspace(-1.0, 1.0, D)
    pat = torch.full((T * L * D + 8,), 3.0, device="cuda")
    P.bs_beam_pattern(plan, torch.from_numpy(ch.reshape(-1)).cuda(), torch.from_numpy(u).cuda(), pat)
    assert plan.device_status() == 0 and (pat[T * L * D:] == 3.0).all()
    p = pat[:T * L * D].cpu().numpy().reshape(T, L, D)
    assert np.isfinite(p).all()
    for s in {0, 1, L // 2, L - 1}:
        f = 10e9 + (((s - L // 2 + 1) - 0.5) / L) * 1e9
        e = np.exp(1j * np.pi * np.outer(np.arange(N), u * (f / 10e9)))
        c = ch[:, s].astype(np.complex128)
        c /= np.abs(c).max(axis=1, keepdims=True)
        ref = np.abs(c.conj() @ e) / (np.linalg.norm(c, axis=1, keepdims=True) * np.sqrt(N))
        assert np.abs(p[:, s] - ref).max() <= max(2e-6, (N / 16 + 8) * 2.0 ** -23)
