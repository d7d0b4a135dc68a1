"""Lifted outputs of short rows on both sides of the line between the SIMT
kernel and the tensor-core tiles: element counts around 32, 64 and 96, targets
and test vectors around the tiles' 32 and 64, one and several waves, a shard,
a NaN row staying its own; on the tiles (more than two waves of the other
kernel) also stage and chunk edges, odd rows and extreme scales.

Tolerance: FP32 sums of at most 97 complex products, or the tiles' 2e-6 of
||c|| ||y||: (2 * 97 + 2) 2^-24 < 2e-5 of the sum of magnitudes."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,L,B,P_te,scale", [
    (1, 1, 2, 16, 1, 1.0), (16, 33, 16, 16, 2, 1.0), (31, 64, 16, 16, 8, 1.0), (32, 65, 32, 16, 8, 1.0), (33, 3, 4, 8, 5, 1.0),
    (64, 64, 32, 16, 8, 1.0), (64, 64, 64, 16, 8, 1.0), (65, 31, 4, 16, 4, 1.0), (96, 32, 32, 16, 8, 1.0), (96, 33, 64, 16, 2, 1.0),
    (97, 5, 4, 16, 3, 1.0), (48, 128, 128, 4, 2, 1.0),
    (1, 65, 64, 16, 8, 1.0), (15, 63, 128, 16, 5, 1e-30), (17, 65, 64, 16, 9, 1e18), (33, 64, 64, 16, 8, 1.0), (65, 65, 64, 16, 8, 1.0)])
def test_short_rows_match_fp64(N, T, L, B, P_te, scale):
    M = 1 << max(4, (N - 1).bit_length())
    kw = dict(N=N, F=max(16, L * B), L=L, M=M, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[min(5, M)] * T, K=[B] * T, P_train=1,
              P_test=P_te, fc=10e9, fs=1e9, fd=10e9, delta=10.0)
    whole, part = P.Plan(**kw), P.Plan(s_begin=L // 2, s_count=L // 2, **kw)
    V = P_te * B
    g = torch.Generator(device="cuda").manual_seed(N + T)
    ch = torch.view_as_complex(torch.randn(T, L, N, 2, generator=g, device="cuda") * scale)
    xc = torch.view_as_complex(torch.randn(1 + P_te, L, B, N, 2, generator=g, device="cuda"))
    bad = T // 2, L - 1
    ch[bad] = float("nan")
    out = torch.full((T * L * V + 8,), 3.0, dtype=torch.complex64, device="cuda")
    P.bs_apply_lifted(whole, xc.reshape(-1), ch.reshape(-1), out)
    assert whole.device_status() == 0 and (out[T * L * V:] == 3.0).all()
    o = out[:T * L * V].cpu().numpy().reshape(T, L, V)
    nan = np.zeros((T, L), bool)
    nan[bad] = True
    assert np.array_equal(np.isnan(o).any(-1), nan) and np.isnan(o[bad]).all()
    c64, y64 = ch.cpu().numpy().astype(np.complex128), xc.cpu().numpy().astype(np.complex128)[1:]
    for s in range(L):
        y = y64[:, s].reshape(V, N)
        ok = ~nan[:, s]
        bound = 2e-5 * (np.abs(c64[ok, s]) @ np.abs(y).T) + 1e-30
        assert (np.abs(o[ok, s] - c64[ok, s].conj() @ y.T) <= bound).all()
    op = torch.empty(T * (L // 2) * V, dtype=torch.complex64, device="cuda")
    P.bs_apply_lifted(part, xc[:, L // 2:].contiguous().reshape(-1), ch[:, L // 2:].contiguous().reshape(-1), op)
    assert np.array_equal(op.cpu().numpy().reshape(T, -1, V), o[:, L // 2:], equal_nan=True)
