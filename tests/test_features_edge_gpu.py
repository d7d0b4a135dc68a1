"""Window features of covariances that are not finite, or zero: every feature
is infinite, NaN, zero or finite where the FP64 definition (entry times 1/tau,
rounded to FP32) is.  Finite ones to a unit in the last place, 2^-23."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


def test_features_of_non_finite_covariances():
    W, T, L, K = 5, 1, 16, 10
    plan = P.Plan(N=64, F=16 * L, L=L, M=128, u=[0.3], W=[W], K=[K], P_train=8, P_test=0, fc=10e9, fs=1e9, fd=10e9, delta=1.0)
    rng = np.random.default_rng(1)
    z = rng.standard_normal((L, K, W)) + 1j * rng.standard_normal((L, K, W))
    R = np.einsum("gki,gkj->gij", z, z.conj()) / K
    re, im = R.real.copy(), R.imag.copy()
    re[0, 3, 1] = np.inf                        # below the diagonal, finite trace
    im[1, 4, 0] = -np.inf
    re[2, 2, 1], im[2, 2, 1] = np.nan, np.inf
    re[3, 2, 2] = np.inf                        # infinite trace
    re[4, 1, 1] = np.nan
    re[5], im[5] = 0.0, 0.0                     # zero trace
    re[6][np.arange(W), np.arange(W)] = 0.0     # zero trace, entries beside it
    re[7, 3, 0] = 1e80                          # beyond FP32 after the scaling
    re[8, 3, 0] = -1e300
    re[9, 3, 0], re[9, 3, 1] = 1e-300, 5e-41
    R = re + 0j
    R.imag = im
    n = W * W + 2 * W + 2
    X = torch.full((L * n + 3,), 5.0, device="cuda")
    Rd = torch.from_numpy(R.reshape(-1)).cuda()
    assert P.lib().bs_features(plan.handle, Rd.data_ptr(), X.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    x = X.cpu().numpy()
    assert (x[L * n:] == 5.0).all()
    off = plan.offsets()
    i, j = np.tril_indices(W, -1)
    for g in range(L):
        with np.errstate(all="ignore"):
            tau = np.trace(re[g]) / W
            itau = 1.0 / tau
            a = off["a_tilde"][off["woff"][g]:off["woff"][g + 1]]
            a = a / np.linalg.norm(a)
            ref = np.concatenate([np.diag(re[g]) * itau, re[g][i, j] * itau, im[g][i, j] * itau, a.real, a.imag,
                                  [np.log10(tau), np.log10(K / W)]])
            ref32 = ref.astype(np.float32)
        got = x[g * n:(g + 1) * n]
        assert np.array_equal(np.isnan(got), np.isnan(ref32)), g
        assert np.array_equal(got[np.isinf(ref32)], ref32[np.isinf(ref32)]) and np.array_equal(np.isinf(got), np.isinf(ref32)), g
        m = np.isfinite(ref32)
        assert (np.abs(got[m] - ref[m]) <= 2.0 ** -23 * np.abs(ref[m]) + 1e-44).all(), g
