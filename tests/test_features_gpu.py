"""Window features against their FP64 definition rounded to FP32, over window
sizes 1..32, streams of several lengths, and covariances at scales far from 1
(every feature but the logarithms is scale-free).

Tolerance: one FP32 rounding of the FP64 value, so a unit in the last place
(2^-23 relative); log10 adds nothing beyond its own rounding."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,K,scale", [(1, [1, 5], 1.0), (2, [4, 4], 1e-30), (9, [18] * 5, 1e6), (16, [32, 40, 32], 1e30),
                                       (9, [18, 30], 1e-200), (32, [64], 1e200), (7, [14] * 9, 1.0)])
def test_features_are_rounded_fp64(W, K, scale):
    T, L = len(K), 8
    plan = P.Plan(N=64, F=16 * L, L=L, M=128, u=np.sin(np.linspace(-1, 1, T)), W=[W] * T, K=K, P_train=8, P_test=0,
                  fc=10e9, fs=1e9, fd=10e9, delta=1.0)
    G = T * L
    rng = np.random.default_rng(W)
    z = rng.standard_normal((G, 2 * W, W)) + 1j * rng.standard_normal((G, 2 * W, W))
    z *= 10.0 ** rng.uniform(-2, 2, (G, 1, 1))
    R = np.einsum("gki,gkj->gij", z, z.conj()) / (2 * W) * scale
    n = W * W + 2 * W + 2
    X = torch.full((G * n + 3,), 5.0, device="cuda")
    Rd = torch.from_numpy(R.reshape(-1)).cuda()
    assert P.lib().bs_features(plan.handle, Rd.data_ptr(), X.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    x = X.cpu().numpy()
    assert (x[G * n:] == 5.0).all()
    x = x[:G * n].reshape(G, n)
    off = plan.offsets()
    il = np.tril_indices(W, -1)
    for g in range(G):
        tau = np.trace(R[g]).real / W
        a = off["a_tilde"][off["woff"][g]:off["woff"][g + 1]]
        a = a / np.linalg.norm(a)
        ref = np.concatenate([np.diag(R[g]).real / tau, (R[g] / tau)[il].real, (R[g] / tau)[il].imag, a.real, a.imag,
                              [np.log10(tau), np.log10(K[g // L] / W)]])
        assert (np.abs(x[g] - ref) <= 2.0 ** -23 * np.abs(ref) + 1e-44).all(), g
