"""Infinite and NaN values through the products that are summed as BF16 parts:
every output is infinite, NaN or finite exactly where the sum of its products
is, with an infinity's sign, so that one part's zero does not turn another's
infinity into NaN.  Values of few bits (whose trailing parts are zero) and of
all bits.  Tolerance of the finite outputs: that of the kernels, 2e-6 of
||c|| ||y|| and 3e-5 of an array's norm."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P
from paper_2508_11790_gb300 import learned as LR

pytestmark = pytest.mark.gpu

INF, NAN = np.float32(np.inf), np.float32(np.nan)


def _same_class(got, ref):
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(np.isinf(got), np.isinf(ref))
    m = np.isinf(ref)
    assert np.array_equal(np.sign(got[m]), np.sign(ref[m]))


def _mm(a, b):
    """Sum of products, in FP64, without BLAS."""
    with np.errstate(invalid="ignore"):
        return (np.asarray(a, np.float64)[:, :, None] * np.asarray(b, np.float64)[None]).sum(1)


@pytest.mark.parametrize("N,few,T,L,B", [(5, True, 3, 2, 8), (48, False, 3, 2, 8), (150, True, 3, 2, 8), (149, False, 3, 2, 8),
                                        (5, True, 35, 64, 32), (48, True, 35, 64, 32), (47, False, 35, 64, 32)])
def test_outputs_of_infinite_vectors_and_weights(N, few, T, L, B):
    P_te = 3   # the last three cases are more than two waves of the SIMT kernel: tensor-core tiles
    M = 1 << max(4, (N - 1).bit_length())
    plan = P.Plan(N=N, F=L * B, L=L, M=M, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[3] * T, K=[B] * T, P_train=1, P_test=P_te,
                  fc=10e9, fs=1e9, fd=10e9, delta=10.0)
    rng = np.random.default_rng(N)

    def draw(*shape):
        return (rng.integers(-3, 4, shape) if few else rng.standard_normal(shape)).astype(np.float32)

    c, y = draw(T, L, N, 2), draw(1 + P_te, L, B, N, 2)
    c[c == 0], y[y == 0] = 1, 2
    y[1, 0, 2, N // 2, 0] = INF
    y[1, 0, 3, 0, 1] = -INF
    y[2, 1, 4, N - 1] = INF, -INF
    y[2, 1, 5, 1, 0], c[1, 1, 1, 0] = INF, 0      # infinity times zero
    y[3, 0, 0, 2, 1] = NAN
    y[3, 0, 1, 0, 0], y[3, 0, 1, N - 1, 0] = INF, -INF
    c[2, 0, 3, 1] = INF
    out = torch.empty(T * L * P_te * B, dtype=torch.complex64, device="cuda")
    P.bs_apply_lifted(plan, torch.view_as_complex(torch.from_numpy(y).cuda()).reshape(-1),
                      torch.view_as_complex(torch.from_numpy(c).cuda()).reshape(-1), out)
    o = out.cpu().numpy().reshape(T, L, P_te * B)
    for s in range(2):   # where the values above are
        cr, ci = c[:, s, :, 0], c[:, s, :, 1]
        v = y[1:, s].reshape(P_te * B, N, 2)
        re = _mm(np.concatenate([cr, ci], 1), np.concatenate([v[..., 0], v[..., 1]], 1).T)
        im = _mm(np.concatenate([cr, -ci], 1), np.concatenate([v[..., 1], v[..., 0]], 1).T)
        for got, ref in ((o[:, s].real, re), (o[:, s].imag, im)):
            _same_class(got, ref)
            m = np.isfinite(ref)
            assert m.any() and np.abs(got[m] - ref[m]).max() <= 2e-6 * 50 * N   # |entries| <= 5 each


@pytest.mark.parametrize("where", ["weight", "input", "target", "nan"])
@pytest.mark.parametrize("n_in,H,n_out,B", [(20, 8, 3, 5), (70, 96, 4, 40), (130, 256, 10, 70), (20, 300, 3, 33)])
def test_network_of_infinite_values(n_in, H, n_out, B, where):
    rng = np.random.default_rng(H + B)
    p = (rng.integers(1, 4, int(LR._lib().bs_mlp_param_count(n_in, H, n_out))) / 8).astype(np.float32)
    w = LR.unflatten(p, n_in, H, n_out)
    X = rng.integers(-3, 4, (B, n_in)).astype(np.float32)
    T = rng.integers(-3, 4, (B, n_out)).astype(np.float32)
    if where == "weight":
        p[2] = w["W1"][0, 2] = np.inf
        X[:, 2] = np.where(np.arange(B) % 2, 1.5, -1.5)
    elif where == "input":
        X[1, 3], X[B - 1, 0] = INF, -INF
    elif where == "nan":
        X[1, 3] = NAN
    else:
        T[1, 0], T[B - 1, n_out - 1] = INF, -INF
    net = LR.LoadingMLP(n_in, n_out, H, capacity=B, params=p)
    Y = torch.empty(B * n_out, device="cuda")
    Xd, Td = torch.from_numpy(X.ravel()).cuda(), torch.from_numpy(T.ravel()).cuda()
    net.forward(Xd, B, Y)
    net.train_step(Xd, Td, B, lr=0.0)
    with np.errstate(invalid="ignore"):
        z1 = _mm(X, w["W1"].T) + w["b1"]
        h1 = np.fmax(z1, 0)          # a NaN is not positive
        z2 = _mm(h1, w["W2"].T) + w["b2"]
        h2 = np.fmax(z2, 0)
        y = _mm(h2, w["W3"].T) + w["b3"]
        dy = 2 * (y - T) / y.size
        d2 = np.where(z2 > 0, _mm(dy, w["W3"]), 0)
        d1 = np.where(z1 > 0, _mm(d2, w["W2"]), 0)
        g = [_mm(d1.T, X), d1.sum(0), _mm(d2.T, h1), d2.sum(0), _mm(dy.T, h2), dy.sum(0)]
    for got, ref in ((Y.cpu().numpy(), y.ravel()), (net.grad.cpu().numpy(), np.concatenate([t.ravel() for t in g]))):
        _same_class(got, ref)
        m = np.isfinite(ref)
        assert np.linalg.norm(got[m] - ref[m]) <= 3e-5 * np.linalg.norm(ref[m])
