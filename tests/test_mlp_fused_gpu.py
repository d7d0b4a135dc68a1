"""The tensor-core network passes (batch slabs, weight gradients) at the
sizes where tiles and chunks end: input counts around the 64-feature chunk,
odd and unaligned hidden sizes, 1 to 64 outputs, batches around the 32-row
slab and the cluster split, and sizes past the fused kernels' range, against
FP64 products of the same BF16 weights.

Tolerance: every product is exact to 2^-24 and a sum takes at most about 60
FP32 accumulations of 2^-23 each per layer; four dependent products give
4 * 60 * 2^-23 = 2.9e-5 of the array's norm."""
import numpy as np
import pytest
import torch

from paper_2508_11790_gb300 import learned as LR

pytestmark = pytest.mark.gpu

TOL = 3e-5


def _reference(p, n_in, H, n_out, X, T):
    w = LR.unflatten(p, n_in, H, n_out)
    for k in ("W1", "W2", "W3"):
        w[k] = torch.from_numpy(w[k].astype(np.float32)).to(torch.bfloat16).double().numpy()
    z1 = X @ w["W1"].T + w["b1"]
    h1 = np.maximum(z1, 0)
    z2 = h1 @ w["W2"].T + w["b2"]
    h2 = np.maximum(z2, 0)
    y = h2 @ w["W3"].T + w["b3"]
    dy = 2 * (y - T) / y.size
    d2 = (dy @ w["W3"]) * (z2 > 0)
    d1 = (d2 @ w["W2"]) * (z1 > 0)
    g = np.concatenate([t.ravel() for t in (d1.T @ X, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0))])
    return y, g, float(((y - T) ** 2).mean())


@pytest.mark.parametrize("n_in,H,n_out,B", [
    (101, 256, 10, 1024), (1, 8, 1, 1), (17, 96, 4, 33), (64, 128, 8, 64), (65, 129, 16, 65), (128, 100, 17, 31),
    (290, 255, 33, 200), (257, 256, 64, 513), (30, 7, 3, 4097), (20, 300, 5, 70), (20, 64, 70, 70)])
def test_network_passes_match_fp64(n_in, H, n_out, B):
    rng = np.random.default_rng(n_in * 1000 + B)
    p = LR.he_uniform_params(n_in, H, n_out, seed=3)
    p += rng.uniform(-0.05, 0.05, p.size).astype(np.float32)
    X = rng.standard_normal((B, n_in)).astype(np.float32)
    T = rng.standard_normal((B, n_out)).astype(np.float32)
    net = LR.LoadingMLP(n_in, n_out, H, capacity=B, params=p)
    Xd, Td = torch.from_numpy(X.ravel()).cuda(), torch.from_numpy(T.ravel()).cuda()
    Y = torch.full((B * n_out + 64,), 7.0, device="cuda")
    net.forward(Xd, B, Y)
    net.train_step(Xd, Td, B, lr=0.0)
    torch.cuda.synchronize()
    y, g, loss = _reference(p, n_in, H, n_out, X.astype(np.float64), T.astype(np.float64))
    yg = Y.cpu().numpy()
    assert (yg[B * n_out:] == 7.0).all()                      # nothing past the batch
    yg = yg[:B * n_out].reshape(B, n_out)
    assert np.linalg.norm(yg - y) <= TOL * np.linalg.norm(y)
    assert np.linalg.norm(net.grad.cpu().numpy() - g) <= TOL * np.linalg.norm(g)
    assert net.loss.item() == pytest.approx(loss, rel=1e-5)
    assert (net.master.cpu().numpy() == p).all() and net.step == 0
    # an Adam step from the gradients on the device, FP32 arithmetic of its formula
    net.train_step(Xd, Td, B, lr=1e-3)
    torch.cuda.synchronize()
    gd = net.grad.cpu().numpy().astype(np.float64)
    m, v = 0.1 * gd, 0.001 * gd * gd
    want = p - 1e-3 * (m / 0.1) / (np.sqrt(v / 0.001) + 1e-8)
    np.testing.assert_allclose(net.master.cpu().numpy(), want, rtol=1e-5, atol=2e-6)
    assert torch.equal(net.bf16, net.master.to(torch.bfloat16)) and net.step == 1
