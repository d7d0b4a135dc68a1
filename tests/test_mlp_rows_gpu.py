"""Forward passes of narrow networks over many rows, where the layer by layer
products take over from the slabs, on both sides of the line, against FP64
products of the same BF16 weights.

Tolerance: every product is exact to 2^-24 and a sum takes at most about 60
FP32 accumulations of 2^-23 each per layer; three dependent layers give
3 * 60 * 2^-23 = 2.2e-5 of the array's norm."""
import numpy as np
import pytest
import torch

from paper_2508_11790_gb300 import learned as LR

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [1, 8, 48, 63, 64])
@pytest.mark.parametrize("n_in,n_out,B", [(20, 3, 4864), (20, 3, 4865), (20, 3, 9729), (101, 10, 29185), (7, 1, 140001)])
def test_forward_of_many_rows(n_in, H, n_out, B):
    p = LR.he_uniform_params(n_in, H, n_out, seed=2) + np.float32(0.03)
    w = LR.unflatten(p, n_in, H, n_out)
    for k in ("W1", "W2", "W3"):
        w[k] = torch.from_numpy(w[k].astype(np.float32)).to(torch.bfloat16).double().numpy()
    X = np.random.default_rng(H).standard_normal((B, n_in)).astype(np.float32)
    h1 = np.maximum(X.astype(np.float64) @ w["W1"].T + w["b1"], 0)
    h2 = np.maximum(h1 @ w["W2"].T + w["b2"], 0)
    y = h2 @ w["W3"].T + w["b3"]
    net = LR.LoadingMLP(n_in, n_out, H, capacity=B, params=p)
    Y = torch.full((B * n_out + 64,), 7.0, device="cuda")
    net.forward(torch.from_numpy(X.ravel()).cuda(), B, Y)
    got = Y.cpu().numpy()
    assert (got[B * n_out:] == 7.0).all()
    assert np.linalg.norm(got[:B * n_out].reshape(B, n_out) - y) <= 2.2e-5 * np.linalg.norm(y)
    h = net.work["h2"].cpu().numpy().reshape(B, H)
    assert np.linalg.norm(h - h2) <= 2.2e-5 * np.linalg.norm(h2)
