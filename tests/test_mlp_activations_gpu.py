"""The network's work buffers after a forward pass and after a training step:
pre-activations and activations of both hidden layers, written for every row
of the batch and nowhere past it, by the slab kernel and by the layer by layer
products alike.

Tolerance: two dependent layers of at most about 60 FP32 accumulations of
2^-23 each, 2 * 60 * 2^-23 of the array's norm."""
import numpy as np
import pytest
import torch

from paper_2508_11790_gb300 import learned as LR

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,H,n_out,B", [(101, 256, 10, 1024), (1, 1, 1, 1), (17, 96, 4, 33), (64, 127, 8, 64), (65, 130, 16, 15),
                                            (30, 255, 3, 2500), (30, 8, 3, 5000), (20, 300, 5, 70)])
def test_work_buffers_hold_the_activations(n_in, H, n_out, B):
    rng = np.random.default_rng(n_in + B)
    p = LR.he_uniform_params(n_in, H, n_out, seed=5)
    p += rng.uniform(-0.05, 0.05, p.size).astype(np.float32)
    X = rng.standard_normal((B, n_in)).astype(np.float32)
    T = rng.standard_normal((B, n_out)).astype(np.float32)
    w = LR.unflatten(p, n_in, H, n_out)
    for k in ("W1", "W2"):
        w[k] = torch.from_numpy(w[k].astype(np.float32)).to(torch.bfloat16).double().numpy()
    z1 = X.astype(np.float64) @ w["W1"].T + w["b1"]
    z2 = np.maximum(z1, 0) @ w["W2"].T + w["b2"]
    ref = {"z1": z1, "h1": np.maximum(z1, 0), "z2": z2, "h2": np.maximum(z2, 0)}
    Xd, Td = torch.from_numpy(X.ravel()).cuda(), torch.from_numpy(T.ravel()).cuda()
    for train in (False, True):
        net = LR.LoadingMLP(n_in, n_out, H, capacity=B + 3, params=p)
        for k in ref:
            net.work[k].fill_(7.0)
        if train:
            net.train_step(Xd, Td, B, lr=0.0)
        else:
            net.forward(Xd, B, torch.empty(B * n_out, device="cuda"))
        for k, r in ref.items():
            got = net.work[k].cpu().numpy().reshape(B + 3, H)
            assert (got[B:] == 7.0).all(), (k, train)
            assert np.linalg.norm(got[:B] - r) <= 1.5e-5 * np.linalg.norm(r), (k, train)
