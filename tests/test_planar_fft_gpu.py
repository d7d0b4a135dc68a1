"""Planar beamspace windows over the shapes that the row-FFT kernel takes and
at its edges: rows of 8 to 1024 beams, columns of 1 to 16, one CTA spanning
several subbands or records, streams that end inside a CTA's vectors, window
entries that wrap on both axes, 16-bit windows, shards, and shapes of the
general kernel, against the 2-D FFT in FP64.

Tolerance: log2(M) butterfly levels of FP32 (2^-24 each, constants included),
below FFT_TOL = 5e-6 of the vector's norm; 16-bit windows are the FP32 ones
rounded (half a unit of their type)."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu

FFT_TOL = 5e-6


@pytest.mark.parametrize("Nx,Nz,Mx,Mz,F,L,win,K,prec,shard", [
    (32, 4, 64, 8, 64, 8, [(8, 4), (4, 2), (1, 1)], [13, 64, 8], P.BS_PREC_FP32, None),
    (32, 4, 64, 8, 64, 16, [(8, 4), (4, 4)], [9, 7], P.BS_PREC_FP16, None),      # B = 4 < 8 vectors per CTA
    (5, 3, 8, 16, 32, 32, [(3, 5), (2, 2)], [2, 1], P.BS_PREC_FP32, None),       # B = 1, 32 vectors per CTA
    (8, 2, 16, 8, 64, 4, [(2, 3)], [30], P.BS_PREC_BF16, None),
    (31, 1, 32, 4, 32, 4, [(7, 1), (2, 4)], [12, 16], P.BS_PREC_FP32, None),
    (100, 5, 128, 16, 16, 2, [(5, 3)], [11], P.BS_PREC_FP32, None),
    (200, 2, 256, 2, 16, 4, [(3, 2), (16, 1)], [5, 8], P.BS_PREC_FP32, None),
    (500, 2, 512, 4, 16, 4, [(4, 4)], [6], P.BS_PREC_FP32, None),
    (512, 2, 1024, 2, 16, 2, [(9, 2)], [10], P.BS_PREC_FP32, None),
    (32, 4, 64, 8, 64, 8, [(8, 4)], [20], P.BS_PREC_FP32, (4, 2)),
    (4, 4, 4, 32, 32, 4, [(2, 4)], [10], P.BS_PREC_FP32, None),                  # general kernel: rows of 4
    (1, 4, 1, 16, 32, 4, [(1, 4)], [10], P.BS_PREC_FP32, None)])
def test_planar_windows(Nx, Nz, Mx, Mz, F, L, win, K, prec, shard):
    T, B, N, M = len(win), F // L, Nx * Nz, Mx * Mz
    u = np.linspace(-0.95, 0.9, T) if T > 1 else np.array([0.97])
    v = np.linspace(0.6, -0.7, T) if T > 1 else np.array([-0.9])
    W, Wz = [a * b for a, b in win], [b for _, b in win]
    P_tr, P_te = -(-max(K) // B), 2
    kw = dict(s_begin=shard[0], s_count=shard[1]) if shard else {}
    plan = P.Plan(N=N, F=F, L=L, M=M, u=u, W=W, K=K, P_train=P_tr, P_test=P_te, fc=10e9, fs=1e9, fd=10e9, delta=1.0,
                  precision=prec, Nz=Nz, Mz=Mz, Wz=Wz, v=v, **kw)
    s0, Ls = shard if shard else (0, L)
    g = torch.Generator(device="cuda").manual_seed(Nx)
    xc = torch.view_as_complex(torch.randn((P_tr + P_te) * Ls * B * N, 2, generator=g, device="cuda"))
    b = P.alloc_buffers(plan)
    b.z_train.zero_()
    P.bs_beamspace(plan, xc, b.z_train, b.z_test)
    torch.cuda.synchronize()
    off = plan.offsets()
    x = xc.cpu().numpy().astype(np.complex128).reshape(P_tr + P_te, Ls, B, Nx, Nz)
    yb = np.fft.fft2(x, s=(Mx, Mz)) / np.sqrt(M)
    norm = np.linalg.norm(x, axis=(-2, -1)).max()
    ztr = b.z_train if prec == P.BS_PREC_FP32 else torch.view_as_complex(b.z_train.float().reshape(-1, 2))
    ztr, zte = ztr.cpu().numpy(), b.z_test.cpu().numpy()
    eps = {P.BS_PREC_FP32: 0.0, P.BS_PREC_FP16: 2.0 ** -11, P.BS_PREC_BF16: 2.0 ** -8}[prec]
    for t in range(T):
        for s in range(Ls):
            k = t * Ls + s
            f = 10e9 + (((s0 + s - L // 2 + 1) - 0.5) / L) * 1e9
            ax = []
            for sine, m, w in ((u[t], Mx, win[t][0]), (v[t], Mz, win[t][1])):
                pos = np.pi * sine * (f / 10e9) * m / (2 * np.pi)
                ax.append((int(np.floor(pos - w / 2 + 1)) + np.arange(w)) % m)
            z = yb[:, s][:, :, ax[0]][:, :, :, ax[1]].reshape(P_tr + P_te, B, W[t])
            ref = z[:P_tr].reshape(-1, W[t])[:K[t]]
            got = ztr[off["ztr_off"][k]:off["ztr_off"][k + 1]].reshape(K[t], W[t])
            tol = FFT_TOL * norm + eps * np.maximum(np.abs(ref.real), np.abs(ref.imag)) * np.sqrt(2)
            assert (np.abs(got - ref) <= tol).all(), (t, s)
            got = zte[off["zte_off"][k]:off["zte_off"][k + 1]].reshape(P_te * B, W[t])
            assert (np.abs(got - z[P_tr:].reshape(-1, W[t])) <= FFT_TOL * norm).all(), (t, s)
