"""Beamformer outputs called by themselves: whole blocks of 32 test vectors
(one and several blocks per warp, with and without a remainder), other vector
counts, windows of 1 to 32 beams, few pairs, enough to give a warp several
blocks, and the number between that takes an output per thread, and test windows that start on 8 bytes only.

Tolerance: a sum of W complex FP32 products, 2 W + 2 roundings of 2^-24 of the
sum of the products' magnitudes."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("T,L,B,P_te", [
    (3, 2, 8, 4), (3, 2, 8, 12), (2, 4, 16, 8), (5, 2, 32, 5), (4, 2, 32, 7), (3, 2, 16, 3), (2, 2, 1, 1),
    (40, 64, 16, 8), (80, 64, 8, 4), (160, 64, 16, 4), (80, 64, 8, 12), (80, 64, 16, 8), (80, 64, 32, 5), (80, 64, 32, 7), (80, 64, 8, 5)])
@pytest.mark.parametrize("widths", [(1, 9, 16), (3,), (17, 2, 32)])
def test_outputs_match_fp64(T, L, B, P_te, widths, shift):
    W = [widths[t % len(widths)] for t in range(T)]
    plan = P.Plan(N=32, F=max(16, L * B), L=L, M=32, u=np.sin(np.linspace(-1.0, 1.0, T)), W=W, K=[B] * T, P_train=1, P_test=P_te,
                  fc=10e9, fs=1e9, fd=10e9, delta=10.0)
    s = plan.sizes
    g = torch.Generator(device="cuda").manual_seed(T + P_te)
    z = torch.view_as_complex(torch.randn(s.ztest_elems + 2, 2, generator=g, device="cuda"))[shift:]
    c = torch.view_as_complex(torch.randn(s.c_elems, 2, generator=g, device="cuda"))
    out = torch.full((s.out_elems + 8,), 3.0, dtype=torch.complex64, device="cuda")
    P.bs_apply(plan, z, c, out)
    torch.cuda.synchronize()
    assert (out[s.out_elems:] == 3.0).all()
    off = plan.offsets()
    o = out[:s.out_elems].cpu().numpy().reshape(s.pairs, s.Vte)
    zh, chh = z.cpu().numpy().astype(np.complex128), c.cpu().numpy().astype(np.complex128)
    for k in range(s.pairs):
        w = int(off["W"][k])
        zk = zh[off["zte_off"][k]:off["zte_off"][k] + s.Vte * w].reshape(s.Vte, w)
        ck = chh[off["woff"][k]:off["woff"][k] + w].conj()
        bound = (2 * w + 2) * 2.0 ** -24 * (np.abs(zk) * np.abs(ck)).sum(1)
        assert (np.abs(o[k] - zk @ ck) <= bound).all(), k
