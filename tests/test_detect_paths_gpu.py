"""Range-Doppler maps and CFAR over their dispatch: 2 to 20 records (register
paths up to 8 and 16, the loop beyond), 16 to 4096 points (one to eight CTAs
per target and a second sweep), against the FP64 definition.

Tolerances: log2(F) + P_test FP32 additions of the row FFT and the Doppler sum,
doubled by the square: below 1e-5 of a target's largest cell.  The CFAR is
decided again in FP32 numpy in the same order from the GPU's own map: floors,
masks, counts and peaks equal."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,L,T,R", [(16, 4, 3, 2), (64, 64, 1, 8), (256, 16, 5, 9), (512, 8, 2, 16), (1024, 16, 3, 17),
                                     (2048, 128, 4, 3), (4096, 32, 2, 20), (4096, 1, 2, 8)])
def test_map_and_cfar(F, L, T, R):
    plan = P.Plan(N=16, F=F, L=L, M=16, u=np.zeros(T), W=[1] * T, K=[1] * T, P_train=1, P_test=R, fc=10e9, fs=1e9,
                  fd=10e9, delta=1.0)
    g = torch.Generator(device="cuda").manual_seed(F + R)
    n = T * R * F
    out = torch.view_as_complex(torch.randn(n, 2, generator=g, device="cuda"))
    pulse = torch.view_as_complex(torch.randn(F, 2, generator=g, device="cuda"))
    out[::37] *= 30
    work = torch.empty(2 * n, dtype=torch.complex64, device="cuda")
    m, floor = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    count, peak = (torch.empty(T, dtype=torch.int32, device="cuda") for _ in range(2))
    mask = torch.empty(n, dtype=torch.uint8, device="cuda")
    P.bs_range_doppler(plan, out, pulse, work, m)
    P.bs_cfar(plan, m, 6.0, floor, count, mask, peak)
    torch.cuda.synchronize()
    B = F // L
    y = np.empty((T, R, F), complex)
    q = (np.arange(F) - F // 2) % F
    y[:, :, q] = out.cpu().numpy().reshape(T, L, R, B).transpose(0, 2, 1, 3).reshape(T, R, F)
    rp = np.fft.ifft(y * pulse.cpu().numpy().astype(complex).conj(), axis=2, norm="ortho")
    ref = np.abs(np.fft.fft(rp, axis=1)) ** 2
    mg = m.cpu().numpy().reshape(T, R, F)
    assert (np.abs(mg - ref) <= 1e-5 * ref.max(axis=(1, 2), keepdims=True)).all()
    ratio = np.float32(10.0) ** np.float32(0.6)
    fl = np.zeros_like(mg)
    for d in range(R):
        for e in range(R):
            if e != d:
                fl[:, d] += mg[:, e]
    fl *= np.float32(1.0) / np.float32(R - 1)
    assert np.array_equal(floor.cpu().numpy().reshape(T, R, F), fl)
    mk = mask.cpu().numpy().reshape(T, R, F)
    sure = np.abs(mg - fl * ratio) > 1e-6 * mg   # the host's power may be a unit off
    assert np.array_equal(mk[sure].astype(bool), (mg > fl * ratio)[sure])
    assert np.array_equal(count.cpu().numpy(), mk.reshape(T, -1).sum(1))
    hit = np.where(mk.astype(bool), mg, -1.0).reshape(T, -1)
    want = [int(h.argmax()) if h.max() >= 0 else -1 for h in hit]   # the first of the largest
    assert peak.cpu().tolist() == want
