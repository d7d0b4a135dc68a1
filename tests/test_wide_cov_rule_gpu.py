"""Covariances of windows above 16 beams on both sides of the rule between the
3 x 3 and the 4 x 4 tiles: widths and stream lengths around its lines with few
and with many pairs, FP32 and 16-bit windows, a shard of the whole.

Tolerance: FP32 products over at most 16 vectors per partial sum, 16 roundings
of 2^-24 of an entry's magnitude."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,K,L,precision", [
    ([32], 63, 128, 0), ([32], 64, 128, 1), ([31, 2], 64, 128, 0), ([30], 70, 128, 0), ([28, 17], 127, 128, 0), ([26], 128, 128, 2),
    ([24], 255, 128, 1), ([22, 9], 256, 128, 0), ([17], 16, 128, 0), ([21, 16], 33, 128, 1), ([25], 16, 4, 0), ([24], 127, 4, 0),
    ([23], 128, 4, 1), ([18, 3], 5, 4, 0)])
def test_covariance_both_tiles(W, K, L, precision):
    T, B = 6, 16
    kw = dict(N=64, F=16 * L if L * 16 <= 4096 else 4096, L=L, M=64, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[W[t % len(W)] for t in range(T)],
              K=[K] * T, P_train=-(-K // B), P_test=0, fc=10e9, fs=1e9, fd=10e9, delta=1.0,
              precision=(P.BS_PREC_FP32, P.BS_PREC_FP16, P.BS_PREC_BF16)[precision])
    whole, part = P.Plan(**kw), P.Plan(s_begin=L // 2, s_count=L // 4, **kw)
    off = whole.offsets()
    rng = np.random.default_rng(K + W[0])
    z = (rng.standard_normal(whole.sizes.ztrain_elems) + 1j * rng.standard_normal(whole.sizes.ztrain_elems)).astype(np.complex64)

    def device(a):
        t = torch.from_numpy(a).cuda()
        if precision:
            t = torch.view_as_real(t).reshape(-1).to((torch.float16, torch.bfloat16)[precision - 1])
        return t

    zt = device(z)
    zq = torch.view_as_complex(zt.float().reshape(-1, 2)).cpu().numpy() if precision else z
    R = torch.full((whole.sizes.r_elems + 2,), 7.0, dtype=torch.complex128, device="cuda")
    P.bs_window_cov(whole, zt, R)
    r = R.cpu().numpy()
    assert (r[-2:] == 7.0).all()
    for g in range(0, T * L, max(1, T * L // 40)):
        w = int(off["W"][g])
        a = zq[off["ztr_off"][g]:off["ztr_off"][g + 1]].reshape(K, w).astype(np.complex128)
        ref = a.T @ a.conj() / K + np.eye(w)
        mag = np.abs(a).T @ np.abs(a) / K + np.eye(w)
        assert (np.abs(r[off["roff"][g]:off["roff"][g + 1]].reshape(w, w) - ref) <= 16 * 2.0 ** -24 * mag).all(), g
    op = part.offsets()
    pairs = [t * L + s for t in range(T) for s in range(L // 2, L // 2 + L // 4)]
    zp = np.concatenate([z[off["ztr_off"][g]:off["ztr_off"][g + 1]] for g in pairs])
    Rp = torch.empty(part.sizes.r_elems, dtype=torch.complex128, device="cuda")
    P.bs_window_cov(part, device(zp), Rp)
    rp = Rp.cpu().numpy()
    for i, g in enumerate(pairs):
        assert np.array_equal(rp[op["roff"][i]:op["roff"][i + 1]], r[off["roff"][g]:off["roff"][g + 1]]), g
