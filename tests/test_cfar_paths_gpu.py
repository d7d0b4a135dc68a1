"""The CFAR's variants against the host's FP32 sums in the same order, bit for
bit: records around the register variants' 4, 8, 16 and 32, one CTA and
several per target, range cells below and above a CTA's 256, ties of the
largest cell, a target without a detection, infinite and NaN cells."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F,T,R", [(16, 3, 2), (256, 2, 4), (512, 5, 5), (2048, 2, 8), (1024, 3, 9), (64, 2, 16), (512, 2, 17), (4096, 1, 31),
                                   (256, 3, 32), (2048, 2, 33), (16, 2, 65), (1024, 1300, 3), (512, 700, 4)])
def test_cfar_is_exact(F, T, R):
    plan = P.Plan(N=16, F=F, L=4, M=16, u=np.zeros(T), W=[1] * T, K=[1] * T, P_train=1, P_test=R, fc=10e9, fs=1e9, fd=10e9, delta=1.0)
    rng = np.random.default_rng(F + R)
    m = rng.exponential(size=(T, R, F)).astype(np.float32)
    m[T // 2] = 1.0                                   # no cell above its floor
    m[0, 1, F // 2] = m[0, 0, F - 1] = 3e4            # a tie: the smaller index
    m[0, R - 1, 1], m[0, 0, 2] = np.inf, np.nan
    n = m.size
    floor = torch.full((n + 4,), 7.0, device="cuda")
    count, peak = (torch.full((T + 1,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    mask = torch.full((n + 4,), 9, dtype=torch.uint8, device="cuda")
    P.bs_cfar(plan, torch.from_numpy(m.ravel()).cuda(), 6.0, floor, count, mask, peak)
    torch.cuda.synchronize()
    assert (floor[n:] == 7.0).all() and (mask[n:] == 9).all() and count[T] == -7 and peak[T] == -7
    fl = np.zeros_like(m)
    with np.errstate(invalid="ignore"):
        for d in range(R):
            for e in range(R):
                if e != d:
                    fl[:, d] += m[:, e]
        fl *= np.float32(1.0) / np.float32(R - 1)
        ratio = np.float32(10.0) ** np.float32(0.6)
        got = mask[:n].cpu().numpy().reshape(T, R, F)
        assert np.array_equal(floor[:n].cpu().numpy().reshape(T, R, F), fl, equal_nan=True)
        sure = ~(np.abs(m - fl * ratio) <= 1e-6 * m)   # the host's 10^0.6 may be a unit off
        assert np.array_equal(got[sure].astype(bool), (m > fl * ratio)[sure])
    assert np.array_equal(count[:T].cpu().numpy(), got.reshape(T, -1).sum(1))
    hit = np.where(got.astype(bool), m, -1.0).reshape(T, -1)
    assert peak[:T].cpu().tolist() == [int(h.argmax()) if h.max() >= 0 else -1 for h in hit]
