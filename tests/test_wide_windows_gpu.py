"""Covariance and solve of windows around and above 16 beams on given windows:
every window size 17..32 and mixed plans (the size classes of the wide solve,
the 4 x 4 tiles of the wide covariance), stream lengths around the staged
chunk, FP32 and 16-bit windows, with and without a preconditioner, and every
pair escalated to FP64 (info checked against the pivot ratio in FP64).

Tolerances: the covariance sums FP32 products over at most 16 vectors (16
roundings of 2^-24 of an entry's magnitude, COV_TOL); weights from the GPU's
own covariance as in the parity tests (SOLVE_TOL: FP32 factor, compensated
residual, one refinement)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu

COV_TOL = 16 * 2.0 ** -24
SOLVE_TOL = 2e-5


def _plan(W, K, precision=P.BS_PREC_FP32, **kw):
    T, L, B = len(W), 4, 16
    u = np.sin(np.linspace(-1.0, 1.0, T))
    P_tr = -(-max(K) // B)
    return P.Plan(N=64, F=L * B, L=L, M=64, u=u, W=W, K=K, P_train=P_tr, P_test=0, fc=10e9, fs=1e9, fd=10e9,
                  delta=1.0, precision=precision, **kw)


def _windows(plan, off, seed):
    g = np.random.default_rng(seed)
    z = []
    for p in range(plan.sizes.pairs):
        W, K = int(off["W"][p]), int(off["K"][p])
        b = np.exp(1j * np.pi * np.arange(W) * g.uniform(-1, 1))
        x = (g.standard_normal((K, W)) + 1j * g.standard_normal((K, W))) * np.sqrt(0.5)
        z.append((x + 20 * (g.standard_normal((K, 1)) + 1j * g.standard_normal((K, 1))) * b).ravel())
    return np.concatenate(z).astype(np.complex64)


@pytest.mark.parametrize("W,K,precision,pre,kappa", [
    (list(range(17, 33)), [40] * 16, P.BS_PREC_FP32, False, 0.0),
    (list(range(17, 33)), [70] * 16, P.BS_PREC_FP32, True, 0.0),
    ([32, 1, 5, 16, 17, 20, 21, 29], [33, 4, 31, 32, 64, 65, 1, 300], P.BS_PREC_FP32, False, 0.0),
    ([32, 30, 3, 25], [129, 31, 16, 32], P.BS_PREC_FP16, False, 0.0),
    ([32, 31, 18, 24], [64, 100, 90, 60], P.BS_PREC_BF16, True, 0.0),
    ([32, 27, 23, 19, 9], [64, 60, 70, 50, 40], P.BS_PREC_FP32, False, 1.0001),
    ([32], [128], P.BS_PREC_FP32, False, 0.0)])
def test_wide_covariance_and_solve(W, K, precision, pre, kappa):
    plan = _plan(W, K, precision, kappa_max=kappa)
    off = plan.offsets()
    z = _windows(plan, off, len(W))
    zt = torch.from_numpy(z).cuda()
    if precision != P.BS_PREC_FP32:
        zt = torch.view_as_real(zt).reshape(-1).to(torch.float16 if precision == P.BS_PREC_FP16 else torch.bfloat16)
        z = torch.view_as_complex(zt.float().reshape(-1, 2)).cpu().numpy()
    s = plan.sizes
    R = torch.empty(s.r_elems, dtype=torch.complex128, device="cuda")
    c = torch.empty(s.c_elems, dtype=torch.complex64, device="cuda")
    info = torch.empty(s.pairs, dtype=torch.int32, device="cuda")
    P.bs_window_cov(plan, zt, R)
    d = np.ones(s.c_elems, np.float32)
    if pre:
        d = (2.0 ** np.random.default_rng(1).uniform(-3, 3, s.c_elems)).astype(np.float32)
        P.bs_mvdr_solve_precond(plan, R, torch.from_numpy(d).cuda(), c, info)
    else:
        P.bs_mvdr_solve(plan, R, c, info)
    torch.cuda.synchronize()
    Rn, cn, inf = R.cpu().numpy(), c.cpu().numpy(), info.cpu().numpy()
    for g in range(s.pairs):
        w, k = int(off["W"][g]), int(off["K"][g])
        zg = z[off["ztr_off"][g]:off["ztr_off"][g + 1]].reshape(k, w).astype(np.complex128)
        Rg = Rn[off["roff"][g]:off["roff"][g + 1]].reshape(w, w)
        ref = zg.T @ zg.conj() / k + np.eye(w)
        mag = np.abs(zg).T @ np.abs(zg) / k
        assert (np.abs(Rg - ref) <= COV_TOL * mag).all(), (g, w, k)
        assert np.array_equal(Rg, Rg.conj().T)
        # FP64 where the pivot ratio of the scaled matrix (powers of two) passes kappa_max
        e = 2.0 ** np.rint(np.log2(d[off["woff"][g]:off["woff"][g + 1]].astype(np.float64)))
        piv = np.diag(np.linalg.cholesky(Rg * np.outer(e, e))).real
        ratio = (piv.max() / piv.min()) ** 2 / (kappa or 1e5)
        if abs(ratio - 1) > 0.01:
            assert inf[g] == (-2 if ratio > 1 else 0), (g, w, inf[g], ratio)
        a = off["a_tilde"][off["woff"][g]:off["woff"][g + 1]]
        co = O.mvdr_weights(Rg, a)
        cg = cn[off["woff"][g]:off["woff"][g + 1]]
        assert np.linalg.norm(cg - co) <= SOLVE_TOL * np.linalg.norm(co), (g, w, k)
