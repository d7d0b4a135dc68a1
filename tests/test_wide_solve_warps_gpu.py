"""The wide solve's warps per CTA follow the number of pairs: the same pairs
solved in a plan of many and in a shard of few give the same weights and info
bit for bit, with a last CTA that is not full, one size class and several, with
and without a preconditioner, and match FP64.

Tolerance against FP64: the parity tests' 2e-5 of a pair's weights."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,L,W,pre", [(1, 2, [32], False), (3, 64, [32], True), (5, 128, [17, 24, 31], False), (7, 64, [28], True),
                                       (11, 256, [20, 32], False), (25, 128, [29], True)])
def test_few_and_many_pairs_agree(T, L, W, pre):
    Ws = [W[t % len(W)] for t in range(T)]
    kw = dict(N=64, F=max(16, 4 * L), L=L, M=64, u=np.sin(np.linspace(-1.0, 1.0, T)), W=Ws, K=[4] * T, P_train=1, P_test=0, fc=10e9, fs=1e9,
              fd=10e9, delta=1.0)
    whole, part = P.Plan(**kw), P.Plan(s_begin=0, s_count=1, **kw)
    off = whole.offsets()
    rng = np.random.default_rng(T + L)
    R, d = [], []
    for t in range(T):
        w = Ws[t]
        x = rng.standard_normal((L, w, 2 * w)) + 1j * rng.standard_normal((L, w, 2 * w))
        R.append(x @ x.conj().transpose(0, 2, 1) / (2 * w) + np.eye(w))
        d.append(2.0 ** rng.uniform(-3, 3, (L, w)))
    flat = lambda v, sel: torch.from_numpy(np.concatenate([a[sel].ravel() for a in v])).cuda()

    def solve(plan, sel):
        s = plan.sizes
        c = torch.full((s.c_elems + 2,), 7.0, dtype=torch.complex64, device="cuda")
        info = torch.full((s.pairs + 1,), 9, dtype=torch.int32, device="cuda")
        if pre:
            P.bs_mvdr_solve_precond(plan, flat(R, sel), flat(d, sel).float(), c, info)
        else:
            P.bs_mvdr_solve(plan, flat(R, sel), c, info)
        torch.cuda.synchronize()
        assert (c[-2:] == 7.0).all() and info[-1] == 9
        return c[:-2].cpu().numpy(), info[:-1].cpu().numpy()

    cw, iw = solve(whole, slice(None))
    cp, ip = solve(part, slice(0, 1))
    at = off["a_tilde"]
    o = 0
    for t in range(T):
        a0 = off["woff"][t * L]
        assert np.array_equal(cw[a0:a0 + Ws[t]], cp[o:o + Ws[t]]) and iw[t * L] == ip[t]
        o += Ws[t]
        for s in {0, L // 2, L - 1}:
            k = t * L + s
            v = np.linalg.solve(R[t][s], at[off["woff"][k]:off["woff"][k + 1]])
            ref = v / np.vdot(at[off["woff"][k]:off["woff"][k + 1]], v)
            got = cw[off["woff"][k]:off["woff"][k + 1]]
            assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref), (t, s)
