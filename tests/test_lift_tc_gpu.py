"""The lifted correlator's tensor-core products and its lift at the sizes
where their tiles end: targets around the 64-target tile, columns around the
128-column (192-direction) tile and below 16, element counts around the 16-element stage and
the 64-element chunk, odd counts (unaligned rows), weights at extreme scales,
subband shards, and a failed pair's NaN weights staying its own.

Tolerance: the six products kept of a split pair leave 2^-24 of the product,
a 64-element chunk is four truncated steps of 2^-23 each, and at most 16
chunks are added in FP32 (2^-24 each): below 2e-6 of ||c|| ||y||; the same
bound holds for a pattern relative to its maximum of 1, whose steering values
carry 4 roundings of 2^-24 more."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu

TOL = 2e-6


def _plan(N, T, L, B, P_te, **kw):
    M = 1 << max(4, (N - 1).bit_length())
    u = np.sin(np.linspace(-1.0, 1.0, T))
    W = [min(5, M)] * T
    return P.Plan(N=N, F=L * B, L=L, M=M, u=u, W=W, K=[B] * T, P_train=1, P_test=P_te, fc=10e9, fs=1e9, fd=10e9,
                  delta=10.0, **kw)


@pytest.mark.parametrize("N,T,L,B,P_te,scale", [
    (1024, 64, 16, 16, 8, 1.0), (1, 1, 16, 1, 1, 1.0), (15, 3, 8, 2, 3, 1.0), (16, 65, 4, 4, 4, 1e-30),
    (17, 63, 4, 8, 2, 1e18), (65, 2, 2, 64, 2, 1.0), (100, 130, 2, 32, 5, 1.0), (301, 37, 8, 4, 33, 1.0),
    (64, 20, 16, 8, 16, 1.0), (33, 5, 2, 128, 1, 1.0), (200, 70, 2, 64, 3, 1.0)])
def test_lifted_products_match_fp64(N, T, L, B, P_te, scale):
    plan = _plan(N, T, L, B, P_te)
    g = torch.Generator(device="cuda").manual_seed(N + T)
    ch = (torch.randn(T * L * N, 2, generator=g, device="cuda") * scale).view(-1, 2)
    ch = torch.view_as_complex(ch.contiguous())
    F, Vte = L * B, P_te * B
    xc = torch.view_as_complex(torch.randn((1 + P_te) * F * N, 2, generator=g, device="cuda"))
    out = torch.full((T * L * Vte + 8,), 3.0, dtype=torch.complex64, device="cuda")
    P.bs_apply_lifted(plan, xc, ch, out)
    u = torch.linspace(-1.0, 1.0, 2 * B + 7, dtype=torch.float64, device="cuda")
    pat = torch.full((T * L * len(u) + 8,), 3.0, device="cuda")
    P.bs_beam_pattern(plan, ch, u, pat)
    assert plan.device_status() == 0
    assert (out[T * L * Vte:] == 3.0).all() and (pat[T * L * len(u):] == 3.0).all()
    c64 = ch.cpu().numpy().astype(np.complex128).reshape(T, L, N)
    y64 = xc.cpu().numpy().astype(np.complex128).reshape(1 + P_te, L, B, N)[1:]
    o = out[:T * L * Vte].cpu().numpy().reshape(T, L, Vte)
    p = pat[:T * L * len(u)].cpu().numpy().reshape(T, L, len(u))
    un = u.cpu().numpy()
    for s in range(L):
        y = y64[:, s].reshape(Vte, N)
        ref = c64[:, s].conj() @ y.T
        bound = TOL * np.linalg.norm(c64[:, s], axis=1)[:, None] * np.linalg.norm(y, axis=1)[None]
        assert (np.abs(o[:, s] - ref) <= bound).all()
        f = 10e9 + (((s - L // 2 + 1) - 0.5) / L) * 1e9
        e = np.exp(1j * np.pi * np.outer(np.arange(N), un * (f / 10e9)))
        pref = np.abs(c64[:, s].conj() @ e) / (np.linalg.norm(c64[:, s], axis=1, keepdims=True) * np.sqrt(N))
        assert np.abs(p[:, s] - pref).max() <= TOL


def test_lifted_products_of_a_shard_and_a_failed_pair():
    T, L, B, P_te, N = 5, 8, 4, 3, 40
    whole, part = _plan(N, T, L, B, P_te), _plan(N, T, L, B, P_te, s_begin=4, s_count=2)
    g = torch.Generator(device="cuda").manual_seed(5)
    ch = torch.view_as_complex(torch.randn(T * L * N, 2, generator=g, device="cuda")).reshape(T, L, N)
    ch[2, 5] = float("nan")
    F, Vte = L * B, P_te * B
    xc = torch.view_as_complex(torch.randn((1 + P_te) * F * N, 2, generator=g, device="cuda")).reshape(1 + P_te, L, B, N)
    u = torch.linspace(-1.0, 1.0, 21, dtype=torch.float64, device="cuda")

    def run(plan, c, x, Ls):
        out = torch.empty(T * Ls * Vte, dtype=torch.complex64, device="cuda")
        pat = torch.empty(T * Ls * 21, device="cuda")
        P.bs_apply_lifted(plan, x.contiguous().reshape(-1), c.contiguous().reshape(-1), out)
        P.bs_beam_pattern(plan, c.contiguous().reshape(-1), u, pat)
        return out.cpu().numpy().reshape(T, Ls, Vte), pat.cpu().numpy().reshape(T, Ls, 21)

    o, p = run(whole, ch, xc, L)
    os_, ps = run(part, ch[:, 4:6], xc[:, 4:6], 2)
    assert np.array_equal(o[:, 4:6], os_, equal_nan=True) and np.array_equal(p[:, 4:6], ps, equal_nan=True)
    bad = np.zeros((T, L), bool)
    bad[2, 5] = True
    assert (np.isnan(o).any(-1) == bad).all() and (np.isnan(p).any(-1) == bad).all() and np.isnan(o[2, 5]).all()


@pytest.mark.parametrize("N,T,W", [(1, 1, 1), (33, 3, 7), (512, 5, 16), (514, 2, 3), (1023, 9, 32), (1024, 6, 9)])
def test_lift_sizes(N, T, W):
    """Tolerance: a W-term Horner sum of FP32 FMAs, W 2^-24 of each term's magnitude, doubled for the two twiddles."""
    M = 1 << max(5, (N - 1).bit_length())
    L = 4
    u = np.sin(np.linspace(-0.9, 0.9, T))
    plan = P.Plan(N=N, F=16, L=L, M=M, u=u, W=[W] * T, K=[4] * T, P_train=1, P_test=0, fc=10e9, fs=1e9, fd=10e9,
                  delta=10.0)
    g = torch.Generator(device="cuda").manual_seed(W)
    c = torch.view_as_complex(torch.randn(T * L * W, 2, generator=g, device="cuda"))
    ch = torch.full((T * L * N + 4,), 3.0, dtype=torch.complex64, device="cuda")
    P.bs_lift(plan, c, ch)
    torch.cuda.synchronize()
    assert (ch[T * L * N:] == 3.0).all()
    start = plan.offsets()["start"]
    c64 = c.cpu().numpy().astype(np.complex128).reshape(T * L, W)
    n = np.arange(N)
    got = ch[:T * L * N].cpu().numpy().reshape(T * L, N)
    for k in range(T * L):
        m = (start[k] + np.arange(W)) % M
        ref = (c64[k][:, None] * np.exp(2j * np.pi * ((m[:, None] * n) % M) / M)).sum(0) / np.sqrt(M)
        assert np.abs(got[k] - ref).max() <= 2 * W * 2.0 ** -24 * np.abs(c64[k]).sum() / np.sqrt(M) + 1e-30
