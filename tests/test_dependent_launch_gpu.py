"""bs_run, whose stages launch dependently, against its stages called one by
one, bit for bit: twice in a row on different inputs without a
synchronisation between, eager and as a captured graph, over every kernel that
a pass can take (one-shot, warp and tensor-core beamspace, the three
covariances, one and several window sizes, wide windows, planar, fused, plain,
whole blocks of outputs and other counts)."""
import numpy as np
import pytest
import torch

import paper_2508_11790_gb300 as P

pytestmark = pytest.mark.gpu

CASES = [   # N, M, L, B, T, W, K, P_train, P_test, plan arguments
    (60, 64, 4, 8, 3, [5], 40, 8, 4, {}),                                          # one-shot, CTA covariance
    (256, 512, 32, 8, 16, [9], 64, 8, 4, {}),                                      # warp covariance, blocks of outputs
    (256, 512, 16, 8, 5, [9], 64, 8, 4, dict(precision=P.BS_PREC_FP16)),           # tensor-core covariance
    (255, 512, 16, 8, 5, [3, 7, 16], 50, 8, 3, dict(precision=P.BS_PREC_BF16)),    # several window sizes
    (700, 1024, 32, 4, 40, [6], 30, 8, 2, {}),                                     # warp beamspace
    (700, 1024, 32, 4, 40, [3, 11], 30, 8, 2, {}),                                 # chains
    (1024, 2048, 16, 16, 8, [9], 128, 8, 2, dict(precision=P.BS_PREC_FP16)),       # tensor-core beamspace
    (100, 128, 8, 8, 5, [32], 64, 8, 4, {}),                                       # wide windows
    (128, 512, 8, 8, 4, [8], 64, 8, 4, dict(Nz=4, Mz=8, Wz=[2] * 4, v=[0.1, 0.0, -0.1, 0.2])),
    (60, 64, 4, 8, 3, [5], 40, 8, 4, dict(flags=P.BS_FLAG_FUSED)),
    (60, 64, 4, 8, 3, [5], 40, 8, 4, dict(flags=P.BS_FLAG_PLAIN)),
    (60, 64, 4, 8, 3, [5], 40, 8, 0, {}),                                          # no test records
    (60, 64, 8, 8, 3, [5], 40, 8, 4, dict(s_begin=4, s_count=4)),                  # a shard
    (64, 512, 32, 32, 40, [7], 200, 8, 2, {}),                                     # several waves of both dependent stages
    (16, 16, 4, 4, 1, [4], 4, 1, 1, {}),                                           # a few CTAs in all
]


def _stages(plan, b):
    xc = torch.empty(plan.P * plan.F * plan.N, dtype=torch.complex64, device="cuda")   # the wrapper asks for the whole cube of a shard too
    P.bs_channelize(plan, b.x, xc)
    b.xc = xc[:plan.sizes.xc_elems]
    P.bs_beamspace(plan, b.xc, b.z_train, b.z_test)
    if plan.flags & P.BS_FLAG_FUSED:
        P.bs_cov_solve(plan, b.z_train, b.c, b.info, R=b.R)
    else:
        P.bs_window_cov(plan, b.z_train, b.R)
        P.bs_mvdr_solve(plan, b.R, b.c, b.info)
    if plan.P_test:
        P.bs_apply(plan, b.z_test, b.c, b.out)


@pytest.mark.parametrize("case", CASES, ids=[str(i) for i in range(len(CASES))])
def test_pass_equals_its_stages(case):
    N, M, L, B, T, W, K, P_tr, P_te, kw = case
    plan = P.Plan(N=N, F=max(16, L * B), L=L, M=M, u=np.sin(np.linspace(-1.0, 1.0, T)), W=[W[t % len(W)] for t in range(T)],
                  K=[K] * T, P_train=P_tr, P_test=P_te, fc=10e9, fs=1e9, fd=10e9, delta=10.0, **kw)
    g = torch.Generator(device="cuda").manual_seed(N + T)
    xs = [torch.view_as_complex(torch.randn(plan.sizes.x_elems, 2, generator=g, device="cuda")) for _ in range(2)]
    want = []
    for x in xs:
        b = P.alloc_buffers(plan)
        b.x.copy_(x)
        _stages(plan, b)
        torch.cuda.synchronize()
        want.append(b)
    b = P.alloc_buffers(plan)
    st = torch.cuda.Stream()
    b.x.copy_(xs[1])
    torch.cuda.synchronize()
    graph = P.Graph(plan, b, st)
    names = ["out", "z_train", "c", "info"] + (["R"] if not plan.flags & P.BS_FLAG_FUSED else []) + (["z_test"] if P_te else [])
    for run in (lambda: P.bs_run(plan, b, st), lambda: graph.launch(st)):
        for first, second in ((0, 1), (1, 0)):
            with torch.cuda.stream(st):
                b.x.copy_(xs[first])
                run()
                b.x.copy_(xs[second])
                run()
            torch.cuda.synchronize()
            assert plan.device_status() == 0
            for n in names:
                if n == "out" and not P_te:
                    continue
                got, ref = getattr(b, n), getattr(want[second], n)
                assert torch.equal(torch.view_as_real(got) if got.is_complex() else got,
                                   torch.view_as_real(ref) if ref.is_complex() else ref), n
