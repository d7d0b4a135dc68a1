"""What the framework's users have it do, as measurable cases.

Every case is one call (or the short chain of calls that belongs together)
through the public entry points of ``paper_2508_11790_gb300``, on a plan and
buffers that a program keeps:

* ``pass``    bs_run (or its CUDA graph): raw IQ cube -> weights and
  beamformed test vectors;
* ``windows`` bs_channelize and bs_beamspace: raw IQ cube -> training and
  test windows, linear or planar array;
* ``weights`` bs_window_cov and bs_mvdr_solve: training windows -> weights;
* ``loading`` learned loading of short streams (K = 2W): unloaded
  covariance, features, network, per-pair loading and preconditioner seed,
  loaded covariance, preconditioned solve;
* ``train``   one Adam step of the loading network;
* ``lifted``  antenna-space weights of every pair and their output;
* ``pattern`` beam patterns of the antenna-space weights;
* ``detect``  range-Doppler maps and CFAR of the beamformed outputs.

The passes return the weights and the outputs.  The windows and covariances
are work buffers of a pass, and ``info`` says which of the two solves a pair
took, a threshold on a rounded condition estimate; a pair that fails has NaN
weights.  The 16-bit windows are FP16: BF16 ones run the same kernels but
miss the weight tolerance, so programs store FP16.
"""
import math

import numpy as np
import torch

import paper_2508_11790_gb300 as P
from paper_2508_11790_gb300 import learned

FC, FS, FD = 10e9, 1e9, 10e9      # carrier, sampling rate, design frequency of the half-wavelength spacing
DELTA = 10.0                      # diagonal loading, noise-variance units
UNEVEN = (3, 5, 7, 9, 11, 15)     # window sizes of the uneven workload


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest workload: a few targets of a small array, latency and launches count
        dict(name="pass_small", kind="pass", call="run", prec="fp32", N=64, F=512, L=16, M=64, T=4, W=5, K=128,
             P_test=8, jam=2),
        # an ordinary grid of targets and subbands in FP32
        dict(name="pass_grid", kind="pass", call="run", prec="fp32", N=256, F=1024, L=64, M=512, T=16, W=7, K=256,
             P_test=8, jam=4),
        # the headline workload: a large array, FP16 windows, captured once and replayed per batch
        dict(name="pass_large_fp16", kind="pass", call="graph", prec="fp16", N=1024, F=2048, L=128, M=2048, T=64, W=9,
             K=512, P_test=8, jam=8),
        # 256 targets with windows and stream lengths of their own (W of UNEVEN, K in 2W..8W), captured
        dict(name="pass_uneven", kind="pass", call="graph", prec="fp32", N=1024, F=2048, L=128, M=2048, T=256, W=0,
             K=0, P_test=8, jam=8),
        # an odd number of elements, a prime number of targets, windows and streams of every length
        dict(name="windows_ragged", kind="windows", prec="fp32", N=301, F=1024, L=32, M=1024, T=37, W=0, K=0,
             P_test=5, jam=5),
        # the paper's 4 x 32 planar array, 8 x 64 beams, its 20 targets and its largest (4 x 8) window
        dict(name="windows_planar", kind="windows", prec="fp32", N=128, Nz=4, F=1024, L=128, M=512, Mz=8, T=20,
             W=32, Wz=4, K=128, P_test=8, jam=6),
        # the weights of those 4 x 8 windows: the widest covariances and solves
        dict(name="weights_wide", kind="weights", prec="fp32", T=20, L=128, W=32, K=128),
        # learned loading of 16384 pairs with K = 2W snapshots
        dict(name="loading_2w", kind="loading", T=128, L=128, W=9, hidden=256),
        # one training step of the loading network at its default minibatch
        dict(name="train_step", kind="train", W=9, hidden=256, batch=1024),
        # antenna-space weights of the headline workload's pairs, applied to its test vectors
        dict(name="lifted_large", kind="lifted", N=1024, F=2048, L=128, M=2048, T=64, W=9, P_test=8),
        # their beam patterns, one degree apart
        dict(name="pattern_large", kind="pattern", N=1024, F=2048, L=128, M=2048, T=64, W=9, dirs=181),
        # range-Doppler maps and detections of its targets
        dict(name="detect_large", kind="detect", F=2048, L=128, T=64, P_test=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def _pow2_at_least(n):
    return 1 << max(0, (n - 1).bit_length())


def draw(rng):
    kind = rng.choice(["pass", "pass", "pass", "linear", "planar", "weights", "loading", "train", "lifted", "pattern",
                       "detect"])
    if kind == "planar":
        Nz, Mz = rng.choice([(2, 4), (4, 4), (4, 8), (8, 8)])
        Wz, Wx = rng.choice([(2, 4), (4, 4), (4, 8), (3, 3), (2, 7), (1, 5)])
        Wz = min(Wz, Mz)
        Nx = _log(rng, 8, 64)
        Mx = min(128, _pow2_at_least(Nx) * rng.choice([1, 2]))
        F = _pow2(rng, 256, 1024)
        L = min(F, _pow2(rng, 16, 128))
        W = Wz * Wx
        return dict(kind="windows", prec=rng.choice(["fp32", "fp32", "fp16"]), N=Nx * Nz, Nz=Nz, F=F, L=L, M=Mx * Mz,
                    Mz=Mz, T=_log(rng, 2, 40), W=W, Wz=Wz, K=rng.randint(4 * W, 8 * W), P_test=rng.randint(2, 8),
                    jam=rng.randint(1, 6))
    if kind == "weights":
        W = rng.randint(2, 32)
        K = rng.randint(2 * W, 16 * W)
        L = _pow2(rng, 16, 128)
        return dict(kind="weights", prec=rng.choice(["fp32", "fp32", "fp16"]), T=min(_log(rng, 2, 128), (1 << 25) // (L * K * W)),
                    L=L, W=W, K=K)
    if kind in ("pass", "linear"):
        prec = rng.choice(["fp32", "fp32", "fp16"])
        N = _log(rng, 24, 1024)
        if rng.random() < 0.5:
            N = _pow2_at_least(N)
        M = _pow2_at_least(N) * rng.choice([1, 2])
        F = _pow2(rng, 128, 2048)
        L = min(F // 4, _pow2(rng, 8, 128))
        T = _log(rng, 2, 160)
        uneven = prec == "fp32" and rng.random() < 0.4
        W = 0 if uneven else rng.randint(3, 16)
        K = 0 if uneven else rng.randint(8 * W, max(8 * W, 512)) if prec == "fp16" else rng.randint(4 * W, 32 * W)
        c = dict(kind=kind, prec=prec, N=N, F=F, L=L, M=M, T=T, W=W, K=K, P_test=rng.randint(2, 8),
                 jam=rng.randint(1, 8))
        if kind == "linear":
            c["kind"] = "windows"
        else:
            c["call"] = rng.choice(["run", "run", "graph"])
        while True:   # no larger than the headline workload's cube and windows
            g = _geometry(c)
            cube, windows = g["P"] * c["F"] * c["N"], c["L"] * sum(w * k for w, k in zip(g["W"], g["K"]))
            if windows > 1 << 25:
                c["T"] //= 2
            elif cube > 1 << 26:
                c["F"], c["L"] = c["F"] // 2, max(1, c["L"] // 2)
            else:
                return c
    if kind == "loading":
        return dict(kind="loading", T=_log(rng, 4, 128), L=_pow2(rng, 16, 128), W=rng.randint(3, 11),
                    hidden=rng.choice([128, 256, 256]))
    if kind == "train":
        return dict(kind="train", W=rng.randint(3, 15), hidden=rng.choice([96, 128, 256, 256]), batch=_log(rng, 128, 4096))
    if kind in ("lifted", "pattern"):
        N = _log(rng, 48, 1024)
        if rng.random() < 0.5:
            N = _pow2_at_least(N)
        F = _pow2(rng, 256, 2048)
        c = dict(kind=kind, N=N, F=F, L=min(F // 4, _pow2(rng, 16, 128)), M=_pow2_at_least(N) * rng.choice([1, 2]),
                 T=_log(rng, 3, 64), W=rng.randint(3, 16))
        if kind == "lifted":
            c["P_test"] = rng.randint(2, 8)
        else:
            c["dirs"] = _log(rng, 31, 181)
        return c
    F = _pow2(rng, 256, 2048)
    return dict(kind="detect", F=F, L=min(F // 2, _pow2(rng, 16, 128)), T=_log(rng, 2, 64), P_test=rng.randint(3, 16))


# ---------------------------------------------------------------- geometry
def _geometry(case):
    """Per-target windows and stream lengths and the records they need."""
    T, B = case["T"], case["F"] // case["L"]
    W, K = [case["W"]] * T, [case.get("K", B)] * T
    if case["W"] == 0:   # uneven: W of UNEVEN, K in 2W .. 8W
        r = np.random.RandomState(T * 1009 + case["F"])
        W = [int(w) for w in r.choice(UNEVEN, size=T)]
        W = [min(w, case["M"]) for w in W]
        K = [int(r.randint(2 * w, 8 * w + 1)) for w in W]
    P_tr = -(-max(K) // B)
    return dict(W=W, K=K, B=B, P_tr=P_tr, P=P_tr + case.get("P_test", 0), pairs=T * case["L"])


def _directions(case, seed):
    """Direction sines (and vertical sines for a planar array) of the targets, within +-60 and +-20 degrees."""
    r = np.random.RandomState(seed % (1 << 31))
    u = np.sin(np.deg2rad(r.uniform(-60, 60, case["T"])))
    v = np.sin(np.deg2rad(r.uniform(-20, 20, case["T"])))
    if case.get("Nz", 1) > 1:
        return u * np.sqrt(1 - v * v), v, r
    return u, None, r


_STREAM = []


def _capture_stream():
    """The program's one stream for captured passes: batches follow one another on it."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _plan(case, geo, u, v):
    kw = dict(N=case["N"], F=case["F"], L=case["L"], M=case["M"], u=u, W=geo["W"], K=geo["K"], P_train=geo["P_tr"],
              P_test=case.get("P_test", 0), fc=FC, fs=FS, fd=FD, delta=DELTA,
              precision=P.BS_PREC_FP16 if case.get("prec") == "fp16" else P.BS_PREC_FP32)
    if v is not None:
        kw.update(Nz=case["Nz"], Mz=case["Mz"], Wz=[case["Wz"]] * case["T"], v=v)
    return P.Plan(**kw)


# ------------------------------------------------------------------ inputs
def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + k)


def _cn(shape, g):
    """Complex white Gaussian noise of unit variance."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda") * math.sqrt(0.5))


def _steer(u, v, case, freqs):
    """[F][N] wideband response of a plane wave at baseband frequencies `freqs`, reduced in FP64."""
    N, Nz = case["N"], case.get("Nz", 1)
    n = torch.arange(N, device="cuda", dtype=torch.float64)
    ph = torch.floor(n / Nz) * u + (n % Nz) * (v or 0.0)
    ph = torch.outer((FC + freqs) / FD, ph)
    ph = (ph - 2 * torch.round(ph / 2)).to(torch.float32) * math.pi
    return torch.polar(torch.ones_like(ph), ph)


def _cube(case, geo, seed, u, v, r):
    """Raw IQ [P][F][N]: white noise, wideband jammers at 20-40 dB in every record, target echoes in the test records."""
    F, N, Np = case["F"], case["N"], geo["P"]
    g = _gen(seed)
    x = _cn((Np, F, N), g)   # per FFT bin; unitary inverse FFT at the end
    freqs = (torch.fft.fftfreq(F, device="cuda", dtype=torch.float64)) * FS
    apart = 4.0 / N   # jammers stay this far from every target in sine, less where the targets leave no room
    for j in range(case["jam"]):
        for trial in range(400):
            uj = math.sin(math.radians(r.uniform(-60, 60)))
            if np.min(np.abs(u - uj)) >= apart * 0.5 ** (trial // 100):
                break
        vj = math.sin(math.radians(r.uniform(-20, 20)))
        a = _steer(uj, vj if v is not None else None, case, freqs)
        s = _cn((Np, F, 1), g)
        s *= 10 ** (r.uniform(20, 40) / 20) / s.abs().clamp_min(1e-3)   # constant-modulus sweep, random phase
        for p in range(Np):
            x[p].addcmul_(s[p].expand(F, N), a)
    if case.get("P_test"):
        for t in range(0, case["T"], max(1, case["T"] // 16)):   # echoes of some of the targets
            a = _steer(float(u[t]), float(v[t]) if v is not None else None, case, freqs)
            s = _cn((case["P_test"], F, 1), g)
            for p in range(case["P_test"]):
                x[geo["P_tr"] + p].addcmul_(s[p].expand(F, N), a)
    for p in range(Np):
        x[p] = torch.fft.ifft(x[p], dim=0, norm="ortho")
    return x


def _windows(case, seed):
    """Training windows [pair][K][W]: beam noise and up to three strong interferers per window."""
    W, G = case["W"], case["T"] * case["L"]
    K = case.get("K", 2 * W)
    g = _gen(seed)
    z = _cn((G, K, W), g)
    for _ in range(3):
        amp = 10 ** (torch.rand(G, 1, 1, generator=g, device="cuda") * 1.75)
        on = (torch.rand(G, 1, 1, generator=g, device="cuda") < 0.6).float()
        off = torch.arange(W, device="cuda") - torch.rand(G, 1, 1, generator=g, device="cuda") * (W - 1)
        b = torch.sinc(off) * torch.exp(1j * math.pi * off)
        z = z + amp * on * _cn((G, K, 1), g) * b
    z = z.to(torch.complex64).reshape(-1).contiguous()
    return torch.view_as_real(z).reshape(-1).half() if case.get("prec") == "fp16" else z


def _window_plan(case, seed):
    """A plan whose pairs' windows are W beams wide: the paper's planar array above 16 beams, else a linear one."""
    u, v, _ = _directions(dict(case, Nz=4) if case["W"] > 16 else case, seed)
    B, K = 16, case.get("K", 2 * case["W"])
    geo = dict(W=[case["W"]] * case["T"], K=[K] * case["T"], P_tr=-(-K // B))
    arr = dict(N=1024, M=2048)
    if v is not None:
        Wz = max(w for w in (1, 2, 3, 4) if case["W"] % w == 0)
        arr = dict(N=128, M=512, Nz=4, Mz=8, Wz=Wz)
    case = dict(case, F=B * case["L"], **arr)
    return case, geo, _plan(case, geo, u, v), u, v


def _network(case, seed):
    """Parameters, moments and biases of a network in the middle of its training."""
    n_in, n_out, H = learned.feature_count(case["W"]), 1 + case["W"], case["hidden"]
    p = learned.he_uniform_params(n_in, H, n_out, seed % 1000)
    r = np.random.RandomState(seed % (1 << 31))
    p = (p + r.uniform(-0.02, 0.02, p.size)).astype(np.float32)
    m = (r.standard_normal(p.size) * 1e-4).astype(np.float32)
    v = (r.uniform(0.5, 1.5, p.size) * 1e-6).astype(np.float32)
    return n_in, n_out, H, p, m, v


def _loading_head(p, n_out, H):
    """The last layer as training leaves it: loadings around 10, preconditioner entries near diag(R + delta)^-1/2."""
    p = p.copy()
    w3 = p[p.size - n_out * (H + 1):p.size - n_out].reshape(n_out, H)
    w3[0] *= 0.2
    w3[1:] *= 0.02
    p[-n_out] = 1.0
    p[p.size - n_out + 1:] = -0.8
    return p


def _batch(case, seed, n_in, n_out):
    """Features and targets: correlated unit-scale columns, as covariance entries over their trace are."""
    g = _gen(seed, 1)
    mix = torch.randn(8, n_in, generator=g, device="cuda") * 0.3
    X = torch.randn(case["batch"], 8, generator=g, device="cuda") @ mix
    X = X + 0.1 * torch.randn(case["batch"], n_in, generator=g, device="cuda")
    T = torch.randn(case["batch"], n_out, generator=g, device="cuda") * 0.5 + 1.0
    return X.contiguous(), T.contiguous()


def _weights(case, seed):
    """Distortionless-like window weights [pair][W]: smooth main part and a random rest."""
    g = _gen(seed)
    G, W = case["T"] * case["L"], case["W"]
    off = torch.arange(W, device="cuda") - (W - 1) / 2
    base = torch.sinc(off / 1.5) * torch.exp(1j * math.pi * off / 2)
    return (base + 0.2 * _cn((G, W), g)).to(torch.complex64).reshape(-1).contiguous()


def _spectra(case, seed):
    """Beamformed outputs [T][L][P_test * B] of targets at a delay and a Doppler bin each in noise, and the pulse."""
    F, L, T, R = case["F"], case["L"], case["T"], case["P_test"]
    r = np.random.RandomState(seed % (1 << 31))
    k = np.arange(F)
    pulse = np.exp(1j * np.pi * k * k / F)   # a full-band sweep, unit modulus per bin
    pulse /= np.linalg.norm(pulse)
    g = _gen(seed)
    y = _cn((T, R, F), g)
    pk = torch.from_numpy(pulse).to("cuda", torch.complex64)
    f = torch.arange(F, device="cuda", dtype=torch.float32)
    for t in range(T):
        tau, d = int(r.randint(0, F)), int(r.randint(0, R))
        ph = -2 * math.pi * ((f * tau) % F) / F
        dop = torch.exp(2j * math.pi * d * torch.arange(R, device="cuda") / R)
        y[t] += 30.0 * (pk * torch.polar(torch.ones_like(ph), ph)) * dop[:, None]
    q = (torch.arange(F, device="cuda") - F // 2) % F   # bin q = s B + i holds FFT bin (q - F/2) mod F
    y = y[:, :, q].reshape(T, R, L, F // L).permute(0, 2, 1, 3).contiguous()
    return y.reshape(-1), pk


# ----------------------------------------------------------------- prepare
def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        n_in, n_out, H, p, m, v = _network(case, seed)
        net = learned.LoadingMLP(n_in, n_out, H, capacity=case["batch"], params=p)
        net.m.copy_(torch.from_numpy(m))
        net.v.copy_(torch.from_numpy(v))
        X, T = _batch(case, seed, n_in, n_out)
        return dict(case=case, net=net, X=X, T=T)
    if kind == "weights":
        plan = _window_plan(case, seed)[2]
        s = plan.sizes
        return dict(case=case, plan=plan, z=_windows(case, seed),
                    R=torch.empty(s.r_elems, dtype=torch.complex128, device="cuda"),
                    c=torch.empty(s.c_elems, dtype=torch.complex64, device="cuda"),
                    info=torch.empty(s.pairs, dtype=torch.int32, device="cuda"))
    if kind == "loading":
        plan = _window_plan(case, seed)[2]
        n_in, n_out, H, p, _, _ = _network(case, seed)
        p = _loading_head(p, n_out, H)
        s = plan.sizes
        return dict(case=case, plan=plan, z=_windows(case, seed),
                    net=learned.LoadingMLP(n_in, n_out, H, capacity=4096, params=p),
                    zero=torch.zeros(s.pairs, device="cuda"), X=torch.empty(s.pairs * n_in, device="cuda"),
                    R0=torch.empty(s.r_elems, dtype=torch.complex128, device="cuda"),
                    R=torch.empty(s.r_elems, dtype=torch.complex128, device="cuda"),
                    c=torch.empty(s.c_elems, dtype=torch.complex64, device="cuda"),
                    info=torch.empty(s.pairs, dtype=torch.int32, device="cuda"))
    if kind == "detect":
        out, pulse = _spectra(case, seed)
        n = case["T"] * case["P_test"] * case["F"]
        plan = P.Plan(N=16, F=case["F"], L=case["L"], M=16, u=np.zeros(case["T"]), W=[1] * case["T"],
                      K=[1] * case["T"], P_train=1, P_test=case["P_test"], fc=FC, fs=FS, fd=FD, delta=DELTA)
        return dict(case=case, plan=plan, out=out, pulse=pulse,
                    work=torch.empty(2 * n, dtype=torch.complex64, device="cuda"), map=torch.empty(n, device="cuda"),
                    floor=torch.empty(n, device="cuda"), count=torch.empty(case["T"], dtype=torch.int32, device="cuda"),
                    mask=torch.empty(n, dtype=torch.uint8, device="cuda"),
                    peak=torch.empty(case["T"], dtype=torch.int32, device="cuda"))
    geo = _geometry(case)
    u, v, r = _directions(case, seed)
    plan = _plan(case, geo, u, v)
    s = plan.sizes
    if kind in ("lifted", "pattern"):
        st = dict(case=case, plan=plan, c=_weights(case, seed),
                  c_hat=torch.empty(s.pairs * case["N"], dtype=torch.complex64, device="cuda"))
        if kind == "lifted":
            jam = dict(case, jam=2)
            st["xc"] = _channelised(jam, geo, seed, u, r).reshape(-1)
            st["out"] = torch.empty(s.out_elems, dtype=torch.complex64, device="cuda")
        else:
            st["u"] = torch.from_numpy(np.sin(np.deg2rad(np.linspace(-90, 90, case["dirs"])))).cuda()
            st["pattern"] = torch.empty(s.pairs * case["dirs"], device="cuda")
            P.bs_lift(plan, st["c"], st["c_hat"])
        return st
    x = _cube(case, geo, seed, u, v, r).reshape(-1)
    b = P.alloc_buffers(plan)
    st = dict(case=case, plan=plan, b=b)
    b.x.copy_(x)
    if case.get("call") == "graph":
        P.bs_run(plan, b)   # once before the capture, as programs do
        torch.cuda.synchronize()
        st["stream"] = _capture_stream()
        st["graph"] = P.Graph(plan, b, st["stream"])
    return st


def _channelised(case, geo, seed, u, r):
    """A channelised cube [P][F][N] as bs_channelize writes it: noise, jammers and some echoes per bin."""
    F, N = case["F"], case["N"]
    g = _gen(seed, 2)
    x = _cn((geo["P"], F, N), g)
    q = torch.arange(F, device="cuda", dtype=torch.float64)
    freqs = (q - F // 2) / F * FS
    us = [math.sin(math.radians(r.uniform(-60, 60))) for _ in range(case["jam"])] + [float(t) for t in u[:4]]
    for j, uj in enumerate(us):
        a = _steer(uj, None, case, freqs)
        s = _cn((geo["P"], F, 1), g) * (20.0 if j < case["jam"] else 1.0)
        for p in range(geo["P"]):
            x[p].addcmul_(s[p].expand(F, N), a)
    return x


# --------------------------------------------------------------------- run
def run(st):
    kind = st["case"]["kind"]
    if kind == "pass":
        b = st["b"]
        if st["case"]["call"] == "graph":
            st["graph"].launch(st["stream"])
        else:
            P.bs_run(st["plan"], b)
        return dict(c=b.c, out=b.out)
    if kind == "windows":
        b = st["b"]
        P.bs_channelize(st["plan"], b.x, b.xc)
        P.bs_beamspace(st["plan"], b.xc, b.z_train, b.z_test)
        return dict(xc=b.xc, z_train=b.z_train, z_test=b.z_test)
    if kind == "weights":
        P.bs_window_cov(st["plan"], st["z"], st["R"])
        P.bs_mvdr_solve(st["plan"], st["R"], st["c"], st["info"])
        return dict(c=st["c"], info=st["info"])
    if kind == "loading":
        plan, net, n = st["plan"], st["net"], st["plan"].sizes.pairs
        P.bs_window_cov(plan, st["z"], st["R0"], delta_pair=st["zero"])
        if P.lib().bs_features(plan.handle, st["R0"].data_ptr(), st["X"].data_ptr(),
                               torch.cuda.current_stream().cuda_stream):
            raise P.BsError("bs_features")
        Y = net.predict(st["X"], n)
        delta = net.loading(Y, n, fallback=DELTA)
        seed = net.precond(Y, n, st["case"]["W"])
        P.bs_window_cov(plan, st["z"], st["R"], delta_pair=delta)
        P.bs_mvdr_solve_precond(plan, st["R"], seed, st["c"], st["info"])
        return dict(c=st["c"], Y=Y, delta=delta)
    if kind == "train":
        net = st["net"]
        net.loss.zero_()
        net.train_step(st["X"], st["T"], st["case"]["batch"], 1e-3)
        return dict(grad=net.grad, master=net.master, m=net.m, v=net.v)
    if kind == "lifted":
        P.bs_lift(st["plan"], st["c"], st["c_hat"])
        P.bs_apply_lifted(st["plan"], st["xc"], st["c_hat"], st["out"])
        return dict(c_hat=st["c_hat"], out=st["out"])
    if kind == "pattern":
        P.bs_beam_pattern(st["plan"], st["c_hat"], st["u"], st["pattern"])
        return dict(pattern=st["pattern"])
    P.bs_range_doppler(st["plan"], st["out"], st["pulse"], st["work"], st["map"])
    P.bs_cfar(st["plan"], st["map"], 10.0, st["floor"], st["count"], st["mask"], st["peak"])
    return dict(map=st["map"], floor=st["floor"], count=st["count"], mask=st["mask"], peak=st["peak"])


# -------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "train":
        I, H, O, B = learned.feature_count(case["W"]), case["hidden"], 1 + case["W"], case["batch"]
        par, mac = H * I + H + H * H + H + O * H + O, H * I + H * H + O * H
        # parameters and moments read and written once, gradients written, the batch read; forward,
        # weight-gradient and (but for the first layer) input-gradient products
        return dict(bytes=4.0 * (7 * par + B * (I + O)) + 2.0 * par, flops=2.0 * B * (3 * mac - H * I))
    if kind == "loading":
        G, W, K = case["T"] * case["L"], case["W"], 2 * case["W"]
        I, H, O = learned.feature_count(W), case["hidden"], 1 + W
        # windows read, weights, network outputs and loadings written; two covariances are one set of
        # products plus a diagonal, network, solve
        return dict(bytes=float(G * (8 * K * W + 8 * W + 16 * W + 4 * O + 4)),
                    flops=float(G * (4 * W * W * K + 2 * (I * H + H * H + H * O) + 8 * W ** 3 / 3)))
    if kind == "detect":
        n = case["T"] * case["P_test"] * case["F"]
        R, F = case["P_test"], case["F"]
        # outputs read, maps, floors and masks written; FFT per record, DFT over the records
        return dict(bytes=float(n * (8 + 4 + 4 + 1)), flops=float(n * (5 * math.log2(F) + 5 * math.log2(max(2, R)) + 10)))
    if kind == "weights":
        G, W, K = case["T"] * case["L"], case["W"], case["K"]
        return dict(bytes=float(G * (8 * W + 4 + K * W * (4 if case["prec"] == "fp16" else 8))),
                    flops=float(G * (4 * W * W * K + 8 * W ** 3 / 3)))
    geo = _geometry(case)
    G, N, F, L, M = geo["pairs"], case["N"], case["F"], case["L"], case["M"]
    if kind == "lifted":
        Vte = case["P_test"] * geo["B"]
        return dict(bytes=8.0 * (G * case["W"] + G * N + case["P_test"] * F * N + G * Vte),
                    flops=float(G * N * (8 * case["W"] + 8 * Vte)))
    if kind == "pattern":
        return dict(bytes=8.0 * G * N + 8.0 * case["dirs"] + 4.0 * G * case["dirs"], flops=8.0 * G * N * case["dirs"])
    Vte = case["P_test"] * geo["B"]
    W, K = np.array(geo["W"], float), np.array(geo["K"], float)
    cube = geo["P"] * F * N
    fft = 5 * cube * math.log2(F) + 5 * geo["P"] * F * M * math.log2(M)
    if kind == "windows":
        # the raw cube read, the channelised cube and the windows written; two FFTs
        return dict(bytes=float(16 * cube + L * ((4 if case["prec"] == "fp16" else 8) * W * K + 8 * W * Vte).sum()),
                    flops=float(fft))
    # the raw cube read, weights and outputs written; two FFTs, covariance, solve and output per pair
    return dict(bytes=float(8 * cube + L * (8 * W.sum() + 8 * Vte * case["T"])),
                flops=float(fft + L * (4 * W * W * K + 8 * W ** 3 / 3 + 8 * W * Vte).sum()))


# ------------------------------------------------------------------- exact
def _axis_window(u, M, W, f):
    """Start of the W beams nearest to a squinted spatial frequency and the windowed steering sum."""
    x = math.pi * u * (f / FD) * M / (2 * math.pi)
    return int(math.floor(x - W / 2 + 1)) % M


def _steered(u, M, N, W, f):
    """Window beams and S D a(Omega) along one axis, by direct summation."""
    om = math.pi * u * (f / FD)
    start = _axis_window(u, M, W, f)
    beams = (start + np.arange(W)) % M
    n = np.arange(N)
    return beams, np.exp(1j * (om * n[None, :] - 2 * np.pi * ((beams[:, None] * n[None, :]) % M) / M)).sum(1) / math.sqrt(M)


def _exact_pass(case, seed):
    geo = _geometry(case)
    u, v, r = _directions(case, seed)
    x = _cube(case, geo, seed, u, v, r)
    F, N, L, M, T, B = case["F"], case["N"], case["L"], case["M"], case["T"], geo["B"]
    Nz, Mz, Wz = case.get("Nz", 1), case.get("Mz", 1), case.get("Wz", 1)
    Vte = case["P_test"] * B
    q = (torch.arange(F, device="cuda") - F // 2) % F
    xc = torch.empty((geo["P"], F, N), dtype=torch.complex128, device="cuda")
    for p in range(geo["P"]):
        xc[p] = torch.fft.fft(x[p].to(torch.complex128), dim=0, norm="ortho")[q]
    del x
    c = [[None] * L for _ in range(T)]
    ztr, zte = [[None] * L for _ in range(T)], [[None] * L for _ in range(T)]
    out = torch.empty((T, L, Vte), dtype=torch.complex128, device="cuda")
    groups = sorted(set(zip(geo["W"], geo["K"])))
    for s in range(L):
        f = FC + ((s - L // 2 + 1 - 0.5) / L) * FS
        y = xc[:, s * B:(s + 1) * B].reshape(-1, N // Nz, Nz)
        yb = torch.fft.fft(torch.fft.fft(y, n=Mz, dim=2), n=M // Mz, dim=1).reshape(-1, M) / math.sqrt(M)
        for W, K in groups:
            ts = [t for t in range(T) if (geo["W"][t], geo["K"][t]) == (W, K)]
            idx, a = [], []
            for t in ts:
                bx, ax = _steered(u[t], M // Mz, N // Nz, W // Wz, f)
                if v is not None:
                    bz, az = _steered(v[t], Mz, Nz, Wz, f)
                    idx.append((bx[:, None] * Mz + bz[None, :]).reshape(-1))
                    a.append(np.kron(ax, az))
                else:
                    idx.append(bx)
                    a.append(ax)
            idx = torch.from_numpy(np.array(idx)).cuda()
            a = torch.from_numpy(np.array(a)).cuda()
            z = yb[:K][:, idx].permute(1, 2, 0)                       # [targets][W][K]
            if case["kind"] == "windows":
                zt = yb[geo["P_tr"] * B:][:, idx].permute(1, 0, 2)
                for k, t in enumerate(ts):
                    ztr[t][s], zte[t][s] = z[k].T.reshape(-1), zt[k].reshape(-1)
                continue
            R = z @ z.mH / K + DELTA * torch.eye(W, device="cuda", dtype=torch.complex128)
            w = torch.cholesky_solve(a[..., None], torch.linalg.cholesky(R))[..., 0]
            w = w / (a.conj() * w).sum(1, keepdim=True)
            zt = yb[geo["P_tr"] * B:][:, idx].permute(1, 0, 2)        # [targets][Vte][W]
            o = (zt * w.conj()[:, None, :]).sum(2)
            for k, t in enumerate(ts):
                c[t][s] = w[k]
                out[t, s] = o[k]
    if case["kind"] == "windows":
        zr = torch.cat([w for row in ztr for w in row])
        return dict(xc=xc.reshape(-1), z_train=torch.view_as_real(zr).reshape(-1) if case["prec"] == "fp16" else zr,
                    z_test=torch.cat([w for row in zte for w in row]))
    cc = torch.cat([w for row in c for w in row])
    return dict(c=cc, out=out.reshape(-1))


def _layers(p, n_in, H, n_out):
    w, o = {}, 0
    for k, shape in (("W1", (H, n_in)), ("b1", (H,)), ("W2", (H, H)), ("b2", (H,)), ("W3", (n_out, H)), ("b3", (n_out,))):
        n = int(np.prod(shape))
        w[k] = torch.from_numpy(p[o:o + n].astype(np.float64)).cuda().reshape(shape)
        o += n
    for k in ("W1", "W2", "W3"):   # the products read the weights in BF16
        w[k] = w[k].to(torch.bfloat16).double()
    return w


def _exact_train(case, seed):
    n_in, n_out, H, p, m, v = _network(case, seed)
    X, T = (t.double() for t in _batch(case, seed, n_in, n_out))
    w = _layers(p, n_in, H, n_out)
    z1 = X @ w["W1"].T + w["b1"]
    h1 = z1.clamp_min(0)
    z2 = h1 @ w["W2"].T + w["b2"]
    h2 = z2.clamp_min(0)
    y = h2 @ w["W3"].T + w["b3"]
    dy = 2 * (y - T) / y.numel()
    d2 = (dy @ w["W3"]) * (z2 > 0)
    d1 = (d2 @ w["W2"]) * (z1 > 0)
    g = torch.cat([t.reshape(-1) for t in (d1.T @ X, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0))])
    p, m, v = (torch.from_numpy(t.astype(np.float64)).cuda() for t in (p, m, v))
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    return dict(grad=g, master=p - 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8), m=m, v=v)


def _window_pairs(case, seed):
    """Windows [pair][K][W], unloaded covariances and windowed steering vectors in 64 bits."""
    W, T, L = case["W"], case["T"], case["L"]
    K = case.get("K", 2 * W)
    z = _windows(case, seed)
    z = torch.view_as_complex(z.double().reshape(-1, 2)) if case.get("prec") == "fp16" else z.to(torch.complex128)
    z = z.reshape(T * L, K, W)
    arr, _, _, u, v = _window_plan(case, seed)
    Nz, Mz, Wz = arr.get("Nz", 1), arr.get("Mz", 1), arr.get("Wz", 1)
    a = []
    for t in range(T):
        for s in range(L):
            f = FC + ((s - L // 2 + 1 - 0.5) / L) * FS
            ax = _steered(u[t], arr["M"] // Mz, arr["N"] // Nz, W // Wz, f)[1]
            a.append(ax if v is None else np.kron(ax, _steered(v[t], Mz, Nz, Wz, f)[1]))
    return z.transpose(1, 2) @ z.conj() / K, torch.from_numpy(np.array(a)).cuda()


def _exact_weights(case, seed):
    R, a = _window_pairs(case, seed)
    R = R + DELTA * torch.eye(case["W"], device="cuda", dtype=torch.float64)
    c = torch.cholesky_solve(a[..., None], torch.linalg.cholesky(R))[..., 0]
    return dict(c=(c / (a.conj() * c).sum(1, keepdim=True)).reshape(-1), info=None)


def _exact_loading(case, seed):
    W, K, T, L = case["W"], 2 * case["W"], case["T"], case["L"]
    G = T * L
    R, a = _window_pairs(case, seed)
    tau = R.diagonal(dim1=1, dim2=2).real.mean(1)
    il = torch.tril_indices(W, W, -1, device="cuda")
    low = R[:, il[0], il[1]] / tau[:, None]
    an = a / torch.linalg.vector_norm(a, dim=1, keepdim=True)
    X = torch.cat([R.diagonal(dim1=1, dim2=2).real / tau[:, None], low.real, low.imag, an.real, an.imag,
                   tau.log10()[:, None], torch.full((G, 1), math.log10(K / W), device="cuda")], 1)
    n_in, n_out, H, p, _, _ = _network(case, seed)
    p = _loading_head(p, n_out, H)
    w = _layers(p, n_in, H, n_out)
    h = (X @ w["W1"].T + w["b1"]).clamp_min(0)
    h = (h @ w["W2"].T + w["b2"]).clamp_min(0)
    Y = h @ w["W3"].T + w["b3"]
    delta = (10.0 ** Y[:, 0]).clamp(0.1, 1e4)
    Rl = R + delta[:, None, None] * torch.eye(W, device="cuda", dtype=torch.float64)
    c = torch.cholesky_solve(a[..., None], torch.linalg.cholesky(Rl))[..., 0]
    c = c / (a.conj() * c).sum(1, keepdim=True)
    return dict(c=c.reshape(-1), Y=Y.reshape(-1), delta=delta)


def _exact_lift(case, seed, u):
    """[pair][N] antenna-space weights by direct summation over the window."""
    W, N, M, L, T = case["W"], case["N"], case["M"], case["L"], case["T"]
    c = _weights(case, seed).to(torch.complex128).reshape(T, L, W)
    starts = np.array([[_axis_window(u[t], M, W, FC + ((s - L // 2 + 1 - 0.5) / L) * FS) for s in range(L)] for t in range(T)])
    st = torch.from_numpy(starts).cuda()
    n = torch.arange(N, device="cuda")
    ch = torch.zeros((T, L, N), dtype=torch.complex128, device="cuda")
    for w in range(W):
        ph = 2 * math.pi * (((st[..., None] + w) * n) % M).double() / M
        ch += c[..., w, None] * torch.polar(torch.ones_like(ph), ph)
    return ch / math.sqrt(M)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pass", "windows"):
        return _exact_pass(case, seed)
    if kind == "weights":
        return _exact_weights(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "loading":
        return _exact_loading(case, seed)
    L, B = case["L"], case["F"] // case["L"]
    if kind == "detect":
        y, pk = _spectra(case, seed)
        F, T, R = case["F"], case["T"], case["P_test"]
        q = (torch.arange(F, device="cuda") - F // 2) % F
        Y = torch.empty((T, R, F), dtype=torch.complex128, device="cuda")
        Y[:, :, q] = y.to(torch.complex128).reshape(T, L, R, B).permute(0, 2, 1, 3).reshape(T, R, F)
        rp = torch.fft.ifft(Y * pk.to(torch.complex128).conj(), dim=2, norm="ortho")
        mp = torch.fft.fft(rp, dim=1).abs() ** 2
        floor = (mp.sum(1, keepdim=True) - mp) / (R - 1)
        return dict(map=mp.reshape(-1), floor=floor.reshape(-1), count=None, mask=None, peak=None)
    geo = _geometry(case)
    u, _, r = _directions(case, seed)
    ch = _exact_lift(case, seed, u)
    N, T = case["N"], case["T"]
    if kind == "lifted":
        xc = _channelised(dict(case, jam=2), geo, seed, u, r)[geo["P_tr"]:]
        Vte = case["P_test"] * B
        out = torch.empty((T, L, Vte), dtype=torch.complex128, device="cuda")
        for s in range(L):
            y = xc[:, s * B:(s + 1) * B].reshape(Vte, N).to(torch.complex128)
            out[:, s] = ch[:, s].conj() @ y.T
        return dict(c_hat=ch.reshape(-1), out=out.reshape(-1))
    # patterns of the FP32 weights that the call is given
    ch = ch.to(torch.complex64).to(torch.complex128)
    dirs = torch.from_numpy(np.sin(np.deg2rad(np.linspace(-90, 90, case["dirs"])))).cuda()
    n = torch.arange(N, device="cuda", dtype=torch.float64)
    pat = torch.empty((T, L, case["dirs"]), dtype=torch.float64, device="cuda")
    for s in range(L):
        ratio = (FC + ((s - L // 2 + 1 - 0.5) / L) * FS) / FD
        ph = math.pi * torch.outer(n, dirs * ratio)
        e = torch.polar(torch.ones_like(ph), ph)
        w = ch[:, s]
        pat[:, s] = (w.conj() @ e).abs() / (torch.linalg.vector_norm(w, dim=1, keepdim=True) * math.sqrt(N))
    return dict(pattern=pat.reshape(-1))
