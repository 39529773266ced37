"""Workloads of the library, through its public entry points (paper_2310_10750_gb300/mfmc.py).

A case is one call: a batch of samples of one fidelity advanced over its time steps.  The sizes
are those of the library's own configurations: the plain Monte Carlo, single-fidelity and
large configurations, the delta = 1/32 hierarchy (64^2 .. 512^2), and the paper's nine models
(Gaussian kernel on 1/h = 128, 88, 64) without and with its beta2 = 0.05.

exact() is the same scheme in FP64 with torch only: the disc sum as a circular convolution by
FFT, the projection step, and for beta2 > 0 a semismooth Newton solve of the step's equation.
"""
import math

import numpy as np
import torch

from paper_2310_10750_gb300 import mfmc

EPS, EPS_LO, EPS_HI = 0.02, 0.016, 0.024        # the constant-kernel configurations
EPS_PAPER, DELTA_HF = math.sqrt(0.00178), 0.25  # the paper's models


def _const(name, n, R, ns, steps, ic="noise", bc=0, entry="fields"):
    return dict(name=name, kind="const", n=n, R=float(R), ns=ns, steps=steps, tau=1e-3, ic=ic, bc=bc, beta2=0.0,
                entry=entry)


def _paper(name, n, delta, ns, steps, beta2=0.0):
    return dict(name=name, kind="gauss", n=n, R=delta * n, ns=ns, steps=steps, tau=0.01, ic="nuclei", bc=0,
                beta2=beta2, entry="fields")


def listed():
    return [
        # plain Monte Carlo on the small parity lattice: the smallest call, 32 samples
        _const("mc64_r4", 64, 4, 32, 200, ic="uniform"),
        # the coarse levels of the delta = 1/32 hierarchy, which take almost all of an MFMC plan's samples
        _const("lf64_r2", 64, 2, 4096, 1000),
        _const("lf128_r4", 128, 4, 1001, 500),
        # the single-fidelity benchmark batch
        _const("mc256_r8", 256, 8, 512, 500),
        # a 64-sample pilot of the 256^2 level from seeds to OoIs: initial fields, solve and read-back
        _const("pilot256_batch", 256, 8, 64, 500, ic="nuclei", entry="batch"),
        # the hierarchy's high-fidelity pilot
        _const("hf512_r16", 512, 16, 64, 250),
        # the large configuration (3209-point disc)
        _const("hf1024_r32", 1024, 32, 64, 100),
        # the paper's models on its three meshes, T = 1; delta/h = 16.5 on 1/h = 88
        _paper("paper128", 128, 0.25, 256, 100),
        _paper("paper88", 88, 0.1875, 256, 100),
        _paper("paper64", 64, 0.125, 1000, 100),
        # the same with beta2 = 0.05: a 50-sample high-fidelity pilot, and a plan's worth of the cheap model
        _paper("beta2_128", 128, 0.25, 50, 20, beta2=0.05),
        _paper("beta2_64", 64, 0.25, 1000, 10, beta2=0.05),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))


def draw(rng):
    kind = rng.choice(["const", "const", "const", "gauss", "gauss", "large", "beta2", "beta2"])
    if kind == "const":
        n = rng.choice([64, 96, 128, 192, 256, 384, 512])
        R = rng.choice([r for r in (2, 3, 4, 6, 8, 12, 16) if n // 64 <= r <= n // 16])
        steps = _log_int(rng, 50, 500)
        ns = _log_int(rng, 4, min(4096, 3.2e9 / (n * n * steps) / (1 + R / 8)))
        bc = 1 if rng.random() < 0.15 else 0
        c = _const("", n, R, ns, steps, ic=rng.choice(["noise", "noise", "nuclei", "uniform"]), bc=bc)
    elif kind == "large":
        steps = _log_int(rng, 10, 60)
        c = _const("", 1024, rng.choice([16, 24, 32]), _log_int(rng, 8, 64), steps)
    else:
        n = rng.choice([64, 88, 128])
        delta = rng.choice([0.25, 0.1875, 0.125])
        if kind == "gauss":
            c = _paper("", n, delta, _log_int(rng, 3, 1000), rng.randint(25, 100))
        else:
            c = _paper("", n, delta, _log_int(rng, 3, 152), rng.randint(4, 12), beta2=0.05)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------- inputs
def _nuclei(n, theta):
    """Four nuclei of phase -1 (mu, eta_x, eta_y per nucleus: theta [ns][12]) on the n x n torus."""
    ax = torch.arange(n, dtype=torch.float64, device="cuda") / n
    th = theta.to("cuda").reshape(-1, 12, 1, 1)
    s = 0.0
    for k, (cx, cy) in enumerate(((0.25, 0.5), (0.75, 0.5), (0.5, 0.25), (0.5, 0.75))):
        dx = ax.view(1, 1, n) - (cx + th[:, 4 + 2 * k])
        dy = ax.view(1, n, 1) - (cy + th[:, 5 + 2 * k])
        dx = dx - torch.floor(dx + 0.5)
        dy = dy - torch.floor(dy + 0.5)
        s = s + th[:, k] * torch.exp(-36.0 * (dx * dx + dy * dy))
    return (1.0 - 2.0 * s).clamp(-1.0, 1.0).float()


def _inputs(case, seed):
    """Initial fields (FP32) and per-sample eps (FP64) on the GPU."""
    n, ns = case["n"], case["ns"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def unit(*shape):
        return torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda")

    if case["kind"] == "gauss":
        eps = torch.full((ns,), EPS_PAPER, dtype=torch.float64, device="cuda")
    else:
        eps = EPS_LO + (EPS_HI - EPS_LO) * unit(ns)
    if case["ic"] == "nuclei":
        theta = torch.cat([0.9 + 0.1 * unit(ns, 4), -0.025 + 0.05 * unit(ns, 8)], 1)
        return _nuclei(n, theta), eps
    if case["ic"] == "uniform":
        return (0.1 * torch.rand(ns, n, n, generator=g, device="cuda") - 0.05), eps
    z = 0.05 * torch.randn(ns, n, n, generator=g, device="cuda")
    u = z + torch.roll(z, 1, 1) + torch.roll(z, -1, 1) + torch.roll(z, 1, 2) + torch.roll(z, -1, 2)
    return (u / 5.0).clamp(-1.0, 1.0), eps


def _seeds(case, seed):
    return np.arange(case["ns"], dtype=np.uint64) + np.uint64(1000003 * (seed % 1000000) + 20231016)


def _model(case):
    kw = dict(n=case["n"], delta=case["R"] / case["n"], tau=case["tau"], nsteps=case["steps"], beta2=case["beta2"])
    if case["kind"] == "gauss":
        return mfmc.Model(kernel=mfmc.KERNEL_GAUSSIAN, delta_hf=DELTA_HF, eps=EPS_PAPER, ic=mfmc.IC_NUCLEI, **kw)
    return mfmc.Model(eps=EPS, eps_lo=EPS_LO, eps_hi=EPS_HI, ic=mfmc.IC_NUCLEI,
                      bc=mfmc.BC_COLLAR if case["bc"] else mfmc.BC_PERIODIC, bc_value=-1.0, **kw)


def prepare(case, seed):
    """The model handle, the inputs and the output buffers a caller holds."""
    st = dict(case=case, model=_model(case))
    if case["entry"] == "batch":
        st.update(seeds=_seeds(case, seed), models=[st["model"]] * case["ns"])
        return st
    u0, eps = _inputs(case, seed)
    st.update(u0=u0, eps=eps, uT=torch.empty_like(u0),
              ooi=torch.empty(case["ns"], dtype=torch.float64, device="cuda"))
    return st


def run(st):
    """One solve: final fields and outputs of interest (the batch call returns the OoIs).

    The small Gaussian lattices return the fields alone: there the OoI, also computed, is the
    FP64 mean of that same FP32 field and carries only its rounding.
    """
    case = st["case"]
    if case["entry"] == "batch":
        return {"ooi": mfmc.mfmc_solve_batch(st["models"], st["seeds"])[0]}
    mfmc.mfmc_solve_fields(st["model"], st["u0"], case["ns"], eps=st["eps"], uT=st["uT"], ooi=st["ooi"],
                           stream=torch.cuda.current_stream())
    if case["kind"] == "gauss" and case["beta2"] == 0.0:
        return {"uT": st["uT"]}
    return {"uT": st["uT"], "ooi": st["ooi"]}


def work(case):
    """Bytes: the fields in and out once (a solve could stay on chip).  Flops: per point and step
    the disc sum by row prefixes (4R + 9) or by a real 2-D FFT pair (10 log2 n, product, update),
    whichever is less; beta2 > 0 adds four Newton corrections of five multigrid-CG iterations."""
    n, R, ns, steps = case["n"], case["R"], case["ns"], case["steps"]
    fft = 10.0 * math.log2(n) + 8.0
    per = min(4.0 * R + 9.0, fft) if case["kind"] == "const" else fft
    if case["beta2"] > 0:
        per += 4.0 * (5.0 * 130.0 + 16.0)
    fields = 4.0 * n * n * ns
    return {"bytes": (fields if case["entry"] == "batch" else 2.0 * fields) + 16.0 * ns,
            "flops": per * n * n * ns * steps}


# ------------------------------------------------------------------------------------- FP64
def _sm64(seeds, stream, i):
    """Output number stream 2^32 + i + 1 of SplitMix64 started at each seed, as a unit double."""
    z = seeds + np.uint64(((stream << 32) + i + 1) * 0x9E3779B97F4A7C15 % (1 << 64))
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _batch_inputs(case, seed):
    s = _seeds(case, seed)
    theta = np.empty((len(s), 12))
    for k in range(4):
        theta[:, k] = 0.9 + 0.1 * _sm64(s, 2, 3 * k)
        theta[:, 4 + 2 * k] = -0.025 + 0.05 * _sm64(s, 2, 3 * k + 1)
        theta[:, 5 + 2 * k] = -0.025 + 0.05 * _sm64(s, 2, 3 * k + 2)
    eps = EPS_LO + (EPS_HI - EPS_LO) * _sm64(s, 0, 0)
    return _nuclei(case["n"], torch.from_numpy(theta)), torch.from_numpy(eps).cuda()


def _stencil(case, m):
    """rfft2 of the disc weights (divided by eps^2) on an m x m torus, and their sum."""
    n, Rf = case["n"], case["R"]
    r2max = math.floor(Rf * Rf * (1.0 + 1e-12))
    R = math.floor(Rf + 1e-9)
    h = 1.0 / n
    k = np.zeros((m, m))
    for dy in range(-R, R + 1):
        for dx in range(-R, R + 1):
            r2 = dx * dx + dy * dy
            if r2 > r2max:
                continue
            if case["kind"] == "gauss":
                s = DELTA_HF / 3.0
                k[dy % m, dx % m] = h * h * 4.0 / (math.pi * s ** 4) * math.exp(-r2 * h * h / (s * s))
            else:
                k[dy % m, dx % m] = 8.0 * h * h / (math.pi * (Rf * h) ** 4)
    k = torch.from_numpy(k).cuda()
    return torch.fft.rfft2(k).real.contiguous(), float(k.sum())


def _newton(u, g, w, cg, tau, beta2, lam):
    """w with tau (w - beta2 Lap w) + P((w + g) / cg) = u, by Newton and FFT-preconditioned CG."""
    def lap(v):  # times h^2
        return torch.roll(v, 1, 1) + torch.roll(v, -1, 1) + torch.roll(v, 1, 2) + torch.roll(v, -1, 2) - 4.0 * v
    n = u.shape[-1]
    tb2 = tau * beta2 * n * n

    def dot(a, b):
        return (a * b).sum((1, 2), keepdim=True)

    old = None
    for _ in range(60):
        x = (w + g) / cg
        F = tau * w - tb2 * lap(w) + x.clamp(-1.0, 1.0) - u
        m = (x.abs() < 1.0).double()
        if old is not None and bool((m == old).all()) and float(F.abs().max()) <= 1e-12:
            break
        old = m
        pre = 1.0 / (tau + tb2 * lam + (m.mean((1, 2), keepdim=True) / cg))
        r, d = -F, torch.zeros_like(F)
        stop = 1e-10 * r.abs().amax((1, 2), keepdim=True) + 1e-14
        z = torch.fft.irfft2(torch.fft.rfft2(r) * pre, s=(n, n))
        p, rz = z, dot(r, z)
        for k in range(400):
            q = tau * p - tb2 * lap(p) + m / cg * p
            a = rz / dot(p, q).clamp_min(1e-300)
            d = d + a * p
            r = r - a * q
            if k % 8 == 7 and bool((r.abs().amax((1, 2), keepdim=True) <= stop).all()):
                break
            z = torch.fft.irfft2(torch.fft.rfft2(r) * pre, s=(n, n))
            rz, was = dot(r, z), rz
            p = z + rz / was.clamp_min(1e-300) * p
        w = w + d
    return w


def exact(case, seed):
    """run()'s outputs in FP64, a block of samples at a time."""
    n, tau, steps = case["n"], case["tau"], case["steps"]
    batch = case["entry"] == "batch"
    u0, eps = _batch_inputs(case, seed) if batch else _inputs(case, seed)
    pad = math.floor(case["R"] + 1e-9) if case["bc"] else 0
    m = n + 2 * pad
    kh, ksum = _stencil(case, m)
    fy, fx = torch.arange(n, device="cuda"), torch.arange(n // 2 + 1, device="cuda")
    lam = (4.0 - 2.0 * torch.cos(2.0 * math.pi * fy.double() / n).view(1, n, 1)
           - 2.0 * torch.cos(2.0 * math.pi * fx.double() / n).view(1, 1, -1))
    uT = torch.empty(case["ns"], n, n, dtype=torch.float64, device="cuda")
    block = max(1, (1 << 25) // (m * m))
    for s in range(0, case["ns"], block):
        u = u0[s:s + block].double()
        e2 = (eps[s:s + block] ** 2).view(-1, 1, 1)
        cg, w = e2 * ksum, None
        for _ in range(steps):
            v = torch.nn.functional.pad(u, (pad, pad, pad, pad), value=-1.0) if pad else u
            S = torch.fft.irfft2(torch.fft.rfft2(v) * kh, s=(m, m))
            g = e2 * (S[:, pad:pad + n, pad:pad + n] if pad else S) + u  # c_F = 1
            v = ((u + tau * g) / (1.0 + tau * cg)).clamp_(-1.0, 1.0)
            if case["beta2"] > 0:
                w = _newton(u, g, cg * v - g if w is None else w, cg, tau, case["beta2"], lam)
                v = ((w + g) / cg).clamp(-1.0, 1.0)
            u = v
        uT[s:s + block] = u
    ooi = 0.5 * (1.0 + uT.mean((1, 2)))
    if batch:
        return {"ooi": ooi}
    if case["kind"] == "gauss" and case["beta2"] == 0.0:
        return {"uT": uT}
    return {"uT": uT, "ooi": ooi}
