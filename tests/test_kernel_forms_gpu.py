"""The forms the dispatch chooses by size, at the sizes where each can go wrong: tile edges,
remainders, the smallest and largest lattice, and each side of a rule.

Tolerances: one FP32 step 4e-6 max|u| and k steps at most k times that (the derivation in
test_parity_gpu.py: the disc sum's rounded adds, scaled by c1); beta2 > 0 fields and OoIs as in
test_active_set_gpu.py (max |F| <= 1e-11 per step on both sides, uT rounded to FP32); forms that are
documented to round alike are compared bit for bit."""
import numpy as np
import pytest

import oracle as O
from oracle import beta2_oracle as B2

pytestmark = pytest.mark.gpu


def fields(mf, g, seeds, keep=None):
    """(u0, uT, ooi) of the samples `keep` (all by default), solved in one batch."""
    import torch
    ns = len(seeds)
    u0 = torch.empty((ns, g.n, g.n), dtype=torch.float32, device="cuda")
    uT = torch.empty_like(u0)
    ooi = torch.empty(ns, dtype=torch.float64, device="cuda")
    eps = torch.tensor(mf.mfmc_sample_eps(g, seeds), dtype=torch.float64, device="cuda")
    mf.mfmc_init_fields(g, seeds, u0)
    mf.mfmc_solve_fields(g, u0, ns, eps=eps, uT=uT, ooi=ooi)
    torch.cuda.synchronize()
    k = list(range(ns)) if keep is None else keep
    return u0[k].cpu().numpy().astype(np.float64), uT[k].cpu().numpy(), ooi.cpu().numpy()[k]


def seeds_of(k, base):
    return np.arange(k, dtype=np.uint64) + base


# resident strips (blocks of four rows to R = 4, of eight above): lattices from 16 (eight strips a warp) to 128 (one row a warp), with idle
# lanes (48: two groups of 12, 96: 24 of 32, 112: 28 of 32) and idle groups
@pytest.mark.parametrize("n,R", [(16, 1), (16, 3), (16, 4), (32, 2), (48, 4), (80, 3), (96, 1), (96, 4), (112, 2),
                                 (128, 1), (128, 4), (16, 6), (32, 8), (48, 5), (64, 8), (96, 6), (112, 8)])
@pytest.mark.parametrize("ic", [1, 2])
def test_resident_strips(gpu_lib, n, R, ic):
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, tau=2e-3, ic=ic, ic_amp=0.05)
    for steps in (1, 5):
        g = mf.Model(nsteps=steps, algo=mf.ALGO_RESIDENT, **kw)
        o = O.OracleModel(nsteps=steps, **kw)
        u0, uT, f = fields(mf, g, seeds_of(3, 10 * n + R))
        for i in range(3):
            ref, mean = o.solve(u0[i], 0.02)
            assert np.abs(uT[i] - ref).max() <= steps * 4e-6 * max(0.1, np.abs(u0[i]).max())
            assert abs(f[i] - 0.5 * (1.0 + mean)) <= steps * 4e-6
        assert np.abs(uT).max() <= 1.0


@pytest.mark.parametrize("n,R,many", [(16, 2, 1300), (32, 4, 700), (64, 1, 200), (64, 4, 200)])
def test_resident_strips_do_not_depend_on_the_batch(gpu_lib, n, R, many):
    # a small batch takes strips of four rows, a large one strips of eight: the same bits
    mf = gpu_lib
    g = mf.Model(n=n, delta=R / n, eps=0.02, tau=2e-3, ic=1, ic_amp=0.05, nsteps=6, algo=mf.ALGO_RESIDENT)
    _, ua, fa = fields(mf, g, seeds_of(2, 7))
    _, ub, fb = fields(mf, g, seeds_of(many, 7), keep=[0, 1])
    assert np.array_equal(ua, ub) and np.array_equal(fa, fb)


# the resident form with the field in shared memory: one CTA a sample (n = 128), clusters of four
# (n = 256; 40 samples are more than one round of clusters), where AUTO takes it
@pytest.mark.parametrize("n,R,ns", [(128, 5, 3), (128, 6, 3), (128, 8, 155), (256, 4, 5), (256, 6, 40), (256, 8, 40)])
@pytest.mark.parametrize("ic", [1, 2])
def test_resident_clusters(gpu_lib, n, R, ns, ic):
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, tau=2e-3, ic=ic, ic_amp=0.05)
    keep = sorted({0, ns // 2, ns - 1})
    for steps in (1, 4):
        g = mf.Model(nsteps=steps, algo=mf.ALGO_RESIDENT if n == 128 else mf.ALGO_AUTO, **kw)
        o = O.OracleModel(nsteps=steps, **kw)
        u0, uT, f = fields(mf, g, seeds_of(ns, 5 * n + R), keep)
        assert n == 128 or g.info().algo == mf.ALGO_RESIDENT
        for i in range(len(keep)):
            ref, mean = o.solve(u0[i], 0.02)
            assert np.abs(uT[i] - ref).max() <= steps * 4e-6 * max(0.1, np.abs(u0[i]).max())
            assert abs(f[i] - 0.5 * (1.0 + mean)) <= steps * 4e-6
        assert np.abs(uT).max() <= 1.0


def test_resident_clusters_served_with_their_own_step_counts(gpu_lib):
    # the server runs 256^2 requests in clusters; steps differ from sample to sample
    mf = gpu_lib
    kw = dict(n=256, delta=8 / 256, eps=0.03, tau=5e-3, ic=2)
    g = mf.Model(nsteps=4, **kw)
    o = O.OracleModel(nsteps=4, **kw)
    srv = mf.Server(1 << 30, 64)
    try:
        steps = [1, 4, 3, 2]
        tickets = [srv.submit(g, 300 + i, params=mf.make_params(1, nsteps=[k])[0]) for i, k in enumerate(steps)]
        srv.drain()
        for i, k in enumerate(steps):
            u0 = o.initial_field(300 + i)
            _, mean = o.solve(u0, 0.03, nsteps=k)
            assert abs(srv.poll(tickets[i])[0] - 0.5 * (1.0 + mean)) <= k * 4e-6
    finally:
        srv.close()


@pytest.mark.parametrize("n,R,many,few", [(512, 16, 45, 3), (256, 12, 200, 5), (384, 6, 70, 4), (512, 8, 50, 3)])
def test_rows_and_tiles_agree_on_each_side_of_the_batch_rule(gpu_lib, n, R, many, few):
    # AUTO's choice (the row kernel for a long batch, the tile kernel for a short one or where it
    # is faster) has the tile kernel's bits
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, eps_lo=0.016, eps_hi=0.024, tau=1e-3, ic=1, ic_amp=0.05, nsteps=3)
    ga, gt = mf.Model(**kw), mf.Model(algo=mf.ALGO_PREFIX_TMA, **kw)
    keep = [0, 1, 2]
    _, ut, ft = fields(mf, gt, seeds_of(many, 77), keep)
    for ns in (many, few):
        _, ua, fa = fields(mf, ga, seeds_of(ns, 77), keep)
        assert np.array_equal(ua, ut) and np.array_equal(fa, ft), ns
    if (n, R) == (512, 16):
        assert ga.info().algo == mf.ALGO_ROWS


def test_forms_auto_alone_chooses_stay_refused(gpu_lib):
    # lattices that AUTO has not tuned in this process
    import torch
    mf = gpu_lib
    u0 = torch.zeros((1, 768, 768), dtype=torch.float32, device="cuda")
    for n, R in ((640, 16), (768, 12)):
        with pytest.raises(mf.MfmcError) as e:
            mf.Model(n=n, delta=R / n, algo=mf.ALGO_ROWS)
        assert e.value.status == mf.MFMC_EINVAL
        with pytest.raises(mf.MfmcError) as e:
            mf.mfmc_solve_fields_algo(mf.Model(n=n, delta=R / n, nsteps=1), mf.ALGO_ROWS, u0, 1)
        assert e.value.status == mf.MFMC_EINVAL


@pytest.mark.parametrize("n,R,ns", [(256, 8, 5), (512, 16, 45)])
def test_the_algorithm_a_query_reports_can_be_asked_for(gpu_lib, n, R, ns):
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, tau=1e-3, ic=2, nsteps=2)
    ga = mf.Model(**kw)
    _, ua, fa = fields(mf, ga, seeds_of(ns, 31), [0, ns - 1])
    gb = mf.Model(algo=ga.info().algo, **kw)
    _, ub, fb = fields(mf, gb, seeds_of(ns, 31), [0, ns - 1])
    assert np.array_equal(ua, ub) and np.array_equal(fa, fb)


@pytest.mark.parametrize("n", [64, 88, 128])
def test_spectral_samples_do_not_depend_on_the_batch(gpu_lib, n):
    mf = gpu_lib
    g = mf.Model(n=n, delta=0.125, kernel=1, delta_hf=0.25, eps=0.04219, tau=0.01, ic=2, nsteps=7,
                 algo=mf.ALGO_SPECTRAL)
    _, ub, fb = fields(mf, g, seeds_of(5, 40))
    for i in (0, 4):
        _, ua, fa = fields(mf, g, seeds_of(1, 40 + i))
        assert np.array_equal(ua[0], ub[i]) and fa[0] == fb[i]


# beta2 > 0 on the on-chip lattices: the direct sum (49 disc points) and the transforms (113 and more),
# a horizon that is no integer, both kernels
@pytest.mark.parametrize("n,delta,kernel", [(64, 4 / 64, 0), (64, 6 / 64, 0), (88, 4 / 88, 0), (88, 0.1875, 1),
                                            (128, 4 / 128, 0), (128, 0.0625, 1)])
def test_active_set_lattices(gpu_lib, n, delta, kernel):
    mf = gpu_lib
    steps = 3
    kw = dict(n=n, delta=delta, kernel=kernel, delta_hf=0.25 if kernel else 0.0, eps=0.04219, tau=0.01, nsteps=steps, ic=2)
    g = mf.Model(beta2=0.05, **kw)
    o = O.OracleModel(**kw)
    seeds = seeds_of(2, 60 + n)
    _, uT, f = fields(mf, g, seeds)
    fr, _, ur, _ = B2.solve_sample(o, int(seeds[1]), 0.05, steps)
    assert abs(f[1] - fr) <= 1e-8 * fr
    assert np.abs(uT[1] - ur).max() <= 1e-6
    assert np.abs(uT).max() <= 1.0


@pytest.mark.parametrize("n", [8, 44, 100, 1028])
def test_nuclei_fields_at_row_block_remainders(gpu_lib, n):
    # both sides round FP64 values to FP32: one ulp
    mf = gpu_lib
    import torch
    g = mf.Model(n=n, delta=2 / n, nsteps=1, ic=2)
    o = O.OracleModel(n=n, delta=2 / n, nsteps=1, ic=2)
    u0 = torch.empty((2, n, n), dtype=torch.float32, device="cuda")
    mf.mfmc_init_fields(g, seeds_of(2, 9), u0)
    for i in range(2):
        ref = o.initial_field(9 + i)
        ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
        assert np.all(np.abs(u0[i].cpu().numpy().astype(np.float64) - ref) <= ulp)
