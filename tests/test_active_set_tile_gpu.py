"""The beta2 > 0 solver's on-chip kernel (n = 64, 88, 128): what it reports when a solve cannot
succeed.  n = 32 runs the other kernel, whose report is the one to match."""
import numpy as np
import pytest

import oracle as O
from oracle import beta2_oracle as B2

pytestmark = pytest.mark.gpu


def model(mf, n, R, **kw):
    return mf.Model(n=n, delta=R / n, eps=0.04219, tau=0.01, nsteps=3, ic=2, beta2=0.05, **kw)


# discs of 49 points (the direct sum, which leaves a NaN where it is) and of 197 (the transforms,
# which spread it)
@pytest.mark.parametrize("n", [32, 64, 88, 128])
@pytest.mark.parametrize("R", [4, 8])
def test_non_finite_samples_report_timeout(gpu_lib, n, R):
    mf = gpu_lib
    g = model(mf, n, R)
    seeds = np.arange(3, dtype=np.uint64) + 17
    good, _ = mf.mfmc_solve_batch([g] * 3, seeds)
    mu, eta = [0.95] * 4, [[0.0, 0.0]] * 4
    bad = [mf.make_params(3, theta=[None, ([np.nan] + mu[1:], eta), None]),
           mf.make_params(3, theta=[None, (mu, [[np.inf, 0.0]] + eta[1:]), None]),
           mf.make_params(3, eps=[0.04219, np.inf, 0.04219])]
    for p in bad:
        with pytest.raises(mf.MfmcError) as e:
            mf.mfmc_solve_batch([g] * 3, seeds, params=p)
        assert e.value.status == mf.MFMC_ETIMEOUT
        again, _ = mf.mfmc_solve_batch([g] * 3, seeds)  # the model and the device stay usable
        assert np.array_equal(again, good)


@pytest.mark.parametrize("n", [64, 88, 128])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_one_non_finite_value_stops_its_sample_alone(gpu_lib, n, value):
    # a stopped sample's outputs are left as they were; its neighbours keep every bit
    import torch
    mf = gpu_lib
    g = model(mf, n, 8)
    u0 = torch.empty((3, n, n), dtype=torch.float32, device="cuda")
    mf.mfmc_init_fields(g, np.arange(3, dtype=np.uint64) + 5, u0)

    def solve(u):
        uT = torch.full_like(u, 7.0)
        ooi = torch.full((3,), 7.0, dtype=torch.float64, device="cuda")
        mf.mfmc_solve_fields(g, u, 3, uT=uT, ooi=ooi)
        torch.cuda.synchronize()
        return uT.cpu().numpy(), ooi.cpu().numpy()

    uT, ooi = solve(u0)
    v0 = u0.clone()
    v0[1, n // 2, 3] = value
    vT, voi = solve(v0)
    assert np.all(vT[1] == 7.0) and voi[1] == 7.0
    for i in (0, 2):
        assert np.array_equal(vT[i], uT[i]) and voi[i] == ooi[i]


# The passes that steps of these samples take with every correction solved to 1e-5, the tolerance of the
# kernel for other lattices: a caller's bound of as many passes is enough.
@pytest.mark.parametrize("n,delta,kernel,steps,ns,passes", [
    (64, 4 / 64, 0, 10, 20, 5), (64, 0.125, 1, 10, 20, 6), (64, 0.25, 1, 10, 20, 6), (88, 0.1875, 1, 8, 12, 6),
    (128, 0.25, 1, 6, 12, 6), (128, 0.0625, 1, 6, 12, 7)])
def test_a_tight_pass_bound_is_met(gpu_lib, n, delta, kernel, steps, ns, passes):
    mf = gpu_lib
    g = mf.Model(n=n, delta=delta, kernel=kernel, delta_hf=0.25 if kernel else 0.0, eps=0.04219, tau=0.01,
                 nsteps=steps, ic=2, beta2=0.05)
    seeds = np.arange(ns, dtype=np.uint64) + 50
    free, _ = mf.mfmc_solve_batch([g] * ns, seeds)
    g.set_iteration_limits(newton_max=passes)
    bound, _ = mf.mfmc_solve_batch([g] * ns, seeds)
    assert np.abs(bound - free).max() <= 1e-8  # both to max |F| <= 1e-11 a step
    newton, _ = mf.mfmc_model_solver_stats(g)
    assert newton <= passes * ns * steps
    g.set_iteration_limits(newton_max=2)
    with pytest.raises(mf.MfmcError) as e:
        mf.mfmc_solve_batch([g] * ns, seeds)
    assert e.value.status == mf.MFMC_ETIMEOUT


# Steps whose active set is close to cycling, which loose corrections alone tip over (small eps, large
# beta2): the solve ends, and agrees with the oracle as in test_active_set_gpu.py.
@pytest.mark.parametrize("n,eps,tau,beta2,seed", [
    (64, 0.002688285082775925, 0.01, 5.0, 5), (64, 0.003613438343137776, 0.03, 1.0, 6), (64, 0.006, 0.01, 5.0, 3),
    (64, 0.006, 0.01, 5.0, 4), (128, 0.002, 0.03, 1.0, 5)])
def test_steps_close_to_cycling_end(gpu_lib, n, eps, tau, beta2, seed):
    mf = gpu_lib
    kw = dict(n=n, delta=0.125, kernel=1, delta_hf=0.25, eps=eps, tau=tau, nsteps=4, ic=2)
    f, _ = mf.mfmc_solve_batch([mf.Model(beta2=beta2, **kw)], np.array([seed], dtype=np.uint64))
    ref, _, _, _ = B2.solve_sample(O.OracleModel(**kw), seed, beta2, 4)
    assert abs(f[0] - ref) <= 1e-8 * ref
