"""A tile shape pinned before AUTO's choice holds where that choice is another kernel."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,ns", [(64, 4, 3), (256, 8, 3), (512, 16, 2), (512, 16, 45)])
def test_pinned_shape_survives_auto(gpu_lib, n, R, ns):
    import torch
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, tau=1e-3, nsteps=2, ic=2)
    pin = 9
    u0 = torch.empty((ns, n, n), dtype=torch.float32, device="cuda")
    out = []
    for pinned in (True, False):
        g = mf.Model(**kw)
        if pinned:
            g.set_tile_variant(pin)
            mf.mfmc_init_fields(g, list(range(ns)), u0)
        uT = torch.empty_like(u0)
        mf.mfmc_solve_fields(g, u0, ns, uT=uT)
        torch.cuda.synchronize()
        assert g.info().algo != mf.ALGO_PREFIX_TMA
        if pinned:
            assert g.info().tile_variant == pin
        out.append(uT)
    assert torch.equal(out[0], out[1])
    # named, the tile kernel runs the pinned shape
    g = mf.Model(**kw)
    g.set_tile_variant(pin)
    mf.mfmc_solve_fields(g, u0, ns)
    a, b = torch.empty(ns, dtype=torch.float64, device="cuda"), torch.empty(ns, dtype=torch.float64, device="cuda")
    mf.mfmc_solve_fields_algo(g, mf.ALGO_PREFIX_TMA, u0, ns, ooi=a)
    t = mf.Model(algo=mf.ALGO_PREFIX_TMA, **kw)
    t.set_tile_variant(pin)
    mf.mfmc_solve_fields(t, u0, ns, ooi=b)
    torch.cuda.synchronize()
    assert g.info().tile_variant == pin and torch.equal(a, b)
