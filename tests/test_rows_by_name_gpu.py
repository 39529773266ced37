"""The row-streaming kernel by name at its long horizons: fields bit for bit those of the tile kernel
(both sum a row's segments and the disc's rows in the same order), at remainders of its sample groups,
with fixed bands, and long and short batches in turn on one handle; one step against the oracle.

Tolerance of a step: 4e-6 max|u| (the derivation in test_parity_gpu.py)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

# gs samples a CTA: 12 or 8 warps over n / 128 strips; 640 / R = 12 leaves two warps out
LATTICES = [(128, 12, 12), (256, 12, 6), (384, 12, 4), (512, 12, 3), (640, 12, 2), (128, 16, 8), (256, 16, 4),
            (512, 16, 2), (1024, 16, 1)]


@pytest.mark.parametrize("n,R,gs", LATTICES)
@pytest.mark.parametrize("band", [0, 24])
def test_rows_match_tiles(gpu_lib, n, R, gs, band):
    import torch
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, tau=2e-3, ic=2, nsteps=2)
    rows, tile = mf.Model(algo=mf.ALGO_ROWS, **kw), mf.Model(algo=mf.ALGO_PREFIX_TMA, **kw)
    rows.set_band_height(band, 4)
    for ns in (2 * gs + 1, 1, 2 * gs + 1):
        u0 = torch.empty((ns, n, n), dtype=torch.float32, device="cuda")
        mf.mfmc_init_fields(rows, list(range(40, 40 + ns)), u0)
        out = []
        for g in (rows, tile):
            uT = torch.full_like(u0, 7.0)
            ooi = torch.empty(ns, dtype=torch.float64, device="cuda")
            mf.mfmc_solve_fields(g, u0, ns, uT=uT, ooi=ooi)
            out.append((uT, ooi))
        torch.cuda.synchronize()
        assert torch.equal(out[0][0], out[1][0])
        assert float((out[0][1] - out[1][1]).abs().max()) <= 1e-12  # FP64 sums in another order


@pytest.mark.parametrize("n,R", [(256, 12), (512, 16)])
def test_rows_one_step_against_the_oracle(gpu_lib, n, R):
    import torch
    mf = gpu_lib
    kw = dict(n=n, delta=R / n, eps=0.02, tau=2e-3, ic=2, nsteps=1)
    g, o = mf.Model(algo=mf.ALGO_ROWS, **kw), O.OracleModel(**kw)
    u0 = torch.empty((2, n, n), dtype=torch.float32, device="cuda")
    uT = torch.empty_like(u0)
    mf.mfmc_init_fields(g, [3, 4], u0)
    mf.mfmc_solve_fields(g, u0, 2, uT=uT)
    torch.cuda.synchronize()
    ref, _ = o.solve(u0[1].cpu().numpy().astype(np.float64), 0.02)
    assert np.abs(uT[1].cpu().numpy() - ref).max() <= 4e-6


def test_auto_long_short_long(gpu_lib):
    # AUTO runs the short batch on the tile kernel, over the scratch that the long ones use plain
    import torch
    mf = gpu_lib
    kw = dict(n=512, delta=16 / 512, eps=0.02, tau=2e-3, ic=2, nsteps=2)
    auto, tile = mf.Model(**kw), mf.Model(algo=mf.ALGO_PREFIX_TMA, **kw)
    u0 = torch.empty((45, 512, 512), dtype=torch.float32, device="cuda")
    mf.mfmc_init_fields(auto, list(range(45)), u0)
    ref = torch.empty_like(u0)
    mf.mfmc_solve_fields(tile, u0, 45, uT=ref)
    for ns in (2, 45, 2, 45, 45):
        uT = torch.full_like(u0, 7.0)
        mf.mfmc_solve_fields(auto, u0, ns, uT=uT)
        torch.cuda.synchronize()
        assert torch.equal(uT[:ns], ref[:ns]) and bool((uT[ns:] == 7.0).all())
