"""A mixed-radix lattice (n = 96) in one launch with tile-form lattices: the CTA then has sixteen warps
where MFMC_ALGO_SPECTRAL's own launch has nine, and the results are the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("other", [64, 88, 128])
def test_generic_items_beside_tile_items(gpu_lib, other):
    mf = gpu_lib

    def model(n, algo):
        return mf.Model(n=n, delta=0.125, kernel=1, delta_hf=0.25, eps=0.04219, tau=0.01, nsteps=5, ic=2, algo=algo)

    seeds = np.arange(24, dtype=np.uint64) + 9
    pair = [model(96, mf.ALGO_AUTO), model(other, mf.ALGO_AUTO)]
    f, u = mf.mfmc_solve_batch_mixed([pair[i % 2] for i in range(24)], seeds)
    for k, n in enumerate((96, other)):
        fs, us = mf.mfmc_solve_batch([model(n, mf.ALGO_SPECTRAL)] * 12, seeds[k::2])
        assert np.array_equal(f[k::2], fs) and np.array_equal(u[k::2], us)
