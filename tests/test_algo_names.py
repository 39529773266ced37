"""Which algorithms may be named for a model: a property of its descriptor alone (no device work)."""
import pytest

from paper_2310_10750_gb300 import mfmc


def accepted(n, R, algo):
    try:
        mfmc.Model(n=n, delta=R / n, nsteps=1, algo=algo)
        return True
    except mfmc.MfmcError as e:
        assert e.status == mfmc.MFMC_EINVAL
        return False


NAMES = (mfmc.ALGO_RESIDENT, mfmc.ALGO_ROWS, mfmc.ALGO_PREFIX_TMA, mfmc.ALGO_PREFIX, mfmc.ALGO_DIRECT, mfmc.ALGO_SPECTRAL)


@pytest.mark.parametrize("n", [128, 256, 384, 512, 640, 768, 896, 1024, 1152, 2048])
@pytest.mark.parametrize("R", [2, 3, 8, 12, 16, 24])
def test_row_streaming_lattices(n, R):
    rows = {2: True, 8: True, 12: n <= 640, 16: n in (128, 256, 512, 1024)}.get(R, False)
    assert accepted(n, R, mfmc.ALGO_ROWS) == rows


@pytest.mark.parametrize("n,R,ok", [(16, 4, True), (64, 8, True), (112, 5, True), (128, 8, True), (128, 12, False),
                                    (72, 4, False), (192, 4, False), (256, 2, False), (256, 4, True), (256, 6, True),
                                    (256, 8, True), (256, 5, False), (512, 8, False)])
def test_resident_lattices(n, R, ok):
    assert accepted(n, R, mfmc.ALGO_RESIDENT) == ok


@pytest.mark.gpu
@pytest.mark.parametrize("n,R,ns", [(256, 6, 5), (256, 4, 3), (384, 12, 9), (640, 16, 2), (768, 12, 2), (128, 4, 5)])
def test_tuning_changes_no_name(gpu_lib, n, R, ns):
    import torch
    before = [accepted(n, R, a) for a in NAMES]
    g = mfmc.Model(n=n, delta=R / n, nsteps=2, ic=2)
    u0 = torch.empty((ns, n, n), dtype=torch.float32, device="cuda")
    mfmc.mfmc_init_fields(g, list(range(ns)), u0)
    ooi = torch.empty(ns, dtype=torch.float64, device="cuda")
    mfmc.mfmc_solve_fields(g, u0, ns, ooi=ooi)
    torch.cuda.synchronize()
    assert [accepted(n, R, a) for a in NAMES] == before
    assert accepted(n, R, g.info().algo)
