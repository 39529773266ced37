"""The caller's fields need only the alignment of a float: a view that starts one, two or three floats
into an allocation gives every algorithm's results bit for bit."""
import pytest

pytestmark = pytest.mark.gpu

CASES = [
    ("AUTO", 256, 8, 5, {}), ("AUTO", 256, 4, 5, {}), ("AUTO", 512, 16, 3, {}), ("AUTO", 512, 16, 45, {}),
    ("AUTO", 512, 8, 3, {}), ("RESIDENT", 64, 4, 3, {}), ("RESIDENT", 64, 2, 700, {}), ("RESIDENT", 96, 6, 3, {}),
    ("RESIDENT", 128, 8, 3, {}), ("ROWS", 256, 8, 9, {}), ("PREFIX_TMA", 96, 3, 3, {}), ("PREFIX_KAHAN", 96, 3, 3, {}),
    ("PREFIX", 64, 4, 3, {}), ("DIRECT", 64, 4, 3, {}), ("DIRECT", 64, 16, 2, {}), ("PLAIN", 64, 4, 2, {}),
    ("PREFIX_TMA", 64, 4, 2, dict(bc=1, bc_value=-1.0)), ("WEIGHTED", 64, 8, 2, dict(kernel=1, delta_hf=0.25)),
    ("FFT", 64, 8, 2, {}), ("SPECTRAL", 1024, 32, 2, {}), ("SPECTRAL", 64, 8, 3, {}), ("SPECTRAL", 88, 8, 3, {}),
    ("SPECTRAL", 96, 8, 3, {}), ("AUTO", 64, 8, 2, dict(beta2=0.05)), ("AUTO", 48, 6, 2, dict(beta2=0.05)),
]


@pytest.mark.parametrize("algo,n,R,ns,kw", CASES)
def test_fields_off_a_16_byte_boundary(gpu_lib, algo, n, R, ns, kw):
    import torch
    mf = gpu_lib
    # (a collar's initial fields are the periodic ones)
    g = mf.Model(n=n, delta=R / n, eps=0.04, tau=2e-3, nsteps=2, ic=2, algo=getattr(mf, "ALGO_" + algo), **kw)
    nn = ns * n * n

    def field(off):
        return torch.full((nn + 4,), 7.0, dtype=torch.float32, device="cuda")[off:off + nn].view(ns, n, n)

    u0 = field(0)
    mf.mfmc_init_fields(g, list(range(ns)), u0)

    def solve(i, o):
        src, dst = field(i), field(o)
        src.copy_(u0)
        ooi = torch.empty(ns, dtype=torch.float64, device="cuda")
        for _ in range(2):  # the second call may replay a graph
            mf.mfmc_solve_fields(g, src, ns, uT=dst, ooi=ooi)
        torch.cuda.synchronize()
        assert torch.equal(src, u0)
        return dst.clone(), ooi

    uT, ooi = solve(0, 0)
    assert float(uT.abs().max()) <= 1.0
    for i, o in ((1, 0), (0, 1), (2, 3)):
        vT, voi = solve(i, o)
        assert torch.equal(vT, uT) and torch.equal(voi, ooi), (i, o)


def test_what_cannot_be_aligned_is_refused(gpu_lib):
    import torch
    mf = gpu_lib
    g = mf.Model(n=64, delta=4 / 64, nsteps=2, ic=2, algo=mf.ALGO_PREFIX)
    buf = torch.zeros(2 * 64 * 64, dtype=torch.float32, device="cuda")
    out = torch.zeros(2 * 64 * 64, dtype=torch.float32, device="cuda")
    ooi = torch.empty(1, dtype=torch.float64, device="cuda")
    for u0, uT in ((buf.data_ptr() + 2, None), (buf.data_ptr(), out.data_ptr() + 1)):
        with pytest.raises(mf.MfmcError) as e:
            mf.mfmc_solve_fields(g, u0, 1, uT=uT, ooi=ooi)
        assert e.value.status == mf.MFMC_EINVAL

    def noalloc(u0, uT):  # (no scratch for an aligned copy)
        return mf._L.mfmc_solve_fields_noalloc(g.handle, None, u0, 1, uT, None, ooi.data_ptr(), None)

    assert noalloc(buf.data_ptr() + 4, None) == mf.MFMC_EINVAL
    assert noalloc(buf.data_ptr(), out.data_ptr() + 8) == mf.MFMC_EINVAL
    assert noalloc(buf.data_ptr(), out.data_ptr()) == mf.MFMC_OK
    torch.cuda.synchronize()
