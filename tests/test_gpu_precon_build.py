"""The set-up of the preconditioners at its edges: hit blocks over spans that do not fill
a block of samples or detectors, and circulant modes with and without floored
eigenvalues, against the FP64 oracle."""
import numpy as np
import pytest

import gen
from oracle import mapmaker as om

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def cmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_7473_gb300 import build
    build.build()
    from paper_1309_7473_gb300 import cmm as c
    return c


def scan_of(n_t, ncols, nrows, ncomp):
    return gen.small_scan(cfg=371, ny=20, nx=24, n_t=n_t, ncols=ncols, nrows=nrows, spacing_px=0.7, throw_px=30.0,
                          ncomp=ncomp)


@pytest.mark.parametrize("n_t,ncols,nrows", [(1, 1, 1), (31, 3, 1), (33, 11, 3), (1000, 43, 3), (4097, 16, 8)])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_mask_of_ragged_scans(cmm, n_t, ncols, nrows, ncomp):
    full = scan_of(8192, ncols, nrows, ncomp)
    scan = gen.Scan(**{**full.__dict__, "bore": np.ascontiguousarray(full.bore[2000:2000 + n_t])})
    got, _ = cmm.Pointing(cmm.Context(0), scan).mask()
    np.testing.assert_array_equal(got.ravel(), om.pixel_mask(scan).ravel())


@pytest.mark.parametrize("n_t,ncols,nrows", [(32, 5, 1), (4096, 8, 4), (4096, 13, 10)])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_binned_blocks(cmm, n_t, ncols, nrows, ncomp):
    scan = scan_of(n_t, ncols, nrows, ncomp)
    noise = gen.noise_params(scan.n_det, fknee=2.0, alpha=3.5, scatter=0.2, cfg=371)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=cmm.PREC_F64)
    oop = om.make_operator(scan, noise)
    m = gen.random_maps(ncomp, scan.ny, scan.nx, 1, cfg=371)[0]
    z = cmm.Precon(op, cmm.PRECON_BINNED).apply(torch.as_tensor(m, device="cuda:0")).cpu().numpy()
    ref = om.BlockPrecon(oop)(m)
    # FP64 sums of at most 1e4 samples and inverses of condition <= 1e3
    assert np.abs(z - ref).max() <= 1e-10 * max(np.abs(ref).max(), 1e-300)


@pytest.mark.parametrize("pd_eps", [1e-6, 0.2, 0.9])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_floored_modes(cmm, pd_eps, ncomp):
    scan = gen.small_scan(cfg=372, ny=18, nx=20, n_t=1 << 12, ncols=4, nrows=3, throw_px=30.0, ncomp=ncomp)
    noise = gen.noise_params(scan.n_det, fknee=2.0, alpha=3.5, scatter=0.2, cfg=372)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=cmm.PREC_F64)
    ref = om.CirculantPrecon(om.make_operator(scan, noise), taper_sigma=6.0, pd_eps=pd_eps)
    pc = cmm.Precon(op, cmm.PRECON_CIRCULANT, taper_sigma_px=6.0, pd_eps=pd_eps)
    m = gen.random_maps(ncomp, scan.ny, scan.nx, 1, cfg=372)[0]
    z = pc.apply(torch.as_tensor(m, device="cuda:0")).cpu().numpy()
    zr = ref(m)
    assert pc.clamped() == ref.n_clamped
    # the FP64 bound of the circulant apply (1e-10): condition of a mode block <= 1 / pd_eps
    assert np.abs(z - zr).max() <= 1e-10 / min(1.0, 1e4 * pd_eps) * np.abs(zr).max()
