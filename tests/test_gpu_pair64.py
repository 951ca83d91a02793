"""FP64 two-detector path against the generic FP64 kernels: every split and row length,
an odd and a single detector, T and TQU, a periodic map, laws that are white, ordinary or
too steep for the tabulated powers of two, and tabulated weights."""
import numpy as np
import pytest

import gen

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


def both(cmm, scan, noise, table=None):
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=cmm.PREC_F64)
    if table is not None:
        op.noise.set_table(table)
    m = torch.as_tensor(gen.random_maps(scan.ncomp, scan.ny, scan.nx, 1, cfg=391)[0], device="cuda:0")
    pair = op.apply(m).clone()
    op.set_pair_packing(False)
    ref = op.apply(m)
    assert float(ref.norm()) > 0
    # FFT and binning rounding of either path is below 1e-14 of A m (a filter's
    # amplification of at most a few hundred here): a tenth of the FP64 operator's bound
    return float((pair - ref).norm() / ref.norm()), float((pair - ref).abs().max() / ref.abs().max())


@pytest.mark.parametrize("log_nt", range(13, 21))
@pytest.mark.parametrize("n_det,ncomp", [(1, 1), (3, 3), (8, 3)])
def test_sizes(cmm, log_nt, n_det, ncomp):
    full = gen.small_scan(cfg=391, ny=48, nx=50, n_t=1 << log_nt, ncols=4, nrows=2, throw_px=60.0, ncomp=ncomp)
    scan = full.subset(np.arange(n_det))
    noise = gen.noise_params(n_det, fknee=2.0, alpha=3.5, scatter=0.2, cfg=391)
    assert max(both(cmm, scan, noise)) < 1e-11


def test_periodic(cmm):
    scan = gen.bccb_scan(8, 16, 1 << 13, diagonal=True)
    assert max(both(cmm, scan, gen.noise_params(scan.n_det, fknee=2.0, alpha=3.5))) < 1e-11


@pytest.mark.parametrize("fknee,alpha", [((0.0, 2.0, 2.0), (3.5, 3.5, 3.5)), ((100.0, 1.0, 2.0), (60.0, 3.5, -1.0)),
                                         ((0.0, 50.0, 0.0), (1.0, 300.0, 1.0))])
def test_laws(cmm, fknee, alpha):
    scan = gen.small_scan(cfg=392, ny=24, nx=20, n_t=1 << 14, ncols=3, nrows=1, throw_px=30.0)
    noise = gen.Noise(np.array([1.0, 0.7, 1.3]), np.array(fknee), np.array(alpha))
    assert max(both(cmm, scan, noise)) < 1e-11


def test_table(cmm):
    scan = gen.small_scan(cfg=393, ny=24, nx=20, n_t=1 << 13, ncols=3, nrows=1, throw_px=30.0)
    w = 1.0 + 0.5 * np.sin(np.arange(scan.n_t // 2 + 1) / 7.0)[None] * np.array([[0.2], [0.9], [0.5]])
    assert max(both(cmm, scan, gen.noise_params(3), w)) < 1e-11


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 1e-5)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("log_nt,n_det,ncomp", [(13, 1, 1), (15, 5, 3), (16, 8, 3), (18, 3, 3)])
def test_rhs_of_stored_data(cmm, prec, tol, dtype, log_nt, n_det, ncomp):
    """The right-hand side on the two-detector path against the one-detector kernels
    (FP32: the operator's bound; the data are white, so no large offsets are filtered)."""
    full = gen.small_scan(cfg=394, ny=30, nx=32, n_t=1 << log_nt, ncols=4, nrows=2, throw_px=40.0, ncomp=ncomp)
    scan = full.subset(np.arange(n_det))
    op = cmm.Operator(cmm.Context(0), scan, gen.noise_params(n_det, scatter=0.2, cfg=394), precision=prec)
    g = torch.Generator(device="cuda:0").manual_seed(394)
    tod = torch.randn((n_det, scan.n_t), dtype=dtype, device="cuda:0", generator=g)
    pair = op.rhs(tod).clone()
    op.set_pair_packing(False)
    ref = op.rhs(tod)
    assert float((pair - ref).norm()) <= tol * float(ref.norm())
    assert float((pair - ref).abs().max()) <= tol * float(ref.abs().max())
