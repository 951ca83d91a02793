"""The right-hand side when the two detectors of one sequence differ: every detector's
pixels against the FP64 oracle to the operator's own bound, whatever its partner holds
(more noise, a cut detector's garbage, a glitch, a drift, no finite number)."""
import numpy as np
import pytest

import gen
from oracle import mapmaker as om

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# The operators' bounds, here for every detector by itself (FP64: a tenth of it).  A
# detector carries at most about four times its own rounding (FP32 3e-7, BF16 3e-3, FP64
# 5e-16), before the binning averages it.
TOL = {0: 1e-11, 1: 1e-5, 2: 2e-2}


@pytest.fixture(scope="module")
def cmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_7473_gb300 import build
    build.build()
    from paper_1309_7473_gb300 import cmm as c
    return c


def setup(n_det, log_nt, ncomp, sigma):
    """Detectors side by side, each sweeping columns of its own, and the pixels that only
    detector d sees."""
    focal = np.stack([30.0 * (np.arange(n_det) - 0.5 * (n_det - 1)), np.zeros(n_det)], 1)
    # four crossings of a pixel at different angles, three of which a TQU block needs
    scan = gen.make_scan(cfg=397, ny=24, nx=30 * n_det, n_t=1 << log_nt, focal_px=focal, throw_px=20.0,
                         segments=((0.25, 2.0, 10.0, True), (0.25, -2.0, -10.0, False), (0.25, 20.0, 30.0, True),
                                   (0.25, -20.0, -30.0, False)), ncomp=ncomp)
    pix = om.sample_pixels(scan, np.arange(n_det))
    seen = np.zeros((n_det, scan.npix), bool)
    for d in range(n_det):
        seen[d, pix[d][pix[d] >= 0]] = True
    alone = seen & (seen.sum(0) == 1) & om.pixel_mask(scan)
    assert alone.sum(1).min() > 50
    return scan, gen.Noise(np.asarray(sigma, float), np.full(n_det, 2.0), np.full(n_det, 3.5)), alone


def data(scan, noise):
    return np.random.default_rng(397).standard_normal((scan.n_det, scan.n_t)) * noise.sigma[:, None]


def errors(got, want, alone, ncomp):
    got, want = got.reshape(ncomp, -1), want.reshape(ncomp, -1)
    return [np.linalg.norm((got - want)[:, a]) / np.linalg.norm(want[:, a]) for a in alone]


def rhs(cmm, op, d, dtype=torch.float64):
    out = op.rhs(torch.as_tensor(d, dtype=dtype, device="cuda:0"))
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("ratio", [1.0, 10.0, 1000.0])
@pytest.mark.parametrize("log_nt,ncomp,dtype,chunk", [(13, 1, torch.float32, 0), (16, 3, torch.float64, 3),
                                                      (18, 1, torch.float32, 0)])
def test_noise_ratios(cmm, prec, ratio, log_nt, ncomp, dtype, chunk):
    scan, noise, alone = setup(5, log_nt, ncomp, [1.0, ratio, ratio, 1.0, 1.0])
    d = data(scan, noise).astype(np.float32).astype(np.float64)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec, det_chunk=chunk)
    want = om.rhs(om.make_operator(scan, noise), d)
    assert max(errors(rhs(cmm, op, d, dtype), want, alone, ncomp)) <= TOL[prec]


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("what", ["cut", "glitch", "drift"])
def test_loud_partner(cmm, prec, what):
    scan, noise, alone = setup(4, 14, 1, np.ones(4))
    d = data(scan, noise)
    w = om.filter_weights(noise, scan.n_t, scan.f_samp)
    if what == "cut":
        d[1] *= 1e6
        w[1] = 0.0
    elif what == "glitch":
        d[1, 4321] += 1e6
    else:
        d[1] += 1e4 * np.sin(2 * np.pi * 3.3 * np.arange(scan.n_t) / scan.n_t)
    d[3] = 0.0
    d = d.astype(np.float32).astype(np.float64)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec)
    if what == "cut":
        op.noise.set_table(w)
    got = rhs(cmm, op, d)
    want = om.rhs(om.make_operator(scan, noise, w=w if what == "cut" else None), d)
    err = errors(got, want, alone[[0, 2]], 1)
    assert max(err) <= TOL[prec]
    zero = alone[3] | (alone[1] if what == "cut" else False)
    assert np.abs(got.ravel()[zero]).max() == 0.0   # no data and no weight: exactly nothing


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("scale", [1e-25, 1e25])
def test_scales(cmm, prec, scale):
    """Data far from their noise model, whose squares leave FP32."""
    scan, noise, alone = setup(4, 13, 1, np.ones(4))
    d = (data(scan, noise) * np.array([scale, 1.0, scale, scale])[:, None]).astype(np.float32).astype(np.float64)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec)
    want = om.rhs(om.make_operator(scan, noise), d)
    assert max(errors(rhs(cmm, op, d), want, alone, 1)) <= TOL[prec]
    # and the same operator's next call starts afresh
    d2 = data(scan, noise)
    assert max(errors(rhs(cmm, op, d2), om.rhs(om.make_operator(scan, noise), d2), alone, 1)) <= TOL[prec]


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite_stays_with_its_detector(cmm, prec, bad):
    scan, noise, alone = setup(5, 13, 1, np.ones(5))
    d = data(scan, noise)
    want = om.rhs(om.make_operator(scan, noise), d)
    d[1, 77] = bad
    d[4, 5000] = bad
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec)
    got = rhs(cmm, op, d)
    assert max(errors(got, want, alone[[0, 2, 3]], 1)) <= TOL[prec]
    assert not np.isfinite(got.ravel()[alone[1] | alone[4]]).any()
    d = data(scan, noise)
    assert max(errors(rhs(cmm, op, d), want, alone, 1)) <= TOL[prec]


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("ratio", [1.0, 1000.0])
def test_correlated(cmm, prec, ratio):
    scan, noise, alone = setup(5, 13, 1, [1.0, ratio, 1.0, 1.0, ratio])
    corr = gen.corr_noise(scan.det_off, r=2)
    d = data(scan, noise).astype(np.float32).astype(np.float64)
    d[2] = 0.0   # only the common modes are left of it
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec, corr=corr)
    want = om.rhs(om.make_operator(scan, noise, corr=corr), d)
    assert max(errors(rhs(cmm, op, d), want, alone, 1)) <= TOL[prec]


def test_more_pairs_than_one_sweep(cmm):
    """Every one of 1100 pairs unbalanced, against the one-detector packing."""
    n = 2199
    full = gen.small_scan(cfg=398, ny=120, nx=140, n_t=1 << 13, ncols=8, nrows=4, throw_px=140.0, ncomp=1)
    idx = np.arange(n) % 32
    scan = full.subset(idx)
    noise = gen.Noise(np.where(np.arange(n) % 2, 1000.0, 1.0), np.full(n, 2.0), np.full(n, 3.5))
    g = torch.Generator(device="cuda:0").manual_seed(398)
    tod = torch.randn((n, scan.n_t), device="cuda:0", generator=g)
    tod[1::2] *= 1000.0
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=1)
    got = op.rhs(tod).clone()
    op.set_pair_packing(False)
    want = op.rhs(tod)
    assert float(want.norm()) > 0
    assert float((got - want).norm()) <= TOL[1] * float(want.norm())
