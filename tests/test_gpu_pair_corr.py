"""Correlated noise on the two-detector path against the one-detector packing: every
number of modes, row length and split, an odd and a single detector, the law and a table,
FP32 and BF16, A and the right-hand side; and the tables after a change of packing."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = {1: 1e-5, 2: 2e-2}   # the FP32 and BF16 operators' bounds


@pytest.fixture(scope="module")
def cmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_7473_gb300 import build
    build.build()
    from paper_1309_7473_gb300 import cmm as c
    return c


def modes(scan, r):
    v = np.stack([np.ones(scan.n_det), scan.det_off[:, 0] / 128.0, scan.det_off[:, 1] / 128.0,
                  np.cos(np.arange(scan.n_det))], 1)[:, :r]
    return gen.CorrNoise(v / np.maximum(np.linalg.norm(v, axis=0), 1e-12), np.array([3.0, 1.0, 1.0, 0.5])[:r],
                         np.array([2.0, 1.0, 1.0, 3.0])[:r], np.array([3.0, 2.5, 2.5, 1.5])[:r])


def close(a, b, tol):
    assert float(b.norm()) > 0
    assert float((a - b).norm()) <= tol * float(b.norm())
    assert float((a - b).abs().max()) <= tol * float(b.abs().max())


@pytest.mark.parametrize("log_nt,n_det,r,prec,ncomp", [(13, 1, 1, 1, 1), (13, 8, 4, 1, 3), (14, 7, 2, 1, 3), (15, 5, 3, 2, 3),
                                                       (16, 8, 3, 1, 3), (17, 3, 2, 1, 1), (18, 5, 4, 1, 3), (20, 3, 2, 1, 3)])
@pytest.mark.parametrize("table", [False, True])
def test_pair_against_one_detector_packing(cmm, log_nt, n_det, r, prec, ncomp, table):
    full = gen.small_scan(cfg=411, ny=48, nx=50, n_t=1 << log_nt, ncols=4, nrows=2, throw_px=60.0, ncomp=ncomp)
    scan = full.subset(np.arange(n_det))
    op = cmm.Operator(cmm.Context(0), scan, gen.noise_params(n_det, scatter=0.2, cfg=411), precision=prec,
                      corr=modes(scan, r))
    if table:
        k = np.arange(scan.n_t // 2 + 1)
        op.noise.set_table(1.0 + 0.4 * np.sin(k / 9.0)[None] * np.linspace(0.3, 1.0, n_det)[:, None])
    m = torch.as_tensor(gen.random_maps(ncomp, scan.ny, scan.nx, 1, cfg=411)[0], device="cuda:0")
    g = torch.Generator(device="cuda:0").manual_seed(411)
    tod = torch.randn((n_det, scan.n_t), dtype=torch.float32, device="cuda:0", generator=g)
    pair, pair_b = op.apply(m).clone(), op.rhs(tod).clone()
    op.set_pair_packing(False)
    close(pair, op.apply(m), TOL[prec])
    close(pair_b, op.rhs(tod), TOL[prec])
    op.set_pair_packing(True)   # back: the tables return to the pair's slot order
    close(op.apply(m), pair, TOL[prec])
