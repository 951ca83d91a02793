"""The cross-detector step over more detectors than one stage of its shared memory holds
(128), the last stage ending in an odd detector: A and the right-hand side against the
one-detector packing and the FP64 oracle, law and table."""
import numpy as np
import pytest

import gen
from oracle import mapmaker as om

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-5   # the FP32 operator's bound


@pytest.fixture(scope="module")
def cmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_7473_gb300 import build
    build.build()
    from paper_1309_7473_gb300 import cmm as c
    return c


def rel(a, b):
    assert np.linalg.norm(b) > 0
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n_det", [128, 131, 257])
@pytest.mark.parametrize("table", [False, True])
def test_stages(cmm, n_det, table):
    scan = gen.small_scan(cfg=412, ny=48, nx=50, n_t=1 << 13, ncols=20, nrows=13, throw_px=60.0).subset(np.arange(n_det))
    noise = gen.noise_params(n_det, scatter=0.2, cfg=412)
    corr = gen.corr_noise(scan.det_off, r=3)
    w = om.filter_weights(noise, scan.n_t, scan.f_samp)
    if table:
        w = w * (1.0 + 0.4 * np.sin(np.arange(w.shape[1]) / 9.0)[None] * np.linspace(0.3, 1.0, n_det)[:, None])
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=1, corr=corr)
    if table:
        op.noise.set_table(w)
    m = gen.random_maps(3, scan.ny, scan.nx, 1, cfg=412)[0]
    d = np.random.default_rng(412).standard_normal((n_det, scan.n_t)).astype(np.float32)
    md, dd = torch.as_tensor(m, device="cuda:0"), torch.as_tensor(d, device="cuda:0")
    y, b = op.apply(md).cpu().numpy(), op.rhs(dd).cpu().numpy()
    op.set_pair_packing(False)
    assert rel(y, op.apply(md).cpu().numpy()) <= TOL and rel(b, op.rhs(dd).cpu().numpy()) <= TOL
    if n_det == 131:   # the oracle solves every bin's dense system
        oop = om.make_operator(scan, noise, corr=corr, w=w)
        assert rel(y, om.apply_A(oop, m)) <= TOL and rel(b, om.rhs(oop, d.astype(float))) <= TOL
