"""The two-detector path's row pairs (k1, R - k1), and the rows 0 and R / 2 that pair
with themselves: tabulated filters that pass one kind of row only, so that a slip in
one of them is not hidden by the others."""
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


@pytest.mark.parametrize("log_nt,R", [(13, 64), (14, 64), (16, 128), (17, 128), (18, 256)])
@pytest.mark.parametrize("rows", ["zero", "half", "one", "last"])
@pytest.mark.parametrize("n_det", [1, 3])
def test_rows_by_themselves(cmm, log_nt, R, rows, n_det):
    n_t = 1 << log_nt
    full = gen.small_scan(cfg=361, ny=20, nx=18, n_t=n_t, ncols=4, nrows=2, throw_px=30.0, ncomp=1)
    scan = full.subset(np.arange(n_det))
    noise = gen.noise_params(n_det, fknee=2.0, alpha=3.5, scatter=0.2, cfg=361)
    k1 = {"zero": 0, "half": R // 2, "one": 1, "last": R // 2 - 1}[rows]
    k = np.arange(n_t // 2 + 1)
    keep = (k % R == k1) | (k % R == (R - k1) % R)
    w = np.where(keep, 1.0 + 0.5 * np.sin(k / 11.0), 0.0)[None] * np.linspace(0.7, 1.3, n_det)[:, None]
    ctx = cmm.Context(0)
    op = cmm.Operator(ctx, scan, noise, precision=cmm.PREC_F32)
    op.noise.set_table(w)
    mask = op.pointing.mask()[0].reshape(scan.ny, scan.nx)
    m = gen.random_maps(1, scan.ny, scan.nx, 1, cfg=361)[0]
    y = op.apply(torch.as_tensor(m, device="cuda:0")).cpu().numpy()
    ref = om.apply_A(om.make_operator(scan, noise, mask.ravel(), w=w), m)
    # the FP32 operator's bound, for an output that keeps 2 / R of the samples' power:
    # FFT rounding of about 2e-7 of the unfiltered samples grows by sqrt(R / 2) <= 11.4
    err = np.linalg.norm(y - ref) / np.linalg.norm(ref)
    assert err < 1e-5, err
