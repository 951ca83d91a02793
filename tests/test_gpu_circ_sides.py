"""The circulant apply over map sides that need one, two and three passes of every radix,
sides that are their own mirror in every way, and sides past the fused kernels (served by
the line FFTs), against the FP64 oracle; and the r^T z that the last kernel forms."""
import numpy as np
import pytest

import gen
from oracle import mapmaker as om

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (ny, nx); the last two go past the fused column kernel (FP32, then FP64 only)
SIDES = [(8, 16), (9, 15), (10, 12), (16, 5), (27, 50), (45, 32), (81, 64), (125, 18), (64, 243), (96, 100), (30, 225), (375, 20),
         (4096, 10), (1440, 12)]


@pytest.fixture(scope="module")
def cmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_7473_gb300 import build
    build.build()
    from paper_1309_7473_gb300 import cmm as c
    return c


@pytest.mark.parametrize("ny,nx", SIDES)
@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-5)])
def test_circulant_apply(cmm, ny, nx, prec, tol):
    # a scan that crosses the middle 40 rows at most: the rest of a tall map is masked
    scan = gen.small_scan(cfg=381, ny=min(ny, 40), nx=nx, n_t=1 << 13, ncols=3, nrows=3, spacing_px=0.8, throw_px=1.4 * nx)
    bore = scan.bore.copy()
    bore[:, 1] += ((ny - scan.ny) // 2) << 16
    scan = gen.Scan(**{**scan.__dict__, "ny": ny, "bore": bore})
    noise = gen.noise_params(scan.n_det, fknee=2.0, alpha=3.5, scatter=0.2, cfg=381)
    oop = om.make_operator(scan, noise)
    ref = om.CirculantPrecon(oop, taper_sigma=5.0)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec)
    pc = cmm.Precon(op, cmm.PRECON_CIRCULANT, taper_sigma_px=5.0)
    m = gen.random_maps(3, ny, nx, 1, cfg=381)[0]
    z = pc.apply(torch.as_tensor(m, device="cuda:0")).cpu().numpy()
    zr = ref(m)
    assert np.abs(z - zr).max() <= tol * np.abs(zr).max()
    assert np.linalg.norm(z - zr) <= tol * np.linalg.norm(zr)
    if prec == 0:
        # rho = r^T z of the solve's first step comes from the apply's own partial sums:
        # one iteration's alpha r^T z against the oracle's
        b = om.apply_A(oop, m)
        _, _, _, terms = cmm.solve(op, pc, torch.as_tensor(b, device="cuda:0"), tol=0.0, maxit=1, history=True)
        zb = ref(b)
        rho = float(np.vdot(b, zb))
        alpha = rho / float(np.vdot(zb, om.apply_A(oop, zb)))
        assert abs(float(terms[0]) - alpha * rho) <= 1e-9 * alpha * rho
