"""P m at the edges of the projection kernel's blocks (samples and detectors that do not
fill one), on cut and periodic maps, in every type, against the FP64 oracle."""
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


@pytest.mark.parametrize("n_t,ncols,nrows", [(32, 1, 1), (256, 3, 3), (1024, 4, 2), (2048, 17, 1)])
@pytest.mark.parametrize("ncomp", [1, 3])
@pytest.mark.parametrize("periodic", [False, True])
# FP32: the map copy, the response and three products round once each: 4e-7 of max |P m|
@pytest.mark.parametrize("prec,dtype,tol", [(0, torch.float64, 1e-14), (1, torch.float32, 1e-6), (1, torch.float64, 1e-6)])
def test_project(cmm, n_t, ncols, nrows, ncomp, periodic, prec, dtype, tol):
    scan = gen.small_scan(cfg=401, ny=20, nx=24, n_t=n_t, ncols=ncols, nrows=nrows, spacing_px=0.7, throw_px=40.0,
                          ncomp=ncomp)
    scan = gen.Scan(**{**scan.__dict__, "periodic": periodic})
    noise = gen.noise_params(scan.n_det, cfg=401)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec)
    m = gen.random_maps(ncomp, scan.ny, scan.nx, 1, cfg=401)[0]
    got = op.project(torch.as_tensor(m, device="cuda:0"), dtype=dtype).cpu().numpy()
    ref = om.project(om.make_operator(scan, noise), m)
    assert got.shape == ref.shape
    assert np.abs(got - ref).max() <= tol * max(np.abs(ref).max(), 1e-300)
