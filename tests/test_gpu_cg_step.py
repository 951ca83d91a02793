"""The plain FP64 PCG step (k_cg_step, k_cg_dir, p^T q from the application's last
kernel) against the same iteration in torch: maps smaller than a block, one pixel over
a multiple of its threads, and more elements than one sweep of the grid."""
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


# Four iterations of a Jacobi-preconditioned solve from FP64 sums over n = 6.6e5
# elements: a sum is sqrt(n) 1e-16 ~ 8e-14 off and each iteration passes an error on by
# a factor of a few, so 1e-10 in FP64; the FP32 application is 5e-7 off A p (the
# operator's own bound is 1e-5), and four iterations pass on less than tenfold.
@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-4)])
@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("ny,nx,ncomp,n_t", [(9, 13, 1, 1 << 13), (9, 19, 3, 1 << 13), (27, 19, 1, 1 << 13),
                                             (200, 1100, 3, 1 << 16)])
def test_against_torch(cmm, ny, nx, ncomp, n_t, prec, graph, tol):
    scan = gen.small_scan(cfg=395, ny=ny, nx=nx, n_t=n_t, ncols=3, nrows=1, throw_px=0.8 * nx, ncomp=ncomp)
    op = cmm.Operator(cmm.Context(0), scan, gen.noise_params(scan.n_det, scatter=0.2, cfg=395), precision=prec)
    ref = cmm.Operator(cmm.Context(0), scan, gen.noise_params(scan.n_det, scatter=0.2, cfg=395), precision=cmm.PREC_F64)
    pc = cmm.Precon(op, cmm.PRECON_BINNED)
    b = ref.apply(torch.as_tensor(gen.random_maps(ncomp, ny, nx, 1, cfg=395)[0], device="cuda:0")).clone()
    x, info, _, _ = cmm.solve(op, pc, b, tol=0.0, maxit=4, use_graph=graph, true_resid=False)
    assert info.iterations == 4
    want = torch.zeros_like(b)
    r, z = b.clone(), pc.apply(b).clone()
    p, rz = z.clone(), float((b * z).sum())
    for _ in range(4):
        q = ref.apply(p).clone()
        a = rz / float((p * q).sum())
        want += a * p
        r -= a * q
        z = pc.apply(r).clone()
        new = float((r * z).sum())
        p, rz = z + (new / rz) * p, new
    assert float(want.norm()) > 0
    assert float((x - want).norm()) <= tol * float(want.norm())
