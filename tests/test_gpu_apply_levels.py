"""A when the two detectors of one sequence have different weights: every detector's own
pixels against the FP64 oracle to the operator's bound, and a detector without weight
gives exactly nothing."""
import numpy as np
import pytest

import gen
from oracle import mapmaker as om
from test_gpu_rhs_levels import TOL, cmm, errors, setup  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def apply(op, m):
    out = op.apply(torch.as_tensor(m, device="cuda:0"))
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("ratio", [1.9, 10.0, 1000.0])
@pytest.mark.parametrize("log_nt,ncomp,chunk,cached", [(13, 1, 0, False), (16, 3, 3, False), (18, 1, 0, True)])
def test_weight_ratios(cmm, prec, ratio, log_nt, ncomp, chunk, cached):  # noqa: F811
    scan, noise, alone = setup(5, log_nt, ncomp, [1.0, ratio, ratio, 1.0, ratio])
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec, det_chunk=chunk)
    if cached and prec:
        op.set_pixel_cache(True)
    m = gen.random_maps(ncomp, scan.ny, scan.nx, 1, cfg=397)[0]
    assert max(errors(apply(op, m), om.apply_A(om.make_operator(scan, noise), m), alone, ncomp)) <= TOL[prec]


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_table_with_cut_detectors(cmm, prec):  # noqa: F811
    scan, noise, alone = setup(5, 14, 1, [1.0, 1.0, 300.0, 1.0, 1.0])
    w = om.filter_weights(noise, scan.n_t, scan.f_samp)
    w[[1, 4]] = 0.0
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec)
    op.noise.set_table(w)
    m = gen.random_maps(1, scan.ny, scan.nx, 1, cfg=397)[0]
    got = apply(op, m)
    want = om.apply_A(om.make_operator(scan, noise, w=w), m)
    assert max(errors(got, want, alone[[0, 2, 3]], 1)) <= TOL[prec]
    assert np.abs(got.ravel()[alone[1] | alone[4]]).max() == 0.0


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("ratio", [1.0, 1000.0])
def test_correlated(cmm, prec, ratio):  # noqa: F811
    scan, noise, alone = setup(5, 13, 1, [1.0, ratio, 1.0, ratio, 1.0])
    corr = gen.corr_noise(scan.det_off, r=2)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec, corr=corr)
    m = gen.random_maps(1, scan.ny, scan.nx, 1, cfg=397)[0]
    assert max(errors(apply(op, m), om.apply_A(om.make_operator(scan, noise, corr=corr), m), alone, 1)) <= TOL[prec]
