"""The stop flag of the plain PCG step, which one block of a kernel sets while others may
still start: a batch of solves on their own streams, whose blocks share the SMs, stopped at
the iteration limit leaves the states that single solves leave, they resume to the same
iterates, and a solve that breaks down in its first step leaves x as it was."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NOT_CONVERGED, BREAKDOWN = 5, 4
SIZES = [(9, 13, 1), (24, 20, 3), (120, 140, 3), (330, 400, 3), (64, 64, 1), (30, 500, 3)]
# Two runs differ by the order of the FP64 sums, 1e-14 of a vector; six steps pass it on
# by at most a factor of ten each.
TOL = 1e-8


@pytest.fixture(scope="module")
def cmm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_7473_gb300 import build
    build.build()
    from paper_1309_7473_gb300 import cmm as c
    return c


def problem(cmm, ny, nx, ncomp, stream=None):
    scan = gen.small_scan(cfg=396, ny=ny, nx=nx, n_t=1 << 14, ncols=4, nrows=1, throw_px=0.8 * nx, ncomp=ncomp)
    op = cmm.Operator(cmm.Context(0, stream), scan, gen.noise_params(scan.n_det, scatter=0.2, cfg=396),
                      precision=cmm.PREC_F64)
    m = torch.as_tensor(gen.random_maps(ncomp, ny, nx, 1, cfg=396)[0], device="cuda:0")
    torch.cuda.synchronize()
    b = op.apply(m)   # on the operator's stream
    torch.cuda.synchronize()
    return scan, op, cmm.Precon(op, cmm.PRECON_JACOBI), b


def state(cmm, op):
    s = torch.zeros(cmm.cmm_solve_state_size(op.h), dtype=torch.float64, device="cuda:0")
    cmm.cmm_solve_state_save(op.h, s)
    return s


def close(a, b, tol=TOL):
    assert float(b.norm()) > 0
    assert float((a - b).norm()) <= tol * float(b.norm())


def test_batch_states_are_those_of_single_solves(cmm):
    streams = [torch.cuda.Stream() for _ in SIZES]
    batch = [problem(cmm, *sz, stream=st.cuda_stream) for sz, st in zip(SIZES, streams)]
    xs = [op.new_map() for _, op, _, _ in batch]
    torch.cuda.synchronize()
    infos = cmm.cmm_batch_solve([p[1].h for p in batch], [p[2].h for p in batch], [p[3] for p in batch], xs, tol=0.0,
                                maxit=6, check_every=4, width=len(SIZES), true_resid=False)
    for sz, (_, op, pc, b), x, info in zip(SIZES, batch, xs, infos):
        assert info.status == NOT_CONVERGED and info.iterations == 6
        _, one, pc1, b1 = problem(cmm, *sz)
        x1, info1, _, _ = cmm.solve(one, pc1, b1, tol=0.0, maxit=6, check_every=4, true_resid=False)
        assert info1.iterations == 6
        close(x, x1)
        n = x.numel()
        got, want = state(cmm, op), state(cmm, one)
        for k in (0, 1):   # r and p
            close(got[k * n:(k + 1) * n], want[k * n:(k + 1) * n])
        close(got[3 * n:], want[3 * n:])
        # resumed, the batch's state goes on to the iterates of the uninterrupted solve
        cmm.cmm_solve_state_load(one.h, got)
        info2 = cmm.cmm_solve(one.h, pc1.h, b1, x, 0.0, 10, 4, True, False, resume=True, true_resid=False)
        assert info2.iterations == 10
        _, whole, pc2, b2 = problem(cmm, *sz)
        xw, _, _, _ = cmm.solve(whole, pc2, b2, tol=0.0, maxit=10, check_every=4, true_resid=False)
        close(x, xw, 100 * TOL)


def test_breakdown_leaves_x(cmm):
    streams = [torch.cuda.Stream() for _ in range(4)]
    batch = [problem(cmm, 330, 400, 3, stream=st.cuda_stream) for st in streams]
    for scan, op, _, _ in batch[::2]:   # A = 0: p^T A p = 0 in the first step
        op.noise.set_table(np.zeros((scan.n_det, scan.n_t // 2 + 1)))
    xs = [op.new_map() for _, op, _, _ in batch]
    torch.cuda.synchronize()
    infos = cmm.cmm_batch_solve([p[1].h for p in batch], [p[2].h for p in batch], [p[3] for p in batch], xs, tol=0.0,
                                maxit=6, check_every=4, width=4, true_resid=False)
    for k, (info, x) in enumerate(zip(infos, xs)):
        assert info.status == (NOT_CONVERGED if k % 2 else BREAKDOWN)
        assert (float(x.abs().max()) == 0.0) == (k % 2 == 0)
