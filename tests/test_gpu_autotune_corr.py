"""The tuner with noise correlated between detectors: it offers the two-detector packing,
times the correlated product, leaves the operator's results as they are, and keeps its
decision to operators with as many modes; cache files from before the mode count."""
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


def setup(cmm, n_det, r, prec=1, log_nt=16):
    scan = gen.small_scan(cfg=399, ny=64, nx=64, n_t=1 << log_nt, ncols=8, nrows=8, throw_px=60.0).subset(np.arange(n_det))
    noise = gen.noise_params(n_det, scatter=0.2, cfg=399)
    op = cmm.Operator(cmm.Context(0), scan, noise, precision=prec, corr=gen.corr_noise(scan.det_off, r=r) if r else None)
    return scan, op


def test_correlated_operator(cmm, tmp_path):
    scan, op = setup(cmm, 61, 3, 1, 18)
    m = torch.as_tensor(gen.random_maps(3, scan.ny, scan.nx, 1, cfg=399)[0], device="cuda:0")
    before = op.apply(m).clone()
    cache = str(tmp_path / "tune.txt")
    lr, pair, ms = cmm.cmm_autotune(op.h, 5, cache)
    assert ms > 0
    # the two-detector packing reads the spectra once less and its pointing once for two
    # detectors: 1.4 times as fast as the one-detector packing at 192 x 2^19
    assert pair
    after = op.apply(m)
    assert float((after - before).norm()) <= 1e-5 * float(before.norm())   # the FP32 operator's bound
    # the time is that of the correlated product, which has two passes more
    _, free = setup(cmm, 61, 0, 1, 18)
    t = cmm.cmm_profile_apply(free.h, m, free.new_map(), 20)[4]
    assert ms > 1.1 * t
    line = open(cache).read().split()
    assert line == [str(scan.n_t), "61", "1", "3", "3", "0"]
    # another mode count is another problem
    assert cmm.cmm_autotune(free.h, 3, cache)[2] > 0
    _, two = setup(cmm, 61, 2, 1, 18)
    assert cmm.cmm_autotune(two.h, 3, cache)[2] > 0
    _, same = setup(cmm, 61, 3, 1, 18)
    assert cmm.cmm_autotune(same.h, 3, cache)[1:] == (True, -1.0)


@pytest.mark.parametrize("prec,line,used", [(1, "{n} 59 1 3 0", True), (1, "{n} 58 1 3 7", False),
                                            (0, "{n} 57 0 3 8", False), (1, "{n} 56 1 3 0 7", True)])
def test_cache_lines(cmm, tmp_path, prec, line, used):
    n_det = int(line.split()[1])
    scan, op = setup(cmm, n_det, 0, prec, 13)
    cache = tmp_path / "tune.txt"
    cache.write_text("# other text\n" + line.format(n=scan.n_t) + "\n")
    lr, pair, ms = cmm.cmm_autotune(op.h, 3, str(cache))
    assert (ms == -1.0) == used
    if used:
        assert pair == (line.split()[-1] == "0") and (pair or lr == 7)


def test_operator_keeps_its_split(cmm):
    """The packing that the tuner chose leaves the split that the pixel cache, correlated
    noise and the one-detector packing need."""
    scan, op = setup(cmm, 55, 0, 1, 16)
    m = torch.as_tensor(gen.random_maps(3, scan.ny, scan.nx, 1, cfg=399)[0], device="cuda:0")
    assert cmm.cmm_autotune(op.h, 5, None)[1]
    op.set_pixel_cache(True)
    corr = gen.corr_noise(scan.det_off, r=1)
    op.noise.set_correlated(corr)
    _, ref = setup(cmm, 55, 1, 1, 16)
    assert float((op.apply(m) - ref.apply(m)).norm()) <= 1e-5 * float(ref.apply(m).norm())


def test_unsupported_correlation_is_still_tuned(cmm):
    """FP64 does not serve correlated noise: its applications fail, its tuning does not."""
    scan, op = setup(cmm, 7, 2, 0, 13)
    assert cmm.cmm_autotune(op.h, 2, None)[2] > 0
    with pytest.raises(cmm.CmmError):
        op.apply(op.new_map().fill_(1.0))
