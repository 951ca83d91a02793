"""The circulant apply at ordinary sides just past the fused kernels' rule (threads a line):
columns of 675 and 1024 in FP32 and of 640 in FP64, which the line FFTs serve, each beside
a side that the fused kernels take."""
import pytest

from test_gpu_circ_sides import cmm  # noqa: F401
from test_gpu_circ_sides import test_circulant_apply as check_apply

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,nx", [(675, 12), (648, 12), (1024, 10), (640, 12), (600, 10)])
@pytest.mark.parametrize("prec,tol", [(0, 1e-10), (1, 1e-5)])
def test_sides(cmm, ny, nx, prec, tol):  # noqa: F811
    check_apply(cmm, ny, nx, prec, tol)
