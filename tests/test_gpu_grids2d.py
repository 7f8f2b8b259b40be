"""The 2D stage kernel at the tile counts where its build changes (FP32: two
threads per cell up to one 32 x 8 tile per SM, 152; the denser build beyond
304 tiles; FP64: 4-row tiles up to 152 8-row ones), against the oracle with the
bars of the other sizes: flags bit-exact off the threshold band, L within
gpu_util.rhs_tolerance2d."""

import pytest

from paper_2002_08816_gb300 import hweno as H
from test_gpu_parity2d import _built, _compare_rhs  # noqa: F401 (the build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [H.HWENO_FP32, H.HWENO_FP64])
@pytest.mark.parametrize("system,ng", [(H.HWENO_EULER, 2), (H.HWENO_EULER, 3), (H.HWENO_BURGERS, 3)])
@pytest.mark.parametrize("size", [(32, 8), (33, 9), (608, 64), (609, 64), (608, 65), (1216, 64),
                                  (1217, 64)])
def test_rhs2d_where_the_build_changes(size, system, ng, prec):
    _compare_rhs(system, size[0], size[1], H.HWENO_BC_OUTFLOW, prec, H.HWENO_TROUBLED_HYBRID, ng,
                 seed=size[0] + size[1])
