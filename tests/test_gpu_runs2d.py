"""2D runs (stages 1 to 3, not the right-hand side alone) of each build of the stage
kernel, against the oracle: FP32 and HWENO_FP32C beyond one tile of 32 x 8 per SM
(152), where a cell has one thread, and beyond 304, where the dense builds run; FP64
beyond 152, with 8-row tiles.  Narrow grids, two tiles wide.  Tolerances as in the
other runs: FP64 1e-12, FP32 1e-4 relative L1 on shocked data; HWENO_FP32C holds its
averages to 2^-48 and its moments in FP32: 1e-5."""

import numpy as np
import pytest

from gpu_util import gpu_run2d, make_pair2d, mixed_burgers2d, mixed_euler2d, round_to, square_domain
from oracle import oracle as O
from paper_2002_08816_gb300 import hweno as H

pytestmark = pytest.mark.gpu

TOL = {H.HWENO_FP32: 1e-4, H.HWENO_FP64: 1e-12, H.HWENO_FP32C: 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _fp32c_run(cfg, u, steps):
    import torch
    h = H.hweno_create(cfg, torch.cuda.current_stream().cuda_stream)
    try:
        u = np.ascontiguousarray(u)
        H.hweno_set_state(h, u.ctypes.data, H.HWENO_FP64, False)
        t = H.hweno_step(h, steps)
        out = np.empty_like(u)
        H.hweno_get_state(h, out.ctypes.data, H.HWENO_FP64, False)
        return out, t
    finally:
        H.hweno_destroy(h)


@pytest.mark.parametrize("prec", [H.HWENO_FP32, H.HWENO_FP32C, H.HWENO_FP64])
@pytest.mark.parametrize("system,ng,bc", [(H.HWENO_EULER, 2, H.HWENO_BC_OUTFLOW), (H.HWENO_EULER, 3, H.HWENO_BC_OUTFLOW),
                                          (H.HWENO_BURGERS, 2, H.HWENO_BC_PERIODIC),
                                          (H.HWENO_BURGERS, 3, H.HWENO_BC_OUTFLOW)])
@pytest.mark.parametrize("size", [(40, 607), (40, 616), (40, 1217)])  # 152, 154 and 306 tiles
def test_runs2d_of_every_build(size, system, ng, bc, prec):
    nx, ny = size
    dom = square_domain(nx, ny)
    u = (mixed_euler2d if system == H.HWENO_EULER else mixed_burgers2d)(nx, ny, dom, nx + ny)
    u = round_to(prec, u)
    cfg, ocfg = make_pair2d(system, nx, ny, dom, bc, prec, ng=ng)
    if prec == H.HWENO_FP32C:
        got, t = _fp32c_run(cfg, u, 2)
    else:
        got, t, _ = gpu_run2d(cfg, u, 2)
    ref, t_ref, troubled = O.run2d(ocfg, u, nsteps=2, cfl=0.4, omp=True)
    assert troubled > 0
    assert np.abs(got - ref).sum() <= TOL[prec] * np.abs(ref).sum()
    assert abs(t - t_ref) <= (1e-13 if prec == H.HWENO_FP64 else 1e-6) * t_ref
