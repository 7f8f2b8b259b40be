"""FP64 single-instance runs (tiles on chip for the whole run, the work of a
cell in tasks of one component, point or characteristic field) against the
oracle, at the sizes where the tiling changes: one tile, a short last tile, the
largest grid of 26-cell tiles and beyond it, more tiles than SMs, and a grid too
large to be resident.  Tolerance: as the other FP64 runs, 1e-12 relative L1."""

import numpy as np
import pytest

from gpu_util import gpu_run1d, make_pair, mixed_burgers
from oracle import oracle as O
from paper_2002_08816_gb300 import hweno as H
from paper_2002_08816_gb300 import workloads as W

pytestmark = pytest.mark.gpu

E, B = H.HWENO_EULER, H.HWENO_BURGERS
PER, OUT, REF = H.HWENO_BC_PERIODIC, H.HWENO_BC_OUTFLOW, H.HWENO_BC_REFLECTIVE
HYB, ALL, NONE = H.HWENO_TROUBLED_HYBRID, H.HWENO_TROUBLED_ALL, H.HWENO_TROUBLED_NONE


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _state(system, nx, bc):
    if system == B:
        return mixed_burgers(nx, 3)
    if bc == OUT:
        return W.euler_riemann_1d(nx, (0.445, 0.698, 3.528), (0.5, 0.0, 0.571), 0.0, 1.0, 0.4)
    return W.cell_moments_1d(lambda x: W.euler_conserved_1d(
        1.0 + 0.3 * np.cos(2 * np.pi * x) + 0.4 * (x > 0.6), 0.2 * np.sin(2 * np.pi * x), 1.0 + 0 * x),
        nx, 0.0, 1.0)


@pytest.mark.parametrize("system,bc,nx,mode,steps", [
    (E, OUT, 4, HYB, 9), (E, REF, 5, HYB, 9),           # below the resident run's 6 cells
    (E, OUT, 6, HYB, 9), (E, REF, 7, HYB, 12), (B, PER, 6, HYB, 9),
    (E, PER, 26, ALL, 12), (E, OUT, 27, HYB, 12), (B, PER, 31, ALL, 12), (E, REF, 53, HYB, 12),
    (E, OUT, 200, HYB, 30), (E, PER, 200, NONE, 12), (E, PER, 333, ALL, 12), (B, OUT, 7903, HYB, 6),
    (E, PER, 7904, HYB, 4), (E, OUT, 7905, HYB, 4), (E, REF, 8001, HYB, 4), (B, PER, 76911, HYB, 3),
    (E, OUT, 76912, HYB, 2), (E, OUT, 76913, HYB, 2)])
def test_fp64_runs_against_the_oracle(system, bc, nx, mode, steps):
    cfg, ocfg = make_pair(system, nx, 0.0, 1.0, bc, H.HWENO_FP64, mode=mode)
    u = _state(system, nx, bc)
    got, t, st = gpu_run1d(cfg, u, steps, chunks=2)
    ref, t_ref, tr = O.run1d(ocfg, u, nsteps=steps, cfl=0.5)
    assert st["steps"] == steps and st["troubled"] == tr
    assert np.abs(got - ref).sum() <= 1e-12 * np.abs(ref).sum()
    assert abs(t - t_ref) <= 1e-13 * t_ref


@pytest.mark.parametrize("variant", [H.HWENO_VARIANT_RAW_COMBINE, H.HWENO_VARIANT_MEAN_EIGEN])
def test_fp64_variants_against_the_per_instance_launches(variant):
    """Against a batch of one, which runs the per-stage launches."""
    import torch
    nx = 300
    u = _state(E, nx, OUT)
    cfg = H.make_config(1, E, nx, bc=OUT, cfl=0.5, precision=H.HWENO_FP64, variant=variant)
    got, t, _ = gpu_run1d(cfg, u, 4)
    h = H.hweno_create_batch(cfg, [nx], torch.cuda.current_stream().cuda_stream)
    try:
        H.hweno_set_state(h, u.ctypes.data, H.HWENO_FP64, False)
        H.hweno_step(h, 4)
        ref = np.empty_like(u)
        H.hweno_get_state(h, ref.ctypes.data, H.HWENO_FP64, False)
    finally:
        H.hweno_destroy(h)
    assert np.abs(got - ref).sum() <= 1e-12 * np.abs(ref).sum()
