"""Every launch a 1D run can take, each against the oracle: per-stage launches of one
instance (grids too large to be resident) and of a batch, the FP64 persistent launch,
the resident launches and the cluster.  A single instance that fits on chip runs there
whatever its handle is set to, so the other launches are reached by batches and by
larger grids.  Tolerances as in the other runs: FP64 1e-12 relative L1, FP32 1e-4
(the target), times 1e-13 and 1e-6."""

import numpy as np
import pytest

from gpu_util import make_pair, mixed_burgers, mixed_euler, round_to
from oracle import oracle as O
from paper_2002_08816_gb300 import hweno as H
from paper_2002_08816_gb300 import workloads as W

pytestmark = pytest.mark.gpu

E, B = H.HWENO_EULER, H.HWENO_BURGERS
PER, OUT, REF = H.HWENO_BC_PERIODIC, H.HWENO_BC_OUTFLOW, H.HWENO_BC_REFLECTIVE
F32, F64, F32C = H.HWENO_FP32, H.HWENO_FP64, H.HWENO_FP32C
TOL = {F32: 1e-4, F64: 1e-12, F32C: 1e-5}
TOL_T = {F32: 1e-6, F64: 1e-13, F32C: 1e-6}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _data(system, bc, nx, seed):
    if system == B:
        return mixed_burgers(nx, seed)
    if bc == OUT:
        return mixed_euler(nx, seed)
    # at rest beside the walls; periodic
    return W.cell_moments_1d(lambda x: W.euler_conserved_1d(
        1.0 + 0.3 * np.cos(2 * np.pi * x) + 0.4 * (x > 0.6), 0.2 * np.sin(2 * np.pi * x), 1.0 + 0 * x),
        nx, 0.0, 1.0)


def _run(h, flat, io, steps, t_final=-1.0, chunks=1):
    H.hweno_set_state(h, flat.ctypes.data, io, False)
    for k in range(chunks):
        t = H.hweno_step(h, steps // chunks, t_final)
    out = np.empty_like(flat)
    H.hweno_get_state(h, out.ctypes.data, io, False)
    return out.astype(np.float64), t


def _close(got, t, ref, t_ref, prec):
    assert np.abs(got - ref).sum() <= TOL[prec] * np.abs(ref).sum()
    assert abs(t - t_ref) <= TOL_T[prec] * t_ref


def _single(system, bc, nx, prec, steps, choice=None, t_final=-1.0, chunks=1, seed=5):
    import torch
    u = round_to(prec, _data(system, bc, nx, seed))
    cfg, ocfg = make_pair(system, nx, 0.0, 1.0, bc, prec)
    io = F32 if prec == F32 else F64
    h = H.hweno_create(cfg, torch.cuda.current_stream().cuda_stream)
    try:
        if choice:
            H.hweno_set_execution(h, *choice)
        got, t = _run(h, u.astype(np.float32 if io == F32 else np.float64), io, steps, t_final, chunks)
        stats = H.hweno_stats(h)
    finally:
        H.hweno_destroy(h)
    ref, t_ref, tr = O.run1d(ocfg, u, nsteps=steps, cfl=0.5, t_final=t_final, omp=True)
    _close(got, t, ref, t_ref, prec)
    if prec == F64:
        assert stats["troubled"] == tr
    return t


@pytest.mark.parametrize("prec", [F32, F32C])
@pytest.mark.parametrize("system,bc", [(E, OUT), (E, REF), (E, PER), (B, PER)])
@pytest.mark.parametrize("nx", [6, 7, 122, 249, 250, 251, 976, 977, 2000, 2003, 3999, 4000, 4001])
def test_cluster_sizes(nx, system, bc, prec):
    """One CTA up to 250 cells, clusters of up to 16 to 4000, and the resident launch
    beyond; 6 and 7 cells with gentle data (they resolve no jump)."""
    if nx < 10 and (system == B or bc == OUT):
        pytest.skip("a jump on six cells")
    _single(system, bc, nx, prec, 12, chunks=2)


@pytest.mark.parametrize("system,bc", [(E, OUT), (E, REF), (E, PER), (B, PER)])
@pytest.mark.parametrize("nx", [76001, 152000, 152001])  # 256-thread tiles up to 152000 cells, then 128
def test_fp32_stage_launches_of_one_instance(nx, system, bc):
    _single(system, bc, nx, F32, 4)


@pytest.mark.parametrize("system,bc", [(E, OUT), (B, PER)])
@pytest.mark.parametrize("choice", [(t, k) for k in (0, 1) for t in (128, 256, 512)])
def test_fp64_launches_of_one_instance(choice, system, bc):
    _single(system, bc, 76913, F64, 2, choice)


def test_fp64_persistent_run_ends_at_t_final():
    nx = 76914
    tf = 1.4 * 0.5 / nx / 2.0  # (two-state data: alpha is about 2)
    assert _single(E, OUT, nx, F64, 6, (256, 1), t_final=tf) == tf


@pytest.mark.parametrize("prec,choice", [(F32, (128, 0)), (F32, (256, 0)), (F32, (512, 0))] +
                         [(F64, (t, k)) for k in (0, 1) for t in (128, 256, 512)])
@pytest.mark.parametrize("system,bc", [(E, OUT), (E, REF), (B, PER)])
def test_batches(system, bc, prec, choice):
    """Every instance of an uneven batch, then the whole batch clipped by t_final."""
    import torch
    sizes = [40, 121, 122, 123, 250, 507, 1003]
    us = [round_to(prec, _data(system, bc, n, 70 + n)) for n in sizes]
    cfg, _ = make_pair(system, 40, 0.0, 1.0, bc, prec)
    flat = np.concatenate([u.reshape(-1) for u in us]).astype(np.float32 if prec == F32 else np.float64)
    h = H.hweno_create_batch(cfg, sizes, torch.cuda.current_stream().cuda_stream)
    try:
        H.hweno_set_execution(h, *choice)
        for steps, t_final in ((9, -1.0), (400, 0.01)):
            got, _ = _run(h, flat, prec, steps, t_final)
            times = H.hweno_batch_times(h, len(sizes))
            off = 0
            for n, u, t in zip(sizes, us, times):
                _, ocfg = make_pair(system, n, 0.0, 1.0, bc, prec)
                ref, t_ref, _ = O.run1d(ocfg, u, nsteps=steps, cfl=0.5, t_final=t_final)
                _close(got[off:off + u.size].reshape(u.shape), t, ref, t_ref, prec)
                off += u.size
    finally:
        H.hweno_destroy(h)


@pytest.mark.parametrize("threads", [256, 512])
def test_resident_threads(threads):
    _single(E, OUT, 20011, F32, 10, (threads, 2), chunks=2)
    _single(E, OUT, 20011, F32C, 10, (threads, 2), chunks=2)


@pytest.mark.parametrize("prec", [F32, F32C])
@pytest.mark.parametrize("bc", [OUT, REF, PER])
@pytest.mark.parametrize("nx", [5251, 37999, 38000, 38001])  # full tiles up to one per SM, then shares of all slots
def test_resident_tilings(nx, bc, prec):
    _single(E, bc, nx, prec, 6, chunks=2)
