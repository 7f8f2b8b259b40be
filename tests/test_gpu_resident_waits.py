"""The bounded waits of the resident 1D launches with limits so short that they run
out before the cell threads of the same CTA have come to the stage: the launch ends
with a status all the same, and the handle then runs as before."""

import numpy as np
import pytest

from gpu_util import mixed_euler
from paper_2002_08816_gb300 import hweno as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _check(prec, nx, threads, limits, silent):
    import torch
    io = H.HWENO_FP32 if prec == H.HWENO_FP32 else H.HWENO_FP64  # (pairs are held in 64 bits)
    dt = np.float32 if io == H.HWENO_FP32 else np.float64
    u = mixed_euler(nx, 4).astype(dt)
    cfg = H.make_config(1, H.HWENO_EULER, nx, bc=H.HWENO_BC_OUTFLOW, cfl=0.5, precision=prec)
    h = H.hweno_create(cfg, torch.cuda.current_stream().cuda_stream)
    try:
        if threads:
            H.hweno_set_execution(h, threads, 2)

        def steps():
            H.hweno_set_state(h, u.ctypes.data, io, False)  # (resets the status)
            H.hweno_step(h, 4)
            out = np.empty_like(u)
            H.hweno_get_state(h, out.ctypes.data, io, False)
            return out
        ref = steps()
        for polls in limits:
            H.hweno_set_state(h, u.ctypes.data, io, False)
            st = H.hweno_check_resident(h, 4, silent, polls)
            assert st in (H.HWENO_OK, H.HWENO_ERR_TIMEOUT) if silent < 0 else st == H.HWENO_ERR_TIMEOUT
            assert np.array_equal(steps(), ref), polls
    finally:
        H.hweno_destroy(h)


@pytest.mark.parametrize("prec,nx,threads", [(H.HWENO_FP32, 65536, 256), (H.HWENO_FP32, 20011, 512),
                                             (H.HWENO_FP32C, 20011, 256)])
@pytest.mark.parametrize("silent", [-1, 3])
def test_fp32_waits_of_a_few_polls_end(prec, nx, threads, silent):
    _check(prec, nx, threads, (1, 2, 3, 5, 9, 17, 40, 100, 300, 1000), silent)


@pytest.mark.parametrize("nx", [200, 8001, 65536])  # 26-cell tiles, and more cells to a tile
@pytest.mark.parametrize("silent", [-1, 3])
def test_fp64_waits_of_a_few_polls_end(nx, silent):
    _check(H.HWENO_FP64, nx, 0, (1, 2, 3, 5, 9, 17, 40, 100, 300, 1000), silent)


@pytest.mark.parametrize("nx,silent", [(200, 0), (8001, 17), (65536, 151)])
def test_fp64_run_gives_up_when_a_cta_never_publishes(nx, silent):
    """Every wait for alpha runs out: a status, nothing written, and the handle
    then steps as a batch of one does (by stage launches)."""
    import torch
    u = mixed_euler(nx, 4)
    cfg = H.make_config(1, H.HWENO_EULER, nx, bc=H.HWENO_BC_OUTFLOW, cfl=0.5, precision=H.HWENO_FP64)
    stream = torch.cuda.current_stream().cuda_stream
    got, back = np.empty_like(u), np.empty_like(u)
    h = H.hweno_create(cfg, stream)
    try:
        H.hweno_set_state(h, u.ctypes.data, H.HWENO_FP64, False)
        assert H.hweno_check_resident(h, 3, silent, 1 << 14) == H.HWENO_ERR_TIMEOUT
        H.hweno_get_state(h, back.ctypes.data, H.HWENO_FP64, False)
        assert np.array_equal(back, u)
        with pytest.raises(H.HwenoError):
            H.hweno_check_resident(h, 3, 1000, 1 << 14)
        H.hweno_set_state(h, u.ctypes.data, H.HWENO_FP64, False)
        assert H.hweno_check_resident(h, 4, -1, 1 << 21) == H.HWENO_OK
        H.hweno_get_state(h, got.ctypes.data, H.HWENO_FP64, False)
    finally:
        H.hweno_destroy(h)
    h = H.hweno_create_batch(cfg, [nx], stream)
    try:
        H.hweno_set_state(h, u.ctypes.data, H.HWENO_FP64, False)
        H.hweno_step(h, 4)
        H.hweno_get_state(h, back.ctypes.data, H.HWENO_FP64, False)
        with pytest.raises(H.HwenoError):  # no resident run
            H.hweno_check_resident(h, 3, -1, 1 << 14)
    finally:
        H.hweno_destroy(h)
    assert np.abs(got - back).sum() <= 1e-12 * np.abs(back).sum()
