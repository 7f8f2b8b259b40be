"""hweno_autotune where the instance leaves nothing, or one launch, to choose: the
answer is the launch that runs, and does not depend on a timing."""

import numpy as np
import pytest

from gpu_util import mixed_euler
from paper_2002_08816_gb300 import hweno as H
from paper_2002_08816_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _tuned(prec, nx, before, sizes=None):
    import torch
    cfg = H.make_config(1, H.HWENO_EULER, nx, bc=H.HWENO_BC_OUTFLOW, cfl=0.5, precision=prec)
    stream = torch.cuda.current_stream().cuda_stream
    io = H.HWENO_FP32 if prec == H.HWENO_FP32 else H.HWENO_FP64
    u = mixed_euler(nx, 3) if sizes is None else np.concatenate([mixed_euler(n, 3).reshape(-1) for n in sizes])
    u = u.astype(np.float32 if io == H.HWENO_FP32 else np.float64)
    h = H.hweno_create(cfg, stream) if sizes is None else H.hweno_create_batch(cfg, sizes, stream)
    try:
        if before:
            H.hweno_set_execution(h, *before)
        H.hweno_set_state(h, u.ctypes.data, io, False)
        got = H.hweno_autotune(h, 4)
        assert H.hweno_stats(h)["steps"] == 0
        back = np.empty_like(u)
        H.hweno_get_state(h, back.ctypes.data, io, False)
        assert np.array_equal(back, u) or prec == H.HWENO_FP32C  # (64 bits into a pair)
        H.hweno_step(h, 2)
        H.hweno_set_execution(h, *got)  # the answer is a choice the handle takes
        return tuple(got)
    finally:
        H.hweno_destroy(h)


@pytest.mark.parametrize("prec,nx,before,want", [
    (H.HWENO_FP64, 300, None, (256, 0)), (H.HWENO_FP64, 300, (512, 1), (512, 1)),
    (H.HWENO_FP64, 65536, (128, 1), (128, 1)), (H.HWENO_FP32, 1000, (128, 0), (128, 0)),
    (H.HWENO_FP32, 1000, (512, 2), (512, 2)), (H.HWENO_FP32C, 1000, (512, 2), (512, 2)),
    (H.HWENO_FP32, 100000, (512, 0), (256, 0)), (H.HWENO_FP32, 200000, (512, 0), (128, 0))])
def test_nothing_to_choose(prec, nx, before, want):
    assert _tuned(prec, nx, before) == want


def test_only_launches_that_differ():
    assert _tuned(H.HWENO_FP32, 20000, (128, 0)) in ((256, 2), (512, 2))
    assert _tuned(H.HWENO_FP64, 80001, None)[1] in (0, 1)
    sizes = W.batch_sizes_1d(9, seed=3, lo=40, hi=900)
    assert _tuned(H.HWENO_FP32, 16, None, sizes)[1] == 0
    assert _tuned(H.HWENO_FP64, 16, None, sizes)[1] in (0, 1)
