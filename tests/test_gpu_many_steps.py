"""A step count that only t_final ends: 3 stages of each no longer fit 32 bits."""

import numpy as np
import pytest

from gpu_util import gpu_run1d
from paper_2002_08816_gb300 import hweno as H
from paper_2002_08816_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("prec,nx", [(H.HWENO_FP32, 64), (H.HWENO_FP32, 5000), (H.HWENO_FP64, 64)])
def test_most_steps_an_int_holds_end_at_t_final(prec, nx):
    u = W.burgers_sine_1d(nx)
    cfg = H.make_config(1, H.HWENO_BURGERS, nx, x0=-1.0, x1=1.0, cfl=0.5, precision=prec)
    tf = 20.3 * 0.5 * (2.0 / nx) / 1.5
    ref, t_ref, st_ref = gpu_run1d(cfg, u, 60, t_final=tf)
    got, t, st = gpu_run1d(cfg, u, 2 ** 31 - 1, t_final=tf)
    assert t == t_ref == tf and st["steps"] == st_ref["steps"] > 0
    assert np.array_equal(got, ref)
