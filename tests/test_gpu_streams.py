"""Handles on streams of their own, driven by one thread and by several: the resident
runs share the GPU (each waits within its own launch only), so the states are those of
the same handles one after the other, bit for bit, and no wait runs out."""

import threading

import numpy as np
import pytest

from gpu_util import mixed_euler
from paper_2002_08816_gb300 import hweno as H

pytestmark = pytest.mark.gpu

F32, F64 = H.HWENO_FP32, H.HWENO_FP64


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _run(specs, how, steps=24):
    import torch
    hs, outs = [], []
    for i, (prec, nx) in enumerate(specs):
        u = mixed_euler(nx, 60 + i).astype(np.float32 if prec == F32 else np.float64)
        s = torch.cuda.Stream()
        cfg = H.make_config(1, H.HWENO_EULER, nx, bc=H.HWENO_BC_OUTFLOW, cfl=0.5, precision=prec)
        hs.append((H.hweno_create(cfg, s.cuda_stream), u, prec, s))
        H.hweno_set_state(hs[-1][0], u.ctypes.data, prec, False)
    torch.cuda.synchronize()

    def steps_of(h):
        for k in (steps // 2, 1, steps - steps // 2 - 1):
            H.hweno_step(h, k, -1.0, wait=False)
    if how == "threads":
        threads = [threading.Thread(target=steps_of, args=(h,)) for h, _, _, _ in hs]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    else:
        for h, _, _, _ in hs:
            steps_of(h)
            if how == "one after the other":
                torch.cuda.synchronize()
    for h, u, prec, _ in hs:
        H.hweno_step(h, 0)  # the status: HwenoError if a wait had run out
        out = np.empty_like(u)
        H.hweno_get_state(h, out.ctypes.data, prec, False)
        outs.append(out)
        H.hweno_destroy(h)
    return outs


@pytest.mark.parametrize("specs", [[(F32, 20000)] * 6, [(F32, 5000)] * 16, [(F32, 70000)] * 3, [(F64, 400)] * 12,
                                   [(F64, 20000)] * 3,
                                   [(F32, 20000), (F64, 400), (F32, 1000), (F64, 20000), (F32, 5000), (F64, 200),
                                    (F32, 70000), (F32, 300)]])
def test_streams_and_threads(specs):
    ref = _run(specs, "one after the other")
    for how in ("streams", "threads"):
        for a, b in zip(_run(specs, how), ref):
            assert np.array_equal(a, b)
