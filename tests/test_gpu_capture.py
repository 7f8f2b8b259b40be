"""hweno_step captured into a caller's CUDA graph, as the first step of the handle:
every launch a 1D handle may take, and 2D."""

import numpy as np
import pytest

from gpu_util import mixed_euler, mixed_euler2d, square_domain
from paper_2002_08816_gb300 import hweno as H
from paper_2002_08816_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    assert torch.cuda.is_available()
    import __graft_entry__
    __graft_entry__.build()


def _both(make, u, choice, prec):
    """Twice 3 steps by a graph captured as the handle's first call, and 6 steps."""
    import torch
    s = torch.cuda.Stream()
    dev = torch.from_numpy(np.ascontiguousarray(u)).to("cuda", torch.float64 if prec == H.HWENO_FP64 else torch.float32)
    torch.cuda.synchronize()
    outs = []
    for captured in (True, False):
        h = make(s.cuda_stream)
        try:
            if choice:
                H.hweno_set_execution(h, *choice)
            H.hweno_set_state(h, dev.data_ptr(), prec, True)
            torch.cuda.synchronize()
            if captured:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    H.hweno_step(h, 3, wait=False)
                with torch.cuda.stream(s):
                    g.replay()
                    g.replay()
            else:
                H.hweno_step(h, 6)
            out = torch.empty_like(dev)
            H.hweno_get_state(h, out.data_ptr(), prec, True)
            torch.cuda.synchronize()
            outs.append(out)
        finally:
            H.hweno_destroy(h)
    assert torch.equal(outs[0], outs[1])
    assert not torch.equal(outs[0], dev)


@pytest.mark.parametrize("prec,nx,choice", [
    (H.HWENO_FP64, 300, (256, 1)), (H.HWENO_FP64, 300, None), (H.HWENO_FP64, 80001, (128, 1)),
    (H.HWENO_FP64, 80001, None), (H.HWENO_FP32, 300, None), (H.HWENO_FP32, 20000, (128, 1)),
    (H.HWENO_FP32, 20000, (512, 2)), (H.HWENO_FP32, 80001, (256, 1))])
def test_single_instance(prec, nx, choice):
    cfg = H.make_config(1, H.HWENO_EULER, nx, bc=H.HWENO_BC_OUTFLOW, cfl=0.5, precision=prec)
    _both(lambda stream: H.hweno_create(cfg, stream), mixed_euler(nx, 3), choice, prec)


@pytest.mark.parametrize("prec", [H.HWENO_FP32, H.HWENO_FP64])
@pytest.mark.parametrize("kind", [0, 1])
def test_batch(prec, kind):
    sizes = W.batch_sizes_1d(9, seed=3, lo=40, hi=900)
    u = np.concatenate([mixed_euler(n, 50 + b).reshape(-1) for b, n in enumerate(sizes)])
    cfg = H.make_config(1, H.HWENO_EULER, 16, bc=H.HWENO_BC_OUTFLOW, cfl=0.5, precision=prec)
    _both(lambda stream: H.hweno_create_batch(cfg, sizes, stream), u, (128, kind), prec)


def test_2d():
    dom = square_domain(70, 50)
    cfg = H.make_config(2, H.HWENO_EULER, 70, 50, x0=dom[0], x1=dom[1], y0=dom[2], y1=dom[3],
                        bc=H.HWENO_BC_OUTFLOW, cfl=0.4, precision=H.HWENO_FP32)
    _both(lambda stream: H.hweno_create(cfg, stream), mixed_euler2d(70, 50, dom, 3), None, H.HWENO_FP32)
