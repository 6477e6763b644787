"""One context per host thread, as the C ABI allows, with grids whose strip kernels run with different
numbers of warps per block (24^2: one block; 200^2: 6 warps of FP32 and 3 of FP64; 512^2: 8): every call
succeeds and gives bitwise what it gives alone.  With timing on, a run is one launch per step, so the
threads' launches interleave thousands of times."""
import threading

import numpy as np
import pytest

from paper_2506_23895_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2506_23895_gb300 import build as B
    B.build()
    from paper_2506_23895_gb300 import lks
    import torch
    assert torch.cuda.is_available()
    return lks


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_contexts_of_several_sizes_in_threads(L, prec):
    import torch

    work = []
    for n, stride, rep in ((24, 1, 40), (200, 1, 40), (512, 1, 40), (200, 0, 80), (512, 0, 80)):
        w = W.small_channel2d(nx=n, ny=n, LD=8, n_steps=60, omega=0.01)
        s = L.Solver(w.problem, getattr(L, prec), stream=torch.cuda.Stream())
        s.set_design(w.gamma)
        s.set_motion(w.motion)
        work.append((s, s.forward(), s.adjoint(), stride, rep))
    torch.cuda.synchronize()
    bad, go = [], threading.Barrier(len(work))

    def run(s, J, g, stride, rep):
        try:
            s.set_timing(stride)
            go.wait()
            for _ in range(rep):
                if s.forward() != J or not np.array_equal(s.adjoint(), g):
                    bad.append("another result")
        except Exception as e:
            bad.append(repr(e))

    ts = [threading.Thread(target=run, args=a) for a in work]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for s, *_ in work:
        s.close()
    assert not bad, bad
