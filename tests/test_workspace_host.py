"""Device memory of 2D contexts (host only, no GPU): a context on the table kernels takes no more than one
on the plain kernels with the same snapshots, but for a state and, in FP32, a transfer slot for each
snapshot slot up to max(ceil(sqrt(N)) + 2, 64), in FP64 half of what the snapshots take (512 MB at most);
so ckpt_bytes bounds the whole."""
import ctypes
import math

import pytest

from paper_2506_23895_gb300 import build as B
from paper_2506_23895_gb300 import lks
from paper_2506_23895_gb300 import workloads as W


@pytest.fixture(scope="module")
def lib():
    B.build()
    return lks.load()


def workspace(lib, p, prec, slots, flags):
    c = lks.make_config(p, prec, ckpt_bytes=slots * lks.state_bytes(p, prec), flags=flags)
    return lib.lks_workspace_bytes(ctypes.byref(c))


@pytest.mark.parametrize("prec", [lks.FP32, lks.FP64])
@pytest.mark.parametrize("n", [24, 512, 4096, 16384])
@pytest.mark.parametrize("steps", [40, 2000, 20000])
@pytest.mark.parametrize("frac", [0.2, 0.68])
def test_2d_contexts_stay_within_their_snapshot_budget(lib, prec, n, steps, frac):
    p = W.small_channel2d(n_steps=steps).problem
    p.n = (n, n, 1)
    side = max(1, int(frac * (n - 6)))
    p.L = (side, side, 1)
    p.obj_box = (0, 0, 1, n - 2, 0, 0)
    state = lks.state_bytes(p, prec)
    for slots in (3, 8, 16, 64, 142):
        P = min(slots, steps + 1)
        kept = min(P, max(math.ceil(math.sqrt(steps)) + 2, 64)) if prec == lks.FP32 else 0
        plain = workspace(lib, p, prec, slots, lks.FLAG_PLAIN_KERNELS)
        table = workspace(lib, p, prec, slots, 0)
        half = min(P * state // 2, 512 << 20) if prec == lks.FP64 else 0
        assert table <= plain + half + (1 + kept) * state + (64 << 10)


@pytest.mark.parametrize("prec", [lks.FP32, lks.FP64])
@pytest.mark.parametrize("n", [48, 96, 256])
def test_3d_contexts_share_scratch_between_forward_and_adjoint(lib, prec, n):
    """Seven states, the snapshots, f^eq of 15 directions, six components of S~ and the static field;
    the adjoint's mu lives where f^eq does.  What is smaller than one number a node is left room for."""
    p = W.small_duct3d(n_steps=20).problem
    p.n = (n, n, n)
    p.L = (0, 0, 0)
    T = 8 if prec == lks.FP64 else 4
    state = lks.state_bytes(p, prec)
    for flags in (0, lks.FLAG_PLAIN_KERNELS):
        assert workspace(lib, p, prec, 3, flags) <= (7 + 3) * state + (15 + 6 + 1 + 1) * n ** 3 * T
