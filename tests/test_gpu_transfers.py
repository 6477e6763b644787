"""The staged general-axis transfer and the listed density filter at the sizes where they can go
wrong: footprint boxes of several 8^3 tiles with remainders, designs that fill their tiles' lists,
coincident lattices, filters of one offset, and of more offsets than a block lists.  Tolerances: a box
node sums 64 products of four factors rounded to 1.1e-16, a filtered value at most 2,500."""
import numpy as np
import pytest

import oracle
from oracle import design_chain as D
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


@pytest.mark.parametrize("n,LD,axis,theta0", [
    (24, 4, (1.0, 1.0, 1.0), 0.0), (40, 17, (0.3, -0.5, 0.81), 0.7),
    (47, 20, (1.0, 0.0, 0.0), np.pi / 4), (47, 20, (0.0, 1.0, 1.0), 2.1)])
def test_axis_transfer_matches_oracle(L, n, LD, axis, theta0):
    w = W.small_duct3d(nx=n, ny=n - 1, nz=n, LD=LD, n_steps=4, rot_axis=W.unit(axis), omega=0.3,
                       trans_amp=0.0, seed=n + LD)
    w.motion[:, 0] += theta0 - w.motion[0, 0]
    w.motion[:, 2:5] = np.array([(n - 1) / 2.0, (n - 2) / 2.0, (n - 1) / 2.0])
    s = L.Solver(w.problem, L.FP64)
    s.set_design(w.gamma)
    s.set_motion(w.motion)
    for t in (1, 4):
        k, us = s.transfer(t)
        ko, uso = oracle.transfer(w.problem, w.gamma, w.motion[t])
        assert np.max(np.abs(k - ko)) < 1e-13 * np.max(np.abs(ko))
        assert np.max(np.abs(us - uso)) < 1e-13 * max(np.max(np.abs(uso)), 1e-3)
    s.close()


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("R", [0.9, 1.0, 2.4, 6.1, 8.2])
def test_filter_radii_match_oracle(L, dim, R):
    w = (W.small_channel2d(nx=40, ny=34, LD=15, n_steps=2, omega=0.0) if dim == 2
         else W.small_duct3d(nx=28, ny=27, nz=28, LD=11, n_steps=2))
    s = L.Solver(w.problem, L.FP64)
    s.set_design(w.gamma)
    s.set_filter(R, 3.0)
    G, dG = s.volume(0.4)
    s.close()
    Go, dGo = D.volume(w.gamma, 0.4, R, 3.0)
    assert abs(G - Go) < 1e-12
    assert np.max(np.abs(dG - dGo)) < 1e-12 * np.max(np.abs(dGo))
