"""The 2D transfer's tiles of 32 x 16 box nodes at the sizes where they can go wrong: boxes a node more or
less than one and two tiles, designs smaller than a tile and larger than two, angles at which the
lattices coincide, cross at 45 degrees and turn over, and steep rows (cosine or sine near 0).  A node
sums 16 products of three factors rounded to 1.1e-16 (FP64) or 6e-8 (FP32)."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("prec,tol", [("FP64", 1e-13), ("FP32", 4e-6)])
@pytest.mark.parametrize("n,LD", [(24, 3), (40, 20), (41, 21), (60, 27), (61, 28), (97, 55)])
@pytest.mark.parametrize("theta", [0.0, 0.003, np.pi / 4, 1.4, np.pi / 2, 3.0, np.pi, 4.0])
def test_transfer_tiles_match_oracle(L, prec, tol, n, LD, theta):
    w = W.small_channel2d(nx=n, ny=n + 1, LD=LD, n_steps=2, omega=0.2)
    w.motion[:, 0] = theta
    w.motion[:, 2:4] = (n - 1) / 2.0
    s = L.Solver(w.problem, getattr(L, prec))
    s.set_design(w.gamma)
    s.set_motion(w.motion)
    k, us = s.transfer(1)
    s.close()
    ko, uso = oracle.transfer(w.problem, w.gamma, w.motion[1])
    assert np.max(np.abs(k - ko)) < tol * np.max(np.abs(ko))
    assert np.max(np.abs(us - uso)) < tol * max(np.max(np.abs(uso)), 1e-3)
