"""The 3D FP64 step and adjoint where their neighbour offsets can go wrong: axes of three nodes (a row
next to two faces), grids whose rows end inside a warp, and periodic axes of three and four nodes.
Nine FP64 steps of about 200 roundings of 1.1e-16 each stay below 1e-12."""
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


def close(a, b):
    return np.max(np.abs(np.asarray(a) - np.asarray(b))) <= 1e-12 * np.max(np.abs(b))


@pytest.mark.parametrize("nx,ny,nz,LD", [(13, 13, 12, 3), (33, 15, 13, 4), (14, 34, 19, 5)])
def test_duct_gradient_matches_oracle(L, nx, ny, nz, LD):
    w = W.small_duct3d(nx=nx, ny=ny, nz=nz, LD=LD, n_steps=9, trans_amp=0.5, seed=nx + ny)
    Jo, go = oracle.gradient(w.problem, w.gamma, w.motion)
    _, so = oracle.forward(w.problem, w.gamma, w.motion)
    s = L.Solver(w.problem, L.FP64)
    s.set_design(w.gamma)
    s.set_motion(w.motion)
    J = s.forward()
    st = s.get_state()
    g = s.adjoint()
    s.close()
    assert close(J, Jo) and close(st, so) and close(g, go)


@pytest.mark.parametrize("n,periodic", [
    ((3, 20, 9), (0, 0, 0)), ((35, 3, 9), (0, 0, 0)), ((31, 17, 3), (0, 0, 0)), ((3, 3, 3), (0, 0, 0)),
    ((3, 20, 9), (1, 0, 0)), ((4, 7, 33), (1, 1, 0)), ((33, 5, 3), (0, 1, 1)), ((3, 3, 4), (1, 1, 1))])
def test_small_axes_match_oracle(L, n, periodic):
    w = W.small_duct3d(nx=n[0], ny=n[1], nz=n[2], LD=5, n_steps=9, obj_kind=W.OBJ_PRESSURE)
    p = w.problem
    p.L = (0, 0, 0)
    p.bc = tuple(W.PERIODIC if periodic[f // 2] else p.bc[f] for f in range(6))
    p.u_init = (0.01, 0.02, 0.04)
    p.obj_box = (n[0] // 2, n[0] // 2, n[1] // 2, n[1] // 2, 0, 0)
    Jo, _, lo = oracle.gradient(p, np.zeros((0,)), w.motion, want_lam0=True)
    _, so = oracle.forward(p, np.zeros((0,)), w.motion)
    s = L.Solver(p, L.FP64)
    s.set_design(np.zeros((0,)))
    s.set_motion(w.motion)
    J = s.forward()
    st = s.get_state()
    s.adjoint()
    lam = s.get_adjoint_state()
    s.close()
    assert close(J, Jo) and close(st, so) and close(lam, lo)
