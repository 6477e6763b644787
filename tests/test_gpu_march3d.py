"""The 3D FP32 row marches (forward step variant 2 and both adjoint variants) where their tiles can go
wrong: axes of three nodes, one column more or less than a tile (30 outputs forward, 28 adjoint), rows
around 4 w - 2 and 4 w - 4 of w warps, a few planes and several chunks of planes, footprint boxes that
cross the seams.  Against the 64-bit oracle; a step's FP32 result carries about 30 roundings of 6e-8 and
nine steps add up to less than 2e-5 of the largest state, four times that on the gradient."""
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


@pytest.mark.parametrize("nx,ny,nz,LD", [
    (13, 13, 12, 3), (32, 28, 13, 5), (33, 29, 14, 6), (31, 27, 19, 8), (29, 25, 35, 9),
    (28, 30, 12, 4), (62, 53, 17, 8), (57, 16, 40, 5), (15, 57, 27, 4)])
def test_row_marches_match_oracle(L, nx, ny, nz, LD):
    w = W.small_duct3d(nx=nx, ny=ny, nz=nz, LD=LD, n_steps=9, trans_amp=0.5, seed=nx + ny)
    Jo, go = oracle.gradient(w.problem, w.gamma, w.motion)
    _, so = oracle.forward(w.problem, w.gamma, w.motion)
    for v in (0, 1):
        s = L.Solver(w.problem, L.FP32)
        s.step_variant(2)
        s.adjoint_variant(v)
        s.set_design(w.gamma)
        s.set_motion(w.motion)
        J = s.forward()
        st = s.get_state()
        g = s.adjoint()
        s.close()
        assert np.max(np.abs(st - so)) <= 2e-5 * np.max(np.abs(so))
        assert abs(J - Jo) <= 2e-5 * abs(Jo)
        assert np.linalg.norm(g - go) <= 8e-5 * np.linalg.norm(go)


@pytest.mark.parametrize("nx,ny,nz", [(3, 20, 9), (40, 3, 9), (31, 17, 3), (3, 3, 3)])
def test_row_march_on_axes_of_three_nodes(L, nx, ny, nz):
    w = W.small_duct3d(nx=nx, ny=ny, nz=nz, LD=5, n_steps=9, obj_kind=W.OBJ_PRESSURE)
    w.problem.L = (0, 0, 0)
    Jo, so = oracle.forward(w.problem, np.zeros((0,)), w.motion)
    for v in (1, 2):
        s = L.Solver(w.problem, L.FP32)
        s.step_variant(v)
        s.set_design(np.zeros((0,)))
        s.set_motion(w.motion)
        J = s.forward()
        st = s.get_state()
        s.close()
        assert abs(J - Jo) <= 2e-5 * max(abs(Jo), 1e-3)
        assert np.max(np.abs(st - so)) <= 2e-5 * np.max(np.abs(so))
